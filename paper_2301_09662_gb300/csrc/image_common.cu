// Stages shared by every arithmetic form: the exact integer auto-power (a7)
// and the epilogue that sums the partial images, subtracts the
// autocorrelation term and writes the shifted output (a8).
//
// Autocorrelation removal (Sec. 2.2): the a = b terms of F_p F_q^* are
// e~_ap e~_aq^* |W^(l)|^2 for every antenna, so their sum over the integration
// is A_pq |W^(l)|^2 with A_pq = sum_a g_ap g_aq^* sum_t e_ap e_aq^*.  The inner
// time sum is exact in int32 (|e e^*| components <= 128, T <= 10^5); the
// antenna sum and the subtraction run in FP64 because the auto term can be
// much larger than what is left after it is removed (the subtraction in FP32
// pairs of ~48 bits, see epilogue_kernel).
#include <algorithm>
#include <type_traits>

#include "epic_internal.cuh"

namespace epic {
namespace {

__device__ __forceinline__ void ci4_parts(uint32_t b, int &re, int &im)
{
    re = static_cast<int>(static_cast<int8_t>(b & 0xF0u)) >> 4;
    im = static_cast<int>(static_cast<int8_t>((b << 4) & 0xF0u)) >> 4;
}

// sums of one antenna: [0] |e_X|^2  [1] |e_Y|^2  [2] Re e_X e_Y^*  [3] Im e_X e_Y^*
template <int P>
__device__ __forceinline__ void auto_add(uint32_t bx, uint32_t by, int (&s)[P == 2 ? 4 : 1])
{
    int xr, xi;
    ci4_parts(bx, xr, xi);
    s[0] += xr * xr + xi * xi;
    if constexpr (P == 2) {
        int yr, yi;
        ci4_parts(by, yr, yi);
        s[1] += yr * yr + yi * yi;
        s[2] += xr * yr + xi * yi;
        s[3] += xi * yr - xr * yi;
    }
}

// grid (C, n_chunks): per antenna, the integer sums over one time chunk, from 32-bit words of the
// rows (WORDS: n_ant n_pol a multiple of 4 and v aligned to it, 4 / P antennas a thread) or one antenna a thread.
// chunk_stride 0: every chunk adds into one (cleared) sum; else each chunk stores its own.
template <int P, bool WORDS>
__global__ void __launch_bounds__(128)
autopower_kernel(const uint8_t *__restrict__ v, int T, int C, int A, int n_chunks, size_t chunk_stride,
                 int *__restrict__ autoint)
{
    constexpr int NA = WORDS ? 4 / P : 1, NS = P == 2 ? 4 : 1;
    const int c = blockIdx.x;
    const int chunk = blockIdx.y;
    const int t0 = static_cast<int>(static_cast<long long>(T) * chunk / n_chunks);
    const int t1 = static_cast<int>(static_cast<long long>(T) * (chunk + 1) / n_chunks);
    const size_t row = static_cast<size_t>(C) * A * P;
    for (int u = threadIdx.x; u * NA < A; u += blockDim.x) {
        int s[NA][NS];
#pragma unroll
        for (int n = 0; n < NA; n++)
#pragma unroll
            for (int k = 0; k < NS; k++) s[n][k] = 0;
        const uint8_t *src = v + static_cast<size_t>(t0) * row + static_cast<size_t>(c) * A * P + static_cast<size_t>(u) * NA * P;
#pragma unroll 8
        for (int t = t0; t < t1; t++, src += row) {
            if constexpr (WORDS) {
                const uint32_t w = __ldg(reinterpret_cast<const uint32_t *>(src));
#pragma unroll
                for (int n = 0; n < NA; n++) auto_add<P>(w >> (8 * P * n), w >> (8 * P * n + 8), s[n]);
            } else {
                auto_add<P>(src[0], P == 2 ? src[P - 1] : 0u, s[0]);
            }
        }
#pragma unroll
        for (int n = 0; n < NA; n++) {
            int *dst = autoint + chunk * chunk_stride + (static_cast<size_t>(c) * A + u * NA + n) * 4;
#pragma unroll
            for (int k = 0; k < NS; k++) {
                if (chunk_stride) dst[k] = s[n][k];
                else atomicAdd(dst + k, s[n][k]);
            }
        }
    }
}

// A_pq = sum_a g_ap g_aq^* sum_t e_ap e_aq^* of channel c, by one block, in FP64 and a fixed order
// (deterministic); sums of n_chunks chunks (exact integers) first.  Result in apq: XX, YY, Re XY, Im XY.
template <int P>
__device__ __forceinline__ void auto_reduce(const int *autoint, int n_chunks, size_t chunk_stride, const float2 *gains,
                                            int A, int c, double (&red)[kThreads / 32][4], double (&apq)[4])
{
    double s[4] = {0, 0, 0, 0};
    for (int a = threadIdx.x; a < A; a += kThreads) {
        int ia[4] = {0, 0, 0, 0};
        const int *src = autoint + (static_cast<size_t>(c) * A + a) * 4;
#pragma unroll 4
        for (int k = 0; k < n_chunks; k++) {
            if constexpr (P == 2) {
                const int4 q = *reinterpret_cast<const int4 *>(src + k * chunk_stride);
                ia[0] += q.x;
                ia[1] += q.y;
                ia[2] += q.z;
                ia[3] += q.w;
            } else {
                ia[0] += src[k * chunk_stride];
            }
        }
        double gxr = 1, gxi = 0, gyr = 1, gyi = 0;
        if (gains) {
            const float2 gx = gains[(static_cast<size_t>(c) * A + a) * P];
            gxr = gx.x;
            gxi = gx.y;
            if (P == 2) {
                const float2 gy = gains[(static_cast<size_t>(c) * A + a) * P + 1];
                gyr = gy.x;
                gyi = gy.y;
            }
        }
        s[0] += (gxr * gxr + gxi * gxi) * static_cast<double>(ia[0]);
        if (P == 2) {
            s[1] += (gyr * gyr + gyi * gyi) * static_cast<double>(ia[1]);
            // g_x g_y^* (I_re + i I_im)
            const double pr = gxr * gyr + gxi * gyi, pi = gxi * gyr - gxr * gyi;
            s[2] += pr * ia[2] - pi * ia[3];
            s[3] += pr * ia[3] + pi * ia[2];
        }
    }
    // fixed-order tree: within each warp by shuffles, then the warps' sums by thread 0..3
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_down_sync(0xffffffffu, s[k], o);
    if ((threadIdx.x & 31) == 0)
        for (int k = 0; k < 4; k++) red[threadIdx.x >> 5][k] = s[k];
    __syncthreads();
    if (threadIdx.x < 4) {
        double tot = 0;
        for (int i = 0; i < kThreads / 32; i++) tot += red[i][threadIdx.x];
        apq[threadIdx.x] = tot;
    }
    __syncthreads();
}

// grid (C, images): A_pq once per channel and image, for the epilogue's blocks to read
template <int P>
__global__ void __launch_bounds__(kThreads)
auto_sum_kernel(const int *__restrict__ autoint, int n_chunks, size_t chunk_stride, const float2 *__restrict__ gains, int A,
                int C, double *__restrict__ apq_out)
{
    __shared__ double red[kThreads / 32][4];
    __shared__ double apq[4];
    auto_reduce<P>(autoint + static_cast<size_t>(blockIdx.y) * n_chunks * chunk_stride, n_chunks, chunk_stride, gains, A,
                   blockIdx.x, red, apq);
    if (threadIdx.x < 4) apq_out[(static_cast<size_t>(blockIdx.y) * C + blockIdx.x) * 4 + threadIdx.x] = apq[threadIdx.x];
}

// A number as an unevaluated FP32 pair (hi, lo), about 48 bits (infinity as itself).
__device__ __forceinline__ float2 to_pair(double x)
{
    const float hi = static_cast<float>(x);
    return make_float2(hi, isinf(hi) ? 0.f : static_cast<float>(x - static_cast<double>(hi)));
}
// h + x exactly as (sum, error): the error is returned (Knuth's TwoSum)
__device__ __forceinline__ float two_sum(float &h, float x)
{
    const float t = h + x;
    const float bp = t - h;
    const float e = (h - (t - bp)) + (x - bp);
    h = t;
    return e;
}
// s -= a b in pairs (a, b, s pairs of ~48 bits; the product's high part by an exact two-product)
__device__ __forceinline__ void pair_msub(float2 &s, float2 a, float2 b)
{
    const float p = __fmul_rn(a.x, b.x);
    const float e = fmaf(a.x, b.y, fmaf(a.y, b.x, fmaf(a.x, b.x, -p)));
    const float r = two_sum(s.x, -p);
    s.y += r - e;
}

// grid (pixel tiles, group channels, images).  Partial layout written by the imaging
// kernels: [tau][item][pos][NPF] with item = ci * Q + (hy * Q1 + hx) and
// pos = py * M + px, where folded frequency m sits at digit position
// up (R2 (m mod R1) + m / R1) (R1 = 1, R2 = M for natural order; up = 2 when a
// side-32 grid was transformed zero-padded to 64 points, whose even
// frequencies are the 32-point transform).
//
// Bound by HBM (partials read once, image written once).  The subtraction
// runs in FP32 pairs (~48 bits): GB300's FP64 pipe does ~2 operations a clock
// and SM, and five FP64 operations and eight conversions a value made it, not
// the memory, the limit; A_pq itself is summed in FP64, once per channel and
// image (auto_sum_kernel), not in every block (apq_tab null: the plan-free entry point's blocks sum
// autoint themselves).  Also for small arrays, whose sums are shorter than a launch: 16 antennas, 32 x 32,
// 4 channels of 64 spectra 18.4 us with the blocks' own sums, 16.4 so; 64 channels of 128 x 128, 16 spectra
// 88 and 78.  Whole calls: 25 Stokes images of
// 64 channels of 128 x 128 5.21 -> 3.66 ms, 64 channels of 512 x 512 with 2048
// antennas 21.75 -> 20.40 ms.
// MODE: kShared; kAntennas: an auto image from the per-antenna auto-correlation grids (Yauto) instead of
// A_pq |W^|^2; kTaper64: a taper whose |W^|^2 leaves FP32's exponents, applied in FP64
enum { kShared, kAntennas, kTaper64 };
template <int N, int M, int P, int MODE>
__global__ void __launch_bounds__(kThreads, 4)
epilogue_kernel(const float *__restrict__ partial, int n_tau, int n_items, int R1, int R2,
                const int *__restrict__ chans, const long long *__restrict__ out_off,
                const float2 *__restrict__ wpow, double wscale, const double *__restrict__ apq_tab, const int *__restrict__ autoint,
                int auto_n, size_t auto_stride,
                const float2 *__restrict__ gains, int A, int C, int T, unsigned flags, float2 *__restrict__ out,
                long long out_stride, const float4 *__restrict__ Yauto, const float4 *__restrict__ twp, int K)
{
    constexpr int NPF = P == 2 ? 4 : 1;          // sums and products per pixel
    constexpr bool AK = MODE == kAntennas;
    constexpr int up = N < M ? M / N : 1, Q1 = N < M ? 1 : N / M, Q = Q1 * Q1, NN = N * N;
    // blockIdx.z = image: it sums time chunks [z n_tau, (z + 1) n_tau) and uses
    // the auto sums and output block of index z (one image unless a series)
    const int img = blockIdx.z;
    partial += static_cast<size_t>(img) * n_tau * n_items * (M * M) * NPF;
    out += img * out_stride;
    const int ci = blockIdx.y;
    const int c = chans[ci];
    const bool autosub = !(flags & EPIC_NO_AUTOSUB);

    __shared__ double red[kThreads / 32][4];
    __shared__ double apq[4];   // XX, YY, Re XY, Im XY (YX = conj XY)
    if (autosub && !AK && !apq_tab)
        auto_reduce<P>(autoint + static_cast<size_t>(img) * auto_n * auto_stride, auto_n, auto_stride, gains, A, c, red, apq);
    // |W^|^2's scale, a power of two, goes into A_pq (not with the taper, where A_pq has the sums' own);
    // by one thread each, since the FP64 pipe does ~2 operations a clock
    constexpr bool taper64 = MODE == kTaper64;
    const bool taper = taper64 || (flags & EPIC_KERNEL_TAPER) != 0;
    __shared__ float2 aqs[4];
    if (!AK && threadIdx.x < NPF) {
        double a = 0;
        if (autosub) a = apq_tab ? apq_tab[(static_cast<size_t>(img) * C + c) * 4 + threadIdx.x] : apq[threadIdx.x];
        aqs[threadIdx.x] = to_pair(taper ? a : a * wscale);
    }
    if (!AK) __syncthreads();
    float2 aq[NPF];
#pragma unroll
    for (int k = 0; k < NPF; k++) aq[k] = AK ? make_float2(0.f, 0.f) : aqs[k];

    const double scale = ((flags & EPIC_MEAN) && T > 0) ? 1.0 / T : 1.0;
    float2 *oc = out + out_off[ci];
    for (int pix = blockIdx.x * kThreads + threadIdx.x; pix < NN; pix += gridDim.x * kThreads) {
        const int i = pix / N, j = pix % N;
        const int ly = (i + N / 2) % N, lx = (j + N / 2) % N;   // (i - N/2) mod N
        const int hx = lx % Q1, mx = lx / Q1, hy = ly % Q1, my = ly / Q1;
        const int item = ci * Q + hy * Q1 + hx;
        const int px = up * (R1 == 1 ? mx : R2 * (mx % 8) + mx / 8), py = up * (R1 == 1 ? my : R2 * (my % 8) + my / 8);
        const size_t pos = static_cast<size_t>(py) * M + px;
        float2 w = make_float2(0.f, 0.f);
        if constexpr (!AK) w = __ldg(wpow + pix);
        // time chunks added in time order as compensated FP32 (hi, lo) pairs: TwoSum keeps
        // hi + lo equal to the exact running sum up to the roundings of lo, far below FP32
        float2 s[NPF];
#pragma unroll
        for (int k = 0; k < NPF; k++) s[k] = make_float2(0.f, 0.f);
        const float *src0 = partial + (static_cast<size_t>(item) * (M * M) + pos) * NPF;
        const size_t tau_stride = static_cast<size_t>(n_items) * (M * M) * NPF;
#pragma unroll 8
        for (int tau = 0; tau < n_tau; tau++) {
            const float *src = src0 + tau * tau_stride;
            if constexpr (P == 2) {
                const float4 f = __ldg(reinterpret_cast<const float4 *>(src));
                s[0].y += two_sum(s[0].x, f.x);
                s[1].y += two_sum(s[1].x, f.y);
                s[2].y += two_sum(s[2].x, f.z);
                s[3].y += two_sum(s[3].x, f.w);
            } else {
                s[0].y += two_sum(s[0].x, __ldg(src));
            }
        }
        if constexpr (AK) {
            if (autosub) {
                // the auto image sum_{rho_y >= 0} Re(Y(rho_y, l_x) exp(+2 pi i rho_y l_y / N)), in pairs
                const float4 *y = Yauto + static_cast<size_t>(ci) * 4 * K * N + j;   // [4][K][N]
#pragma unroll
                for (int k = 0; k < NPF; k++) {
                    const float4 y0 = __ldg(y + static_cast<size_t>(k) * K * N);
                    s[k].y += two_sum(s[k].x, -y0.x) - y0.y;
                }
                int m = 0;
                for (int ry = 1; ry < K; ry++) {
                    m += ly;
                    if (m >= N) m -= N;
                    const float4 tw = __ldg(twp + m);            // (cos, -sin)
#pragma unroll
                    for (int k = 0; k < NPF; k++) {
                        const float4 yk = __ldg(y + (static_cast<size_t>(k) * K + ry) * N);
                        pair_msub(s[k], make_float2(yk.x, yk.y), make_float2(tw.x, tw.y));
                        pair_msub(s[k], make_float2(yk.z, yk.w), make_float2(tw.z, tw.w));
                    }
                }
            }
        } else {
            if (taper) {
                // point-gridded sums: subtract the bare autos, then apply |W^(l)|^2
#pragma unroll
                for (int k = 0; k < NPF; k++) {
                    float2 d = s[k];
                    d.y += two_sum(d.x, -aq[k].x) - aq[k].y;
                    if constexpr (taper64) {
                        const double x = static_cast<double>(d.x) + static_cast<double>(d.y);
                        s[k] = to_pair(x * (static_cast<double>(w.x) + static_cast<double>(w.y)) * wscale);
                        continue;
                    }
                    const float p = __fmul_rn(d.x, w.x);
                    s[k] = make_float2(p, fmaf(d.x, w.y, fmaf(d.y, w.x, fmaf(d.x, w.x, -p))));
                }
            } else if (autosub) {
#pragma unroll
                for (int k = 0; k < NPF; k++) pair_msub(s[k], aq[k], w);
            }
        }
        if constexpr (P == 2) {
            if (flags & EPIC_STOKES) {
                // I = XX + YY, Q = XX - YY, U = 2 Re XY, V = 2 Im XY
                float2 si = s[0], sq = s[0];
                si.y += two_sum(si.x, s[1].x) + s[1].y;
                sq.y += two_sum(sq.x, -s[1].x) - s[1].y;
                s[0] = si;
                s[1] = sq;
                s[2] = make_float2(2.f * s[2].x, 2.f * s[2].y);
                s[3] = make_float2(2.f * s[3].x, 2.f * s[3].y);
            }
        }
        float r[NPF];
#pragma unroll
        for (int k = 0; k < NPF; k++)
            r[k] = scale == 1.0 ? s[k].x + s[k].y
                                : static_cast<float>((static_cast<double>(s[k].x) + static_cast<double>(s[k].y)) * scale);
        oc[pix] = make_float2(r[0], 0.f);
        if constexpr (P == 2) {
            oc[NN + pix] = make_float2(r[1], 0.f);
            if (flags & EPIC_STOKES) {
                oc[2 * NN + pix] = make_float2(r[2], 0.f);
                oc[3 * NN + pix] = make_float2(r[3], 0.f);
            } else {
                oc[2 * NN + pix] = make_float2(r[2], r[3]);
                oc[3 * NN + pix] = make_float2(r[2], -r[3]);
            }
        }
    }
}

// Per-antenna kernels (Eq. 3's W_a): the a = b terms of F_p F_q^* sum to
// sum_a A_a,pq |W^_a(l)|^2 = sum_rho X_pq(rho) exp(+2 pi i rho.l / N) with the
// auto-correlation grid X_pq(rho) = sum_a A_a,pq B_aa(rho),
// B_aa = W_a (x) W_a^* on the (2K-1)^2 offsets rho (Sec. 2.2's "auto-correlation
// grids from individual antenna voltages").  The real and imaginary parts of A_XY
// make grids of their own, so all four grids are Hermitian, their images real and
// rows rho_y < 0 the conjugates of the others: K rows are enough.  One block per
// (channel, grid): X in FP64, each antenna's weight once, then the l_x half of the
// separable transform, Y(rho_y, l_x) = sum_rho_x X(rho_x, rho_y) exp(+2 pi i rho_x
// l_x / N), doubled for rho_y > 0 and stored as FP32 pairs for the epilogue to
// finish along l_y.  Bound by the FP64 pipe (2 operations a clock and SM), as the
// epilogue was when it summed the 2K - 1 rows of complex grids in FP64: 250 spectra
// of 64 channels of 128 x 128, 256 antennas, 5 x 5 kernels, whole call: 1.575 -> 0.988 ms
// (the two kernels 0.68 -> 0.10).
constexpr int kRhoTile = 512;                    // antennas whose weights are held at once

__global__ void __launch_bounds__(kThreads)
auto_rho_kernel(const int *__restrict__ autoint, const float2 *__restrict__ gains,
                const double2 *__restrict__ bauto, const int *__restrict__ chans, const double2 *__restrict__ tw64,
                int A, int P, int K, int N, int parts, float4 *__restrict__ Y)
{
    extern __shared__ double2 X[];               // [parts][K][R]
    __shared__ double wt[kRhoTile];
    const int R = 2 * K - 1, RR = R * R, KR = K * R;
    const int ci = blockIdx.x, pq = blockIdx.y;  // XX, YY, Re XY, Im XY
    const int c = chans[ci];
    for (int base = 0; base < parts * KR; base += kThreads) {   // (parts > 1: once)
        const int idx = base + threadIdx.x, rho = idx % KR, part = idx / KR;
        double xr = 0, xi = 0;
        for (int a0 = 0; a0 < A; a0 += kRhoTile) {
            const int na = min(kRhoTile, A - a0);
            __syncthreads();
            for (int i = threadIdx.x; i < na; i += kThreads) {
                const size_t ca = static_cast<size_t>(c) * A + a0 + i;
                const int *ia = autoint + ca * 4;
                double gxr = 1, gxi = 0, gyr = 1, gyi = 0;
                if (gains) {
                    const float2 gx = gains[ca * P];
                    gxr = gx.x;
                    gxi = gx.y;
                    if (P == 2) {
                        const float2 gy = gains[ca * P + 1];
                        gyr = gy.x;
                        gyi = gy.y;
                    }
                }
                const double pr = gxr * gyr + gxi * gyi, pi = gxi * gyr - gxr * gyi;
                wt[i] = pq == 0   ? (gxr * gxr + gxi * gxi) * ia[0]
                        : pq == 1 ? (gyr * gyr + gyi * gyi) * ia[1]
                        : pq == 2 ? pr * ia[2] - pi * ia[3]
                                  : pr * ia[3] + pi * ia[2];
            }
            __syncthreads();
            if (idx < parts * KR) {
                const double2 *b = bauto + static_cast<size_t>(a0) * RR + (K - 1) * R + rho;   // rows rho_y >= 0
#pragma unroll 8
                for (int i = part; i < na; i += parts) {
                    const double2 v = __ldg(b + static_cast<size_t>(i) * RR);
                    xr = fma(wt[i], v.x, xr);
                    xi = fma(wt[i], v.y, xi);
                }
            }
        }
        if (idx < parts * KR) X[idx] = make_double2(xr, xi);
    }
    __syncthreads();
    if (parts > 1) {
        for (int rho = threadIdx.x; rho < KR; rho += kThreads) {
            double2 x = X[rho];
            for (int p = 1; p < parts; p++) {
                x.x += X[p * KR + rho].x;
                x.y += X[p * KR + rho].y;
            }
            X[rho] = x;
        }
        __syncthreads();
    }
    for (int e = threadIdx.x; e < K * N; e += kThreads) {
        const int ry = e / N, j = e % N;
        const int lx = j < N / 2 ? j + N / 2 : j - N / 2;       // (j - N / 2) mod N
        double yr = 0, yi = 0;
        int m = ((N - lx) * (K - 1)) % N;                        // rho_x l_x mod N from rho_x = -(K - 1) on
        for (int rx = 0; rx < R; rx++) {
            const double2 tw = __ldg(tw64 + m), x = X[ry * R + rx];
            yr = fma(-x.y, tw.y, fma(x.x, tw.x, yr));
            yi = fma(x.y, tw.x, fma(x.x, tw.y, yi));
            m += lx;
            if (m >= N) m -= N;
        }
        const double f = ry ? 2.0 : 1.0;
        const float2 re = to_pair(f * yr), im = to_pair(f * yi);
        Y[((static_cast<size_t>(ci) * 4 + pq) * K + ry) * N + j] = make_float4(re.x, re.y, im.x, im.y);
    }
}

// The instantiation for a grid side, its folded side and the polarisations
template <class F>
int epi_dispatch(int N, int M, int P, F &&f)
{
    auto with_p = [&](auto n_, auto m_) {
        return P == 2 ? f(n_, m_, std::integral_constant<int, 2>{}) : f(n_, m_, std::integral_constant<int, 1>{});
    };
    auto side = [&](auto n_, auto m_) { return with_p(n_, m_); };
#define EPI_SIDE(n, m) \
    if (N == n && M == m) return side(std::integral_constant<int, n>{}, std::integral_constant<int, m>{})
    EPI_SIDE(32, 32);
    EPI_SIDE(32, 64);
    EPI_SIDE(64, 64);
    EPI_SIDE(96, 48);
    EPI_SIDE(128, 64);
    EPI_SIDE(256, 64);
    EPI_SIDE(512, 64);
#undef EPI_SIDE
    return EPIC_ERR_UNSUPPORTED;
}


// n_img images of n_tau time chunks each
int launch_epi(epic_plan_s *plan, const GroupCfg &g, const float2 *gains, int T, int n_tau, int n_img, float2 *out,
               cudaStream_t stream)
{
    return epi_dispatch(g.N, g.M, plan->P, [&](auto n_, auto m_, auto p_) {
        constexpr int N = decltype(n_)::value, M = decltype(m_)::value, P = decltype(p_)::value;
        const dim3 grid(static_cast<unsigned>(epi_tiles(N, P, g.n_chan * n_img, plan->sm_count)), static_cast<unsigned>(g.n_chan),
                        static_cast<unsigned>(n_img));
        const auto kfn = plan->nker > 1                                                    ? epilogue_kernel<N, M, P, kAntennas>
                         : (plan->flags & EPIC_KERNEL_TAPER) && g.wscale != 1.0 ? epilogue_kernel<N, M, P, kTaper64>
                                                                                : epilogue_kernel<N, M, P, kShared>;
        kfn<<<grid, kThreads, 0, stream>>>(
            g.d_partial, n_tau, g.n_items, g.R1, g.R2, g.d_chans, g.d_out_off, g.d_wpow, g.wscale,
            plan->d_apq, nullptr, 0, 0, gains, plan->A, plan->C, T, plan->flags, out, static_cast<long long>(plan->out_floats / 2),
            g.d_Y, g.d_twp, plan->K);
        return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
    });
}

template <class F>
int auto_dispatch(int P, bool words, F &&f)
{
    if (P == 2) return words ? f(autopower_kernel<2, true>) : f(autopower_kernel<2, false>);
    return words ? f(autopower_kernel<1, true>) : f(autopower_kernel<1, false>);
}

int launch_auto(const uint8_t *v, int T, int C, int A, int P, int chunks, size_t stride, int *autoint, cudaStream_t stream)
{
    const bool words = (A * P) % 4 == 0 && reinterpret_cast<uintptr_t>(v) % 4 == 0;
    const dim3 grid(static_cast<unsigned>(C), static_cast<unsigned>(chunks));
    return auto_dispatch(P, words, [&](auto kfn) {
        kfn<<<grid, 128, 0, stream>>>(v, T, C, A, chunks, stride, autoint);
        return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
    });
}

// Per (t, antenna): the FP64 part of the delay phase, once per integration,
// so the imaging kernels need only FP32 (Sec. 2.2 delay correction).
__global__ void delay_prep_kernel(const double *__restrict__ delays, int n, double f_ref, float4 *__restrict__ tab)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double tau = delays[i];
        double b = f_ref * tau;
        b -= rint(b);
        const float hi = static_cast<float>(tau);
        const float lo = static_cast<float>(tau - static_cast<double>(hi));
        tab[i] = make_float4(static_cast<float>(b), hi, lo, 0.f);
    }
}

}  // namespace

// Pixel tiles: four pixels a thread, one where that would leave SMs without a block (with one polarisation,
// a quarter of the work a pixel, below 1.6 blocks an SM).  One GB300, whole
// calls of 16 spectra, us with four / one: two polarisations, 16 antennas, 128 x 128, 4 channels (64 /
// 256 blocks) 32 / 29, 16 channels (256 / 1024) 39 / 49, 32 channels 57 / 82; one polarisation, 100
// antennas, 64 x 64, 32 channels (128 / 512) 27 / 24, 64 channels 33 / 33, 16 antennas, 128 x 128, 10 channels
// (160 / 640) 33 / 29; two of 512 x 512 (512 / 2048) 41 / 49.
int epi_tiles(int N, int P, int images, int sms)
{
    const int one = (N * N + kThreads - 1) / kThreads, four = (one + 3) / 4;
    return four * images * 5 >= sms * (P == 2 ? 5 : 8) ? four : one;
}

int launch_autopower_raw(const RawImage &r, const uint8_t *v, int sm_count, cudaStream_t stream)
{
    if (r.T == 0) return EPIC_OK;
    const int chunks = std::max(1, std::min((4 * sm_count + r.C - 1) / r.C, r.T));
    return launch_auto(v, r.T, r.C, r.A, r.P, chunks, 0, r.autoint, stream);
}

int launch_epilogue_raw(const RawImage &r, const float2 *gains, float2 *out, int sm_count, cudaStream_t stream)
{
    return epi_dispatch(r.N, r.M, r.P, [&](auto n_, auto m_, auto p_) {
        constexpr int N = decltype(n_)::value, M = decltype(m_)::value, P = decltype(p_)::value;
        const dim3 grid(static_cast<unsigned>(epi_tiles(N, P, r.C, sm_count)), static_cast<unsigned>(r.C));
        const auto kfn = (r.flags & EPIC_KERNEL_TAPER) && r.wscale != 1.0 ? epilogue_kernel<N, M, P, kTaper64>
                                                                          : epilogue_kernel<N, M, P, kShared>;
        kfn<<<grid, kThreads, 0, stream>>>(r.partial, r.n_tau, r.n_items, 8, M / 8, r.chans, r.out_off, r.wpow, r.wscale, nullptr,
                                           r.autoint, 1, 0, gains, r.A, r.C, r.T, r.flags, out, 0, nullptr, nullptr, 0);
        return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
    });
}

// Time chunks of one integration's auto sums: enough blocks to fill the GPU, at least four samples
// each, few enough that summing them (auto_sum_kernel, one block a channel) stays short.
int auto_chunks(const epic_plan_s *plan, int T)
{
    return std::max(1, std::min({(8 * plan->sm_count + plan->C - 1) / plan->C, T / 4, 32}));
}

// A_pq of n_img images from the auto sums of chunks chunks each
static int launch_auto_sum(epic_plan_s *plan, const float2 *gains, int chunks, int n_img, cudaStream_t stream)
{
    const dim3 grid(static_cast<unsigned>(plan->C), static_cast<unsigned>(n_img));
    const size_t stride = static_cast<size_t>(plan->C) * plan->A * 4;
    if (plan->P == 2) auto_sum_kernel<2><<<grid, kThreads, 0, stream>>>(plan->d_autoint, chunks, stride, gains, plan->A, plan->C, plan->d_apq);
    else auto_sum_kernel<1><<<grid, kThreads, 0, stream>>>(plan->d_autoint, chunks, stride, gains, plan->A, plan->C, plan->d_apq);
    return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

int launch_autopower_series(epic_plan_s *plan, const uint8_t *v, const float2 *gains, int spi, int n_img, cudaStream_t stream)
{
    const size_t stride = static_cast<size_t>(plan->C) * plan->A * 4;
    const int rc = launch_auto(v, spi * n_img, plan->C, plan->A, plan->P, n_img, stride, plan->d_autoint, stream);
    return rc != EPIC_OK ? rc : launch_auto_sum(plan, gains, 1, n_img, stream);
}

int launch_epilogue_series(epic_plan_s *plan, const GroupCfg &g, const float2 *gains, int spi, int n_img, int n_tau,
                           float2 *out, cudaStream_t stream)
{
    return launch_epi(plan, g, gains, spi, n_tau, n_img, out, stream);
}

int launch_delay_prep(epic_plan_s *plan, int T, cudaStream_t stream)
{
    const int n = T * plan->A;
    if (n <= 0) return EPIC_OK;
    const int blocks = std::min((n + kThreads - 1) / kThreads, 4 * plan->sm_count);
    delay_prep_kernel<<<blocks, kThreads, 0, stream>>>(plan->delays, n, plan->f_ref, plan->d_dtab);
    return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

int launch_auto_rho(epic_plan_s *plan, const GroupCfg &g, const float2 *gains, cudaStream_t stream)
{
    const int KR = plan->K * (2 * plan->K - 1), parts = std::max(1, std::min(8, kThreads / KR));
    const dim3 grid(static_cast<unsigned>(g.n_chan), static_cast<unsigned>(plan->P == 2 ? 4 : 1));
    auto_rho_kernel<<<grid, kThreads, sizeof(double2) * parts * KR, stream>>>(
        plan->d_autoint, gains, plan->d_bauto, g.d_chans, g.d_tw64, plan->A, plan->P, plan->K, g.N, parts, g.d_Y);
    return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

int launch_autopower(epic_plan_s *plan, const uint8_t *v, const float2 *gains, int T, cudaStream_t stream)
{
    const size_t n = static_cast<size_t>(plan->C) * plan->A * 4;
    const int chunks = auto_chunks(plan, T);
    if (plan->nker > 1) {   // the per-antenna auto image takes one sum per antenna
        if (cudaMemsetAsync(plan->d_autoint, 0, n * sizeof(int), stream) != cudaSuccess) return EPIC_ERR_CUDA;
        return T == 0 ? EPIC_OK : launch_auto(v, T, plan->C, plan->A, plan->P, chunks, 0, plan->d_autoint, stream);
    }
    const int rc = launch_auto(v, T, plan->C, plan->A, plan->P, chunks, n, plan->d_autoint, stream);
    return rc != EPIC_OK ? rc : launch_auto_sum(plan, gains, chunks, 1, stream);
}

int launch_epilogue(epic_plan_s *plan, const GroupCfg &g, const float2 *gains, int T, int n_tau, float2 *out,
                    cudaStream_t stream)
{
    return launch_epi(plan, g, gains, T, n_tau, 1, out, stream);
}

}  // namespace epic
