// E-field images of the compact kernel's groups (grid sides 64, 96, 128, at most 64 x
// 64 occupied cells): fp32_compact.cu's method up to the column transforms, whose
// outputs are written out as F_p(l, t) instead of being squared and summed.
//
// Two signals at a time in the halves of packed FP32 pairs (fft32_pair.cuh): both
// polarisations of a sample, or two samples of a single polarisation.  A lane
// holds a column of both, so a warp writes 32 consecutive pixels of each, and
// without time sums to keep the 32-point classes leave room for it.  The
// imaging kernel's lanes hold one polarisation and 16 columns a warp: 0.404 ms
// for 50 spectra of 64 channels of 128 x 128 (840 MB written), 0.311 ms here.  (With
// products this form was the slower one: 3.44 ms against 3.10 for 1000 spectra.)
//
// An origin (x0, y0) other than 0 leaves a factor w_N^{x0 lx + y0 ly} on the
// transform.  The array is placed from the origin's quarter of the grid on
// (efield_place), so that the factor is a power of i and rounds nothing: 1.28e-7
// of the fields' norm in that case, 1.35e-7 with factors from a table (0.319 ms).
// An aperture that is too far off the grid's centre for that takes the table's.
#include <algorithm>
#include <type_traits>

#include "epic_internal.cuh"
#include "fft32_pair.cuh"
#include "tc_ptx.cuh"

namespace epic {
namespace {

constexpr int kES = 65;                      // row stride of G (elements of 16 bytes)
constexpr int kBarFFT = 1, kBarGrid = 2;      // named barriers of the transform and the gridding warps
constexpr int kMaxAE = 1024;                  // antennas (10 bits of a list entry)
constexpr uint16_t kNoCell = 0xFFFFu;      // (bit 15 of a cell offset: odd row, not used here)

// Rows of R: whole blocks of eight (pair_load), the last ones zeros.
__host__ __device__ inline int efield_pad(int rows) { return (rows + 7) & ~7; }

// Where the transforms see a channel's occupied cells (rows x cols from (x0, y0)): moved by (dx, dy)
// from the corner, with origins kx N/4 and ky N/4; quarter 0: from the corner, with origin (x0, y0).
struct EfieldPlace {
    int dx, dy, kx, ky, quarter;
};
__host__ __device__ inline EfieldPlace efield_place(int N, int rows, int cols, int x0, int y0)
{
    auto axis = [N](int at, int n, int &d, int &k) {
        k = at >= N / 4 && at - N / 4 + n <= 64;
        d = at - k * (N / 4);
        return d + n <= 64;
    };
    EfieldPlace p{};
    p.quarter = axis(x0, cols, p.dx, p.kx) && axis(y0, rows, p.dy, p.ky);
    if (!p.quarter) p.dx = p.dy = 0;
    return p;
}

// Byte offsets of the shared-memory regions.
struct EfieldSmem {
    unsigned R, es, gp, taps, tab, total;
};
// pairs: signal pairs per iteration; rows: most rows of G, rrows: of R; taps: the kernels of every
// antenna are staged (nker > 1)
__host__ __device__ inline EfieldSmem efield_smem(int P, int pairs, int N, int rows, int rrows, int A, int K, int nker,
                                                    bool taps, int words)
{
    auto up = [](unsigned b) { return (b + 15u) & ~15u; };
    EfieldSmem s;
    s.R = static_cast<unsigned>(pairs * rows * kES) * 16u;
    s.es = s.R + static_cast<unsigned>(pairs * efield_pad(rrows)) * (N + 1) * 16u;
    s.gp = s.es + 2u * pairs * A * 16u;
    s.taps = s.gp + up(static_cast<unsigned>(A * P) * 8u);
    s.tab = s.taps + (nker > 1 ? (taps ? up(static_cast<unsigned>(nker * K * K) * 8u) : 0u)
                               : static_cast<unsigned>(K * (K + 1) + 1) * 8u * 16u);
    s.total = s.tab + up(static_cast<unsigned>(words) * 2u);
    return s;
}

template <int Q, int P, int PAIRS>
struct EfieldShape {
    static constexpr int N = 32 * Q;
    static constexpr int SPI = PAIRS * (P == 1 ? 2 : 1);       // samples per iteration
    static constexpr int GW = kCompactGatherWarps, FW = 12 - GW;   // gridding and transform warps
    static constexpr int FT = 32 * FW, GT = 32 * GW;
    static constexpr int TASKS = PAIRS * Q * Q;                // column tasks per iteration: 32 columns, one class
    static constexpr int SL = (TASKS + FW - 1) / FW;           // column tasks of a warp
    static constexpr int KA = (kMaxAE + GT - 1) / GT;          // antennas a gridding thread unpacks
};
constexpr int kEThreads = 384;

// staged: bit 0 the gather lists, bit 1 the antennas' kernels (AK) are in shared memory; rmax and
// rrows: most rows of G and of R
template <int Q, int P, int PAIRS, bool AK>
__global__ void __launch_bounds__(kEThreads, 1)
efield_kernel(const uint8_t *__restrict__ v, const float2 *__restrict__ gains, const float2 *__restrict__ kern,
                    int K, const int *__restrict__ chans, const uint16_t *__restrict__ ltab,
                    const int2 *__restrict__ lidx, const int4 *__restrict__ lchan, int A, int C, int T, int n_chan,
                    int n_tau, int rmax, int rrows, int staged, const float2 *__restrict__ twN, float2 *__restrict__ ef_out,
                    const long long *__restrict__ ef_off, long long ef_stride, int *__restrict__ status,
                    long long wait_budget)
{
    using S = EfieldShape<Q, P, PAIRS>;
    constexpr int N = S::N, RS = N + 1, SPI = S::SPI;
    extern __shared__ __align__(16) unsigned char smem_c[];
    // G holds a sample (gridding warps arrive); G has been read, R has been read (transform warps)
    __shared__ __align__(8) uint64_t bar_full, bar_free, bar_read;
    const int AP = A * P, KK = K * K, TPN = K * (K + 1);
    const EfieldSmem L = efield_smem(P, PAIRS, N, rmax, rrows, A, K, AK ? A : 1, (staged & 2) != 0, 0);
    float4 *G = reinterpret_cast<float4 *>(smem_c);              // [PAIRS][rmax][65]: (re a, re b, im a, im b)
    float4 *R = reinterpret_cast<float4 *>(smem_c + L.R);        // [PAIRS][padded rrows][N + 1]
    float4 *es = reinterpret_cast<float4 *>(smem_c + L.es);      // [2][PAIRS][A]
    float2 *gp = reinterpret_cast<float2 *>(smem_c + L.gp);      // [A P]
    float4 *tw2 = reinterpret_cast<float4 *>(smem_c + L.taps);   // [K (K + 1) + 1][8 copies] (one kernel)
    uint16_t *stab = reinterpret_cast<uint16_t *>(smem_c + L.tab);
    const float2 *tapw = staged & 2 ? reinterpret_cast<const float2 *>(smem_c + L.taps) : kern;   // [A][K K] (AK)
    const int gplane = rmax * kES, rplane = efield_pad(rrows) * RS;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ci = blockIdx.x % n_chan, tau = blockIdx.x / n_chan;
    const int c = chans[ci];
    const int t0 = static_cast<int>(static_cast<long long>(T) * tau / n_tau);
    const int t1 = static_cast<int>(static_cast<long long>(T) * (tau + 1) / n_tau);
    const int4 ch = lchan[2 * ci];                               // (block start, block words, rows, columns)
    const int rows = ch.z, cols = ch.w;
    const int4 org = lchan[2 * ci + 1];                          // (x0, y0, -, -)
    EfieldPlace pl = efield_place(N, rows, cols, org.x, org.y);
    if (pl.dy + rows > rrows) pl = EfieldPlace{};                // no room for the moved rows

    if (tid == 0) {
        tc::mbar_init(&bar_full, S::GW);
        tc::mbar_init(&bar_free, S::FW);
        tc::mbar_init(&bar_read, S::FW);
        tc::fence_mbar_init();
    }
    // ---- set-up: a zero G (the cells no list names stay zero), zeros before and past R's rows, gains, taps, lists
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = tid; i < PAIRS * gplane; i += kEThreads) G[i] = zero4;
    const int ry = pl.dy, rpad = (efield_pad(ry + rows) - rows) * RS;
    for (int i = tid; i < PAIRS * rpad; i += kEThreads)
        R[(i / rpad) * rplane + (i % rpad < ry * RS ? 0 : rows * RS) + i % rpad] = zero4;
    for (int i = tid; i < AP; i += kEThreads)
        gp[i] = gains ? gains[static_cast<size_t>(c) * AP + i] : make_float2(1.f, 0.f);
    if constexpr (AK) {
        if (staged & 2)
            for (int i = tid; i < A * KK; i += kEThreads) reinterpret_cast<float2 *>(smem_c + L.taps)[i] = kern[i];
    } else {
        // tap pairs (w(dy, dxl), w(dy, dxl + 1)), zero outside the footprint row; eight interleaved
        // copies, so the eight lanes of one 16-byte request never share a bank group; the last slot
        // is zero, for the lists' empty steps
        for (int i = tid; i < 8 * (TPN + 1); i += kEThreads) {
            const int tp = i >> 3, dyi = tp / (K + 1), j = tp % (K + 1);
            float2 w[2];
            for (int u = 0; u < 2; u++) {
                const int dx = j - 1 + u;
                w[u] = (tp < TPN && dx >= 0 && dx < K) ? kern[dyi * K + dx] : make_float2(0.f, 0.f);
            }
            tw2[i] = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
        }
    }
    if (staged & 1)
        for (int i = tid; i < ch.y; i += kEThreads) stab[i] = __ldg(ltab + ch.x + i);
    __syncthreads();
    // Waits are bounded: a warp whose wait runs out records it and waits no more, so the block ends
    // (its output undefined) and nothing hangs.
    bool dead = false;
    auto wait = [&](uint64_t &bar, uint32_t parity) {
        if (!dead && !tc::mbar_wait(&bar, parity, wait_budget)) {
            dead = true;
            atomicOr(status, kStatusTimeout);
        }
    };
    auto arrive = [&](uint64_t &bar) {   // one arrival a warp
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar);
    };
    if (warp < S::FW) {
        // ================ transforms
        const int rb = (rows + 31) >> 5, nbx = (pl.dx + cols + 7) >> 3, nby = (ry + rows + 7) >> 3;
        const int n_row = PAIRS * Q * rb;
        const int last_k = (S::TASKS - 1 - warp) / S::FW;        // the warp's last column task (TASKS - 1 < warp: none)
        uint32_t ph = 0;
        for (int t = t0; t < t1; t += SPI, ph ^= 1u) {
            wait(bar_full, ph);                                  // G holds sample t
            if (warp >= n_row) arrive(bar_free);
            bool r_free = t == t0;
            for (int task = warp; task < n_row; task += S::FW) {
                const int h = task % Q, y = ((task / Q) % rb) * 32 + lane, pr = task / (Q * rb);
                const bool ok = y < rows;
                float2 xr[32], xi[32];
                pair_load<Q, 1>(xr, xi, G + pr * gplane + (ok ? y : 0) * kES, nbx, h);
                if (task + S::FW >= n_row) arrive(bar_free);     // this warp has read G
                pair_turn<Q>(xr, xi, nbx, h);
                float4 *dst = R + pr * rplane + (ry + y) * RS + h;
                if (!r_free) {
                    wait(bar_read, ph ^ 1u);                     // the columns of the sample before have been read
                    r_free = true;
                }
                pair_fft32(xr, xi, [&](int k1, auto &r, auto &i) {
                    if (ok) {
#pragma unroll
                        for (int k2 = 0; k2 < 4; k2++)
                            dst[Q * (k1 + 8 * k2)] = make_float4(r[k2].x, r[k2].y, i[k2].x, i[k2].y);
                    }
                });
            }
            if (!r_free) wait(bar_read, ph ^ 1u);
            tc::named_bar_sync(kBarFFT, S::FT);                  // R is complete
            if (warp >= S::TASKS) arrive(bar_read);
#pragma unroll 1
            for (int k = 0; k < S::SL; k++) {
                const int task = warp + k * S::FW;
                if (task >= S::TASKS) break;
                // (where a round of tasks holds whole blocks the class shifts by k, so that a warp's classes differ)
                const int h = (S::FW % Q ? task : task + k) % Q, col = ((task / Q) % Q) * 32 + lane, pr = task / (Q * Q);
                float2 xr[32], xi[32];
                pair_load<Q, RS>(xr, xi, R + pr * rplane + col, nby, h);
                if (k == last_k) arrive(bar_read);
                pair_turn<Q>(xr, xi, nby, h);
                // F(l) of the placed array times the origin's factor, on the shifted layout
                const long long NN = static_cast<long long>(N) * N;
                const int ta = P == 2 ? t + pr : t + 2 * pr;
                float2 *dst = ef_out + static_cast<long long>(ta) * ef_stride + ef_off[ci] +
                              (col >= N / 2 ? col - N / 2 : col + N / 2);
                float2 *dst_b = dst + (P == 2 ? NN : ef_stride);   // Y, or the next sample
                const bool ok_a = ta < t1, ok_b = P == 2 ? ok_a : ta + 1 < t1;
                pair_fft32(xr, xi, [&](int k1, auto &r, auto &i) {
                    // i^{kx lx + ky ly}, the same for the four k2 (8 Q is a multiple of 4)
                    const int e = pl.kx * col + pl.ky * (Q * k1 + h);
                    const float s = e & 2 ? -1.f : 1.f;
                    float2 w = e & 1 ? make_float2(0.f, s) : make_float2(s, 0.f);
#pragma unroll
                    for (int k2 = 0; k2 < 4; k2++) {
                        const int ly = Q * (k1 + 8 * k2) + h;
                        if (!pl.quarter) w = __ldg(twN + (org.x * col + org.y * ly) % N);
                        pair_mul(r[k2], i[k2], make_float2(w.x, w.x), make_float2(w.y, w.y), make_float2(-w.y, -w.y));
                        const long long o = static_cast<long long>(ly >= N / 2 ? ly - N / 2 : ly + N / 2) * N;
                        if (ok_a) dst[o] = make_float2(r[k2].x, i[k2].x);
                        if (ok_b) dst_b[o] = make_float2(r[k2].y, i[k2].y);
                    }
                });
            }
        }
    } else {
        // ================ unpack, calibrate, grid
        const int gt = tid - S::FT, gw = warp - S::FW;
        const int2 my = lidx[ci * S::GW + gw];                   // (first batch, batches)
        const bool two = P == 2 && (reinterpret_cast<uintptr_t>(v) & 1) == 0;   // an antenna's two bytes at once
        // antennas gt, gt + GT, ..: the bytes of both signals (polarisations, or samples t and t + 1)
        uint32_t pre[PAIRS][S::KA];
        auto prefetch = [&](int t) {
#pragma unroll
            for (int pr = 0; pr < PAIRS; pr++) {
                const int ta = P == 2 ? t + pr : t + 2 * pr;
                const uint8_t *row = v + (static_cast<size_t>(ta) * C + c) * AP;
#pragma unroll
                for (int k = 0; k < S::KA; k++) {
                    const int a = gt + k * S::GT;
                    pre[pr][k] = 0u;                             // an absent sample: zeros
                    if (a < A && ta < t1) {
                        if constexpr (P == 2) {
                            pre[pr][k] = two ? __ldg(reinterpret_cast<const uint16_t *>(row) + a)
                                             : __ldg(row + 2 * a) | static_cast<uint32_t>(__ldg(row + 2 * a + 1)) << 8;
                        } else {
                            pre[pr][k] = __ldg(row + a);
                            if (ta + 1 < t1) pre[pr][k] |= static_cast<uint32_t>(__ldg(row + static_cast<size_t>(C) * A + a)) << 8;
                        }
                    }
                }
            }
        };
        auto unpack = [&](int buf) {
#pragma unroll
            for (int pr = 0; pr < PAIRS; pr++) {
                float4 *dst = es + (buf * PAIRS + pr) * A;
#pragma unroll
                for (int k = 0; k < S::KA; k++) {
                    const int a = gt + k * S::GT;
                    if (a >= A) break;
                    const float2 ga = gp[a * P], gb = P == 2 ? gp[a * P + 1] : ga;
                    float2 ea = cmul(ga, ci4_decode(pre[pr][k])), eb = cmul(gb, ci4_decode(pre[pr][k] >> 8));
                    dst[a] = make_float4(ea.x, eb.x, ea.y, eb.y);
                }
            }
        };
        // gather of the warp's batches: [d][32 left-cell offsets, 0xFFFF: empty lane]
        // [d x 32 entries tp << 10 | a]; empty steps name the zero tap slot
        auto gather = [&](int buf) {
            const uint16_t *bt = (staged & 1 ? stab : ltab + ch.x) + my.x;
            auto ld = [](const uint16_t *q) -> uint32_t { return *q; };   // shared or global
            const float4 *e0 = es + buf * PAIRS * A;
            const uint32_t empty = static_cast<uint32_t>(TPN) << 10;
            const float4 *tw8 = tw2 + (lane & 7);
            auto taps = [&](uint32_t en) -> float4 {
                if constexpr (AK) {
                    const int tp = static_cast<int>(en >> 10), a = static_cast<int>(en & 1023u);
                    const int dyi = tp / (K + 1), dxl = tp - dyi * (K + 1) - 1;
                    const float2 *wrow = tapw + a * KK + dyi * K;
                    const float2 w0 = dyi < K && dxl >= 0 ? wrow[dxl] : make_float2(0.f, 0.f);
                    const float2 w1 = dyi < K && dxl + 1 < K ? wrow[dxl + 1] : make_float2(0.f, 0.f);
                    return make_float4(w0.x, w0.y, w1.x, w1.y);
                } else {
                    return tw8[(en >> 10) << 3];
                }
            };
            struct Volt {
                float4 e[PAIRS];
            };
            auto volts = [&](uint32_t en) {
                Volt x;
#pragma unroll
                for (int pr = 0; pr < PAIRS; pr++) x.e[pr] = e0[pr * A + (en & 1023u)];
                return x;
            };
            int d = 0;
            uint32_t off = kNoCell, ea = empty;
            if (my.y > 0) {
                d = static_cast<int>(ld(bt));
                off = ld(bt + 1 + lane);
                ea = ld(bt + 33 + lane);
            }
            for (int b = 0; b < my.y; b++) {
                const uint16_t *ent = bt + 33 + lane;
                const uint16_t *nbt = bt + 33 + 32 * d;
                int dn = 0;
                uint32_t offn = kNoCell, ean = empty;
                if (b + 1 < my.y) {                              // the next batch's header, a batch ahead
                    dn = static_cast<int>(ld(nbt));
                    offn = ld(nbt + 1 + lane);
                    ean = ld(nbt + 33 + lane);
                }
                float4 acc[PAIRS][2];
#pragma unroll
                for (int pr = 0; pr < PAIRS; pr++) acc[pr][0] = acc[pr][1] = zero4;
                // entries two steps ahead, taps and voltages one step ahead
                uint32_t en1 = d > 1 ? ld(ent + 32) : empty;
                float4 ww = taps(ea);
                Volt ee = volts(ea);
#pragma unroll 2
                for (int j = 0; j < d; j++) {
                    const uint32_t en2 = j + 2 < d ? ld(ent + (j + 2) * 32) : empty;
                    const float4 wwn = taps(en1);
                    const Volt een = volts(en1);
                    const float wr[2] = {ww.x, ww.z}, wi[2] = {ww.y, ww.w};
#pragma unroll
                    for (int pr = 0; pr < PAIRS; pr++)
#pragma unroll
                        for (int u = 0; u < 2; u++) {
                            const float4 e = ee.e[pr];
                            float4 &o = acc[pr][u];
                            o.x = fmaf(-wi[u], e.z, fmaf(wr[u], e.x, o.x));
                            o.y = fmaf(-wi[u], e.w, fmaf(wr[u], e.y, o.y));
                            o.z = fmaf(wi[u], e.x, fmaf(wr[u], e.z, o.z));
                            o.w = fmaf(wi[u], e.y, fmaf(wr[u], e.w, o.w));
                        }
                    ww = wwn;
                    ee = een;
                    en1 = en2;
                }
                if (off != kNoCell) {
#pragma unroll
                    for (int pr = 0; pr < PAIRS; pr++)
#pragma unroll
                        for (int u = 0; u < 2; u++) G[pr * gplane + pl.dx + (off & 0x7FFFu) + u] = acc[pr][u];
                }
                bt = nbt;
                d = dn;
                off = offn;
                ea = ean;
            }
        };
        int buf = 0;
        if (t0 < t1) {
            prefetch(t0);
            unpack(0);
            prefetch(t0 + SPI);
            tc::named_bar_sync(kBarGrid, S::GT);
            gather(0);
            arrive(bar_full);
        }
        uint32_t ph = 0;
        for (int t = t0; t + SPI < t1; t += SPI, ph ^= 1u) {
            buf ^= 1;
            unpack(buf);
            prefetch(t + 2 * SPI);
            tc::named_bar_sync(kBarGrid, S::GT);                 // the sample's voltages are complete
            wait(bar_free, ph);                                  // the row transforms hold G(t)
            gather(buf);
            arrive(bar_full);
        }
    }
}

// signal pairs per iteration: two at side 64 (samples, to fill the transform warps), else one
constexpr int efield_pairs(int N, int P) { return N == 64 && P == 2 ? 2 : 1; }

template <int V>
using IC = std::integral_constant<int, V>;

// The instantiation that serves a group: grid side, polarisations, signal pairs per iteration.
template <class F>
int efield_dispatch(const GroupCfg &g, int P, F &&f)
{
    auto with_p = [&](auto p_) {
        if (g.N == 128) return f(IC<4>{}, p_, IC<1>{});
        if (g.N == 96) return f(IC<3>{}, p_, IC<1>{});
        return f(IC<2>{}, p_, IC<efield_pairs(64, decltype(p_)::value)>{});
    };
    return P == 2 ? with_p(IC<2>{}) : with_p(IC<1>{});
}

template <int Q, int P, int PAIRS, bool AK>
int launch_efield_t(epic_plan_s *plan, const GroupCfg &g, const uint8_t *v, const float2 *gains, int T, int n_tau,
                    float2 *out, long long stride, cudaStream_t stream)
{
    const EfieldSmem L = efield_smem(P, PAIRS, g.N, g.crows, g.erows, plan->A, plan->K, plan->nker, g.etaps, g.estage ? g.cwords : 0);
    efield_kernel<Q, P, PAIRS, AK><<<static_cast<unsigned>(g.n_chan * n_tau), kEThreads, L.total, stream>>>(
        v, gains, plan->d_kernel, plan->K, g.d_chans, g.d_ltab, g.d_lidx, g.d_lchan, plan->A, plan->C, T, g.n_chan, n_tau,
        g.crows, g.erows, (g.estage ? 1 : 0) | (g.etaps ? 2 : 0), g.d_twN, out, g.d_ef_off, stride, plan->d_status, plan->wait_budget);
    return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

}  // namespace

size_t efield_smem_bytes(int N, int P, int rows, int rrows, int A, int K, int nker, bool taps, int words)
{
    return efield_smem(P, efield_pairs(N, P), N, rows, rrows, A, K, nker, taps, words).total;
}

int efield_rows(int N, const std::vector<int4> &lchan)
{
    int most = 0;
    for (size_t i = 0; i < lchan.size(); i += 2)
        most = std::max(most, lchan[i].z + efield_place(N, lchan[i].z, lchan[i].w, lchan[i + 1].x, lchan[i + 1].y).dy);
    return most;
}

// A CTA here transforms all classes of a sample one after the other
// where the per-class kernel has a CTA for each.  Where those find room on the SMs at
// once (a CTA takes one sample, or two of one polarisation) the call is its latency.  One GB300, us per
// class / here: side 128, two polarisations, 4 channels x 8 spectra (128 CTAs) 12.3 / 18.4, 4 x 12 (192) 15.4
// / 18.5, 8 x 8 with 1000 antennas (256) 35 / 39, 5 x 14 (280) 14.4 / 18.5,
// 4 x 20 (320) 22.5 / 18.5, 64 x 2 (512) 28.7 / 20.5; one, 4
// x 8 (64) 10.3 / 16.4, 16 x 8 (256) 16.4 / 18.5, 64 x 2 (256 in one sample's classes) 20.7 / 18.5; side
// 96, two, 4 x 12 14.4 / 15.4, 4 x 20 19.5 / 16.0.  At side 64 this kernel is not the slower one.
bool efield_per_class(int N, int P, int n_items, int T, int sms)
{
    const long long ctas = static_cast<long long>(n_items) * (P == 1 ? (T + 1) / 2 : T);
    return (N == 96 || N == 128) && n_items <= sms && ctas <= 2LL * sms;
}

// Whether a plan keeps the per-class tables for such calls: for few channels, where they cost little, and
// where its longest call is one (37 channels at three sides, 16 ms of plan, would pay 2 ms for them).
bool efield_tables(int N, int P, int n_items, int max_spectra, int sms)
{
    return efield_per_class(N, P, n_items, n_items <= 16 ? 1 : std::max(1, max_spectra), sms);
}

int prepare_efield(const epic_plan_s *plan, const GroupCfg &g)
{
    const size_t need = efield_smem_bytes(g.N, plan->P, g.crows, g.erows, plan->A, plan->K, plan->nker, g.etaps, g.estage ? g.cwords : 0);
    return efield_dispatch(g, plan->P, [&](auto q_, auto p_, auto pr_) {
        constexpr int Q = decltype(q_)::value, P = decltype(p_)::value, PAIRS = decltype(pr_)::value;
        return plan->nker > 1 ? raise_dyn_smem_cap(reinterpret_cast<const void *>(efield_kernel<Q, P, PAIRS, true>), need)
                              : raise_dyn_smem_cap(reinterpret_cast<const void *>(efield_kernel<Q, P, PAIRS, false>), need);
    });
}

int launch_compact_efield(epic_plan_s *plan, const GroupCfg &g, const uint8_t *v, const float2 *gains, int T,
                          float2 *out, long long stride, cudaStream_t stream)
{
    const int n_tau = g.cimage ? choose_tau(plan, g, T) : compact_pick_tau(g.n_chan, g.n_items, T, plan->sm_count);
    return efield_dispatch(g, plan->P, [&](auto q_, auto p_, auto pr_) {
        constexpr int Q = decltype(q_)::value, P = decltype(p_)::value, PAIRS = decltype(pr_)::value;
        return plan->nker > 1 ? launch_efield_t<Q, P, PAIRS, true>(plan, g, v, gains, T, n_tau, out, stride, stream)
                              : launch_efield_t<Q, P, PAIRS, false>(plan, g, v, gains, T, n_tau, out, stride, stream);
    });
}

}  // namespace epic
