// E-field-domain gain solver for one calibrator (the feedback calibration Sec. 1
// cites for EPIC, and the real-time calibration Sec. 5 names as future work).
// Per (channel, polarisation), from unit gains, n_iter times:
//
//   E(t) = (1/A) sum_a g_a e_a(t) conj(phi_a)              the calibrator field
//   g_a  = phi_a sum_t E(t) conj(e_a(t)) / sum_t |e_a(t)|^2  per-antenna least squares
//   then antenna 0's phase -> 0 and the RMS |g| -> 1
//
// phi_a = exp(-2 pi i (kx_a lx + ky_a ly) / N) for a source at the image offset
// (lx, ly) = (l N du, m N du) pixels (a source there has e_a ~ phi_a and appears
// at +(lx, ly) in the image).
//
// gain_solve_cluster_kernel (n_ant n_pol <= 1024, but for the shortest calls): one thread-block cluster per channel, each CTA
// a share of the samples.  A warp takes a sample at a time: its lanes hold the row's voltages
// (words lane, lane + 32, ..), form E(t) of both polarisations by one warp reduction and add
// E conj(e) to the sums of their own antennas in registers, so an iteration reads the voltages
// once.  The CTAs' sums meet through distributed shared memory: each CTA finishes a slice of the
// antennas and hands its gains to the others, so there is no workspace and one launch.  Bound by
// issue and latency (about 20 instructions a voltage and iteration; 40 % issue).  256 antennas, 64 channels, two
// polarisations, 1000 spectra, two iterations: 91 us, against 322 us for one CTA per channel and
// polarisation, whose loads' latency was the limit.
// gain_solve_kernel (larger arrays, short calls): one CTA per (channel, polarisation), E(t) of all samples in
// shared memory, the voltages read twice per iteration.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include <cooperative_groups.h>

#include "dft_small.cuh"
#include "epic_internal.cuh"

namespace epic {
namespace {

constexpr int kCalThreads = 256;

__device__ __forceinline__ float block_sum(float x, float *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    float s = 0.f;
    for (int w = 0; w < kCalThreads / 32; w++) s += red[w];
    return s;
}

__global__ void __launch_bounds__(kCalThreads)
gain_solve_kernel(const uint8_t *__restrict__ v, const short2 *__restrict__ cells, const int *__restrict__ chans,
                  int A, int C, int P, int T, int N, double lx, double ly, int n_iter, float2 *__restrict__ gains)
{
    extern __shared__ float2 sm[];
    float2 *phi = sm;                        // [A]
    float2 *g = phi + A;                     // [A]
    float2 *E = g + A;                       // [T]
    int *den = reinterpret_cast<int *>(E + T);   // [A] exact sum_t |e_a(t)|^2
    __shared__ float red[kCalThreads / 32];
    __shared__ float2 ref;
    const int c = chans[blockIdx.x / P], p = blockIdx.x % P;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto byte = [&](int t, int a) {
        return static_cast<uint32_t>(__ldg(v + ((static_cast<size_t>(t) * C + c) * A + a) * P + p));
    };

    for (int a = tid; a < A; a += kCalThreads) {
        const short2 k = cells[static_cast<size_t>(c) * A + a];
        double turns = (static_cast<double>(k.x) * lx + static_cast<double>(k.y) * ly) / N;
        turns -= rint(turns);
        double s, co;
        sincospi(-2.0 * turns, &s, &co);
        phi[a] = make_float2(static_cast<float>(co), static_cast<float>(s));
        g[a] = make_float2(1.f, 0.f);
        int acc = 0;
#pragma unroll 8
        for (int t = 0; t < T; t++) {
            const float2 e = ci4_decode(byte(t, a));
            acc += static_cast<int>(e.x * e.x + e.y * e.y);
        }
        den[a] = acc;
    }
    __syncthreads();

    const float invA = 1.f / static_cast<float>(A);
    for (int it = 0; it < n_iter; it++) {
        // E(t) = (1/A) sum_a g_a conj(phi_a) e_a(t): one warp per sample
        for (int t = warp; t < T; t += kCalThreads / 32) {
            float2 acc = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int a = lane; a < A; a += 32) {
                const float2 w = cmul(g[a], make_float2(phi[a].x, -phi[a].y));
                const float2 e = ci4_decode(byte(t, a));
                acc.x = fmaf(w.x, e.x, fmaf(-w.y, e.y, acc.x));
                acc.y = fmaf(w.x, e.y, fmaf(w.y, e.x, acc.y));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            }
            if (lane == 0) E[t] = make_float2(acc.x * invA, acc.y * invA);
        }
        __syncthreads();
        // g_a = phi_a sum_t E(t) conj(e_a(t)) / sum_t |e_a(t)|^2
        for (int a = tid; a < A; a += kCalThreads) {
            float2 num = make_float2(0.f, 0.f);
#pragma unroll 8
            for (int t = 0; t < T; t++) {
                const float2 e = ci4_decode(byte(t, a));
                const float2 x = E[t];
                num.x = fmaf(x.x, e.x, fmaf(x.y, e.y, num.x));    // x conj(e)
                num.y = fmaf(x.y, e.x, fmaf(-x.x, e.y, num.y));
            }
            g[a] = den[a] > 0 ? cscale(cmul(phi[a], num), 1.f / static_cast<float>(den[a])) : make_float2(0.f, 0.f);
        }
        __syncthreads();
        // antenna 0's phase to zero, then RMS amplitude to one
        if (tid == 0) {
            const float2 g0 = g[0];
            const float r = sqrtf(g0.x * g0.x + g0.y * g0.y);
            ref = r > 0.f ? make_float2(g0.x / r, -g0.y / r) : make_float2(1.f, 0.f);
        }
        float ss = 0.f;
        for (int a = tid; a < A; a += kCalThreads) ss += g[a].x * g[a].x + g[a].y * g[a].y;
        ss = block_sum(ss, red);
        const float rms = sqrtf(ss * invA);
        const float sc = rms > 0.f ? 1.f / rms : 1.f;
        for (int a = tid; a < A; a += kCalThreads) g[a] = cscale(cmul(g[a], ref), sc);
        __syncthreads();
    }
    for (int a = tid; a < A; a += kCalThreads) gains[(static_cast<size_t>(c) * A + a) * P + p] = g[a];
}

constexpr int kCalWarps = kCalThreads / 32;

// Bytes 2 k and 2 k + 1 of four 4+4-bit voltages x (as ci4_decode) as pairs (re, re), (im, im): with the
// sign bits flipped a nibble is n + 8 in 0..15; or-ed into the mantissa of 2^23 at bit s it reads
// 2^23 + (n + 8) 2^s, and one packed FMA takes the offsets and the scales away, exactly.
struct Ci4Pair {
    float2 re, im;
};
__device__ __forceinline__ Ci4Pair ci4_pair(uint32_t x, int k)
{
    const uint32_t y = (k ? x >> 16 : x) ^ 0x8888u;
    auto bits = [&](int s) { return __uint_as_float((y & (0xFu << s)) | 0x4B000000u); };
    constexpr float o0 = -(8388608.f + 8.f), o4 = -(8388608.f / 16.f + 8.f), o8 = -(8388608.f / 256.f + 8.f),
                    o12 = -(8388608.f / 4096.f + 8.f);
    Ci4Pair e;
    e.re = pfma(make_float2(bits(4), bits(12)), make_float2(1.f / 16.f, 1.f / 4096.f), make_float2(o4, o12));
    e.im = pfma(make_float2(bits(0), bits(8)), make_float2(1.f, 1.f / 256.f), make_float2(o0, o8));
    return e;
}

size_t cal_cluster_smem(int AP)   // sums of every warp, the CTA's sums, gains, phases, sum |e|^2
{
    return sizeof(float2) * static_cast<size_t>(AP) * (kCalWarps + 3) + sizeof(int) * static_cast<size_t>(AP) * (kCalWarps + 2);
}

// grid (cluster size x n_chan); R: words a lane holds of a sample's row (n_ant n_pol <= 128 R)
template <int R>
__global__ void __launch_bounds__(kCalThreads, R <= 4 ? 2 : 1)
gain_solve_cluster_kernel(const uint8_t *__restrict__ v, const short2 *__restrict__ cells, const int *__restrict__ chans,
                          int A, int C, int P, int T, int N, double lx, double ly, int n_iter, float2 *__restrict__ gains)
{
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.barrier_arrive();                             // met before the first store to another CTA's shared memory
    const int rank = static_cast<int>(cl.block_rank()), CL = static_cast<int>(cl.num_blocks());
    extern __shared__ float2 sm[];
    const int AP = A * P;
    float2 *red = sm;                                // [warps][AP]
    float2 *part = red + kCalWarps * AP;             // [AP] the CTA's sums
    float2 *g = part + AP;                           // [AP]
    float2 *phi = g + AP;                            // [AP] (per antenna, repeated per polarisation)
    float *wden = reinterpret_cast<float *>(phi + AP);   // [warps][AP] exact sum |e|^2 of the first iteration
    int *iden = reinterpret_cast<int *>(wden + kCalWarps * AP);   // [AP] the CTA's
    int *den = iden + AP;                            // [AP] over the cluster
    __shared__ float ss_part[2];                     // the CTA's slice of sum |g|^2 per polarisation
    __shared__ float red2[kCalWarps][2];
    __shared__ float2 ref[2];
    __shared__ float scale[2];
    const int c = chans[blockIdx.x / CL];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i0 = static_cast<int>(static_cast<long long>(AP) * rank / CL);
    const int i1 = static_cast<int>(static_cast<long long>(AP) * (rank + 1) / CL);

    // the lattice phases of the CTA's slice, to every CTA of the cluster; another CTA's shared memory may be
    // accessed only once that CTA runs
    cl.barrier_wait();
    for (int i = i0 + tid; i < i1; i += kCalThreads) {
        const short2 k = cells[static_cast<size_t>(c) * A + i / P];
        double turns = (static_cast<double>(k.x) * lx + static_cast<double>(k.y) * ly) / N;
        turns -= rint(turns);
        double s, co;
        sincospi(-2.0 * turns, &s, &co);
        const float2 f = make_float2(static_cast<float>(co), static_cast<float>(s));
        for (int r = 0; r < CL; r++) cl.map_shared_rank(phi, r)[i] = f;
    }
    for (int i = tid; i < AP; i += kCalThreads) {
        g[i] = make_float2(1.f, 0.f);
    }
    cl.sync();

    const bool words = (AP & 3) == 0 && (reinterpret_cast<uintptr_t>(v) & 3) == 0;
    const int step = CL * kCalWarps;
    auto load = [&](int t, uint32_t (&x)[R]) {
        const uint8_t *row = v + (static_cast<size_t>(t) * C + c) * AP;
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int w = lane + 32 * r;
            x[r] = 0u;                               // decodes to zero
            if (t >= T) continue;
            if (words) {
                if (4 * w < AP) x[r] = __ldg(reinterpret_cast<const uint32_t *>(row) + w);
            } else {
#pragma unroll
                for (int b = 0; b < 4; b++)
                    if (4 * w + b < AP) x[r] |= static_cast<uint32_t>(__ldg(row + 4 * w + b)) << (8 * b);
            }
        }
    };
    const float invA = 1.f / static_cast<float>(A);
    // one iteration over the CTA's samples; FIRST adds up |e|^2 as well (FP32 holds these integers
    // exactly: at most 128 a sample, far fewer than 2^17 samples a warp)
    auto sweep = [&](auto first) {
        constexpr bool FIRST = decltype(first)::value;
        // w = g conj(phi) of the lane's values, two bytes (both polarisations, or two antennas) to a packed pair
        float2 wr[R][2], wi[R][2], wn[R][2], nr[R][2], ni[R][2];
        float2 dd[FIRST ? R : 1][2];
        const float2 zero = make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
            for (int k = 0; k < 2; k++) {
                float2 w[2];
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const int i = 4 * (lane + 32 * r) + 2 * k + u;
                    w[u] = i < AP ? cmul(g[i], make_float2(phi[i].x, -phi[i].y)) : zero;
                }
                wr[r][k] = make_float2(w[0].x, w[1].x);
                wi[r][k] = make_float2(w[0].y, w[1].y);
                wn[r][k] = make_float2(-w[0].y, -w[1].y);
                nr[r][k] = ni[r][k] = zero;
                if (FIRST) dd[r][k] = zero;
            }
        uint32_t x[R], xn[R];
        load(rank * kCalWarps + warp, x);
        for (int t = rank * kCalWarps + warp; t < T; t += step) {
            load(t + step, xn);
            // the halves of a pair: polarisations 0 and 1 (P = 2), or antennas of one polarisation
            float2 er = zero, ei = zero;
#pragma unroll
            for (int r = 0; r < R; r++)
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const Ci4Pair e = ci4_pair(x[r], k);
                    er = pfma(wr[r][k], e.re, pfma(wn[r][k], e.im, er));
                    ei = pfma(wr[r][k], e.im, pfma(wi[r][k], e.re, ei));
                }
            if (P == 1) {
                er = make_float2(er.x + er.y, er.x + er.y);
                ei = make_float2(ei.x + ei.y, ei.x + ei.y);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                er = padd(er, make_float2(__shfl_xor_sync(0xffffffffu, er.x, o), __shfl_xor_sync(0xffffffffu, er.y, o)));
                ei = padd(ei, make_float2(__shfl_xor_sync(0xffffffffu, ei.x, o), __shfl_xor_sync(0xffffffffu, ei.y, o)));
            }
            er = pmul(er, make_float2(invA, invA));
            ei = pmul(ei, make_float2(invA, invA));
            const float2 en = make_float2(-er.x, -er.y);
#pragma unroll
            for (int r = 0; r < R; r++)
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const Ci4Pair e = ci4_pair(x[r], k);
                    nr[r][k] = pfma(er, e.re, pfma(ei, e.im, nr[r][k]));      // E conj(e)
                    ni[r][k] = pfma(ei, e.re, pfma(en, e.im, ni[r][k]));
                    if (FIRST) dd[r][k] = pfma(e.re, e.re, pfma(e.im, e.im, dd[r][k]));
                }
#pragma unroll
            for (int r = 0; r < R; r++) x[r] = xn[r];
        }
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
            for (int k = 0; k < 2; k++)
#pragma unroll
                for (int u = 0; u < 2; u++) {
                    const int i = 4 * (lane + 32 * r) + 2 * k + u;
                    if (i >= AP) continue;
                    red[warp * AP + i] = u ? make_float2(nr[r][k].y, ni[r][k].y) : make_float2(nr[r][k].x, ni[r][k].x);
                    if (FIRST) wden[warp * AP + i] = u ? dd[r][k].y : dd[r][k].x;
                }
    };
    for (int it = 0; it < n_iter; it++) {
        if (it == 0) sweep(std::true_type{});
        else sweep(std::false_type{});
        __syncthreads();
        for (int i = tid; i < AP; i += kCalThreads) {
            float2 s = red[i];
            for (int k = 1; k < kCalWarps; k++) s = cadd(s, red[k * AP + i]);
            part[i] = s;
            if (it == 0) {
                int d = 0;
                for (int k = 0; k < kCalWarps; k++) d += static_cast<int>(wden[k * AP + i]);
                iden[i] = d;
            }
        }
        cl.sync();
        // the CTA's slice: sums over the cluster in rank order, gains before normalisation
        float s0 = 0.f, s1 = 0.f;
        for (int i = i0 + tid; i < i1; i += kCalThreads) {
            float2 s = make_float2(0.f, 0.f);
            int dd = 0;
            for (int r = 0; r < CL; r++) {
                s = cadd(s, cl.map_shared_rank(part, r)[i]);
                if (it == 0) dd += cl.map_shared_rank(iden, r)[i];
            }
            if (it == 0) den[i] = dd;
            else dd = den[i];
            const float2 gi = dd > 0 ? cscale(cmul(phi[i], s), 1.f / static_cast<float>(dd)) : make_float2(0.f, 0.f);
            const float q = gi.x * gi.x + gi.y * gi.y;
            if (P == 2 && (i & 1)) s1 += q;
            else s0 += q;
            for (int r = 0; r < CL; r++) cl.map_shared_rank(g, r)[i] = gi;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        }
        if (lane == 0) {
            red2[warp][0] = s0;
            red2[warp][1] = s1;
        }
        __syncthreads();
        if (tid < 2) {
            float s = 0.f;
            for (int k = 0; k < kCalWarps; k++) s += red2[k][tid];
            ss_part[tid] = s;
        }
        cl.sync();
        // antenna 0's phase to zero, then RMS amplitude to one
        if (tid < P) {
            float s = 0.f;
            for (int r = 0; r < CL; r++) s += cl.map_shared_rank(ss_part, r)[tid];
            const float rms = sqrtf(s * invA);
            scale[tid] = rms > 0.f ? 1.f / rms : 1.f;
            const float2 g0 = g[tid];
            const float r = sqrtf(g0.x * g0.x + g0.y * g0.y);
            ref[tid] = r > 0.f ? make_float2(g0.x / r, -g0.y / r) : make_float2(1.f, 0.f);
        }
        __syncthreads();
        for (int i = tid; i < AP; i += kCalThreads) {
            const int p = P == 2 ? i & 1 : 0;
            g[i] = cscale(cmul(g[i], ref[p]), scale[p]);
        }
        __syncthreads();
    }
    for (int i = i0 + tid; i < i1; i += kCalThreads) gains[static_cast<size_t>(c) * AP + i] = g[i];
    cl.sync();   // no CTA leaves while another may still read its shared memory
}

template <int R>
int launch_cal_cluster(const epic_plan_s *plan, const GroupCfg &g, int cl, const uint8_t *v, int T, double lx, double ly,
                       int n_iter, float2 *gains, cudaStream_t s)
{
    const size_t smem = cal_cluster_smem(plan->A * plan->P);
    const auto kfn = gain_solve_cluster_kernel<R>;
    if (cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(cal_cluster_smem(128 * R))) !=
        cudaSuccess)
        return EPIC_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(g.n_chan * cl));
    cfg.blockDim = dim3(kCalThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = static_cast<unsigned>(cl);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kfn, v, plan->d_cells, g.d_chans, plan->A, plan->C, plan->P, T, g.N, lx, ly, n_iter,
                              gains) == cudaSuccess
               ? EPIC_OK
               : EPIC_ERR_CUDA;
}

}  // namespace

// CTAs of a channel's cluster, or 0 for one CTA per channel and polarisation.  One wave of CTAs (two an SM
// up to 512 values a row, one above), each with at least a sample per warp.  The cluster's barriers and
// gain exchange take about 20 us (30 above 512 values) that short calls do not earn back, nor do long rows of both
// polarisations read by bytes where the clusters come to more than a wave.  One GB300, us one CTA per channel and polarisation / cluster, two iterations:
// 256 antennas x 2, 61 channels, 8 spectra 10 / 21, 20: 14 / 19, 66: 27 / 25; 200 channels, 66: 47 / 47; 34 x 1, 8
// channels, 20: 11 / 12; 512 x 2, 8 channels, 20: 23 / 27, 200 channels, 66: 84 / 98; 297 x 2, 200 channels,
// 1000: 1044 / 1266; 600 x 1, 8 channels, 8: 19 / 25.
int cal_cluster_size(int AP, int P, int n_chan, int T, int sms)
{
    const bool wide = AP > 512, bytes = (AP & 3) != 0 && P == 2;
    int t_min = !wide ? 48 : P == 1 ? 16 : bytes ? 96 : 64;
    if (n_chan > sms) t_min = !wide ? 64 : bytes ? 1 << 30 : 128;
    if (AP > 1024 || T < t_min) return 0;
    int cl = 1;
    while (cl < 8 && 2 * cl * n_chan <= (wide ? 1 : 2) * sms && 2 * cl * kCalWarps <= T) cl *= 2;
    return cl;
}

namespace {

size_t cal_smem(int A, int T) { return sizeof(float2) * (2 * static_cast<size_t>(A) + T) + sizeof(int) * A; }

}  // namespace
}  // namespace epic

extern "C" int epic_solve_gains(epic_plan_t plan, const uint8_t *ci4, int n_spectra, double l, double m, int n_iter,
                                float *gains_out, void *stream)
{
    if (!plan || !ci4 || !gains_out || n_spectra < 1 || n_spectra > plan->max_spectra || n_iter < 1 || n_iter > 64 ||
        !std::isfinite(l) || !std::isfinite(m))
        return EPIC_ERR_ARG;
    const size_t smem = epic::cal_smem(plan->A, n_spectra);
    if (smem > 200 * 1024) return EPIC_ERR_TOO_LARGE;
    if (cudaFuncSetAttribute(epic::gain_solve_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem)) != cudaSuccess)
        return EPIC_ERR_CUDA;
    auto s = static_cast<cudaStream_t>(stream);
    for (const auto &g : plan->groups) {
        const double lx = l * g.N * plan->du, ly = m * g.N * plan->du;
        const int AP = plan->A * plan->P;
        const int cl = epic::cal_cluster_size(AP, plan->P, g.n_chan, n_spectra, plan->sm_count);
        if (cl > 0) {
            auto *out = reinterpret_cast<float2 *>(gains_out);
            const int rc = AP <= 128   ? epic::launch_cal_cluster<1>(plan, g, cl, ci4, n_spectra, lx, ly, n_iter, out, s)
                           : AP <= 256 ? epic::launch_cal_cluster<2>(plan, g, cl, ci4, n_spectra, lx, ly, n_iter, out, s)
                           : AP <= 512 ? epic::launch_cal_cluster<4>(plan, g, cl, ci4, n_spectra, lx, ly, n_iter, out, s)
                                       : epic::launch_cal_cluster<8>(plan, g, cl, ci4, n_spectra, lx, ly, n_iter, out, s);
            if (rc != EPIC_OK) return rc;
            continue;
        }
        epic::gain_solve_kernel<<<static_cast<unsigned>(g.n_chan * plan->P), epic::kCalThreads, smem, s>>>(
            ci4, plan->d_cells, g.d_chans, plan->A, plan->C, plan->P, n_spectra, g.N, lx, ly, n_iter,
            reinterpret_cast<float2 *>(gains_out));
        if (cudaGetLastError() != cudaSuccess) return EPIC_ERR_CUDA;
    }
    return EPIC_OK;
}
