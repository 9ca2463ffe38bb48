// FP32 form for grid sides 64, 96 and 128 whose aperture occupies at most 64 x 64
// cells (any 2x-padded array): one CTA images a whole channel, all pixel
// classes, from one gridding of each sample.
//
// The occupied cells are gridded into a compact array whose corner is the first
// occupied cell.  Moving the origin multiplies F(l) by one unit factor common to
// both polarisations, which cancels in every product, so nothing is folded and
// no class phase is needed (E-field images: fp32_efield.cu).  Rows are
// transformed to all N columns, then columns to all N rows, each N-point
// transform as N / M classes of M-point register transforms (fft_class.cuh).
//
// What this replaces: the per-class kernel (fp32_reg64.cu) grids every sample
// once per pixel class (4x at side 128), transforms the rows of each class
// (x-phase) separately per y-class (2x), and passes the finished planes through
// shared memory to form products.
//
//  * Warps 0-7 (transform): rows of sample t from G into R (lane = row and
//    polarisation), then columns of R (lane = column and polarisation, 16
//    columns of each per warp).  The lanes of a column's two polarisations
//    exchange half of their outputs by shuffles, so each lane forms XX, YY, XY of
//    half of the column's pixels from registers.  Y rows carry the sign (-1)^y,
//    which moves Y's outputs by M / 2: both lanes then keep the first half of
//    each output group and send the second, without selects.
//  * The time sums of all N^2 pixels live in tensor memory (4 floats a pixel:
//    all 512 columns at side 128), read and written by the lane that owns the
//    pixel, so they cost neither registers nor shared memory.
//  * Warps 8-11 (gridding) work a sample ahead: unpack and calibrate t + 1 while
//    t's rows are read, then gather t + 1 into G while t's columns are
//    transformed.  G is free as soon as the row transforms hold their inputs.
//
// Measured against the per-class kernel (one GB300, whole calls): 256 antennas, 64 channels of
// 128 x 128, 1000 spectra 5.78 -> 3.10 ms; the same as 25 Stokes images with delays 8.30 -> 3.55 ms;
// per-antenna kernels, 250 spectra 2.55 -> 0.99 ms with their auto image (image_common.cu);
// 37 channels at 64, 96 and 128 0.67 -> 0.46 ms.  Bound by the transform warps' issue: the FMA
// pipe is active 55 % of the time (42 % there, for half the work), 8 transform warps an SM.
//
// Shared memory: G [P][rows][65], R [P][rows][N + 1], voltages of two samples,
// gains, taps and gather lists (read through L1 where they do not fit).
// Side 64 takes two samples at a time, so that its transforms fill the 8 warps.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "epic_internal.cuh"
#include "fft_class.cuh"
#include "tc_ptx.cuh"

namespace epic {
namespace {

constexpr int kFW = 8;                       // transform warps
constexpr int kGW = kCompactGatherWarps;     // gridding warps
constexpr int kFT = 32 * kFW, kGT = 32 * kGW;
constexpr int kCThreads = kFT + kGT;
constexpr int kCS = 65;                      // row stride of G (float2)
constexpr int kBarFFT = 1, kBarGrid = 2;      // named barriers of the transform and the gridding warps
constexpr int kPreC = 4;                     // voltage words a gridding thread holds per sample (A P <= 2048)
constexpr uint16_t kNoCell = 0xFFFFu, kOddRow = 0x8000u;

// Rows of R: whole blocks of eight (class_load), the last ones zeros.
__host__ __device__ inline int compact_pad(int rows) { return (rows + 7) & ~7; }

// Byte offsets of the shared-memory regions (taps: with a kernel per antenna, the kernels are staged).
struct CompactSmem {
    unsigned R, es, gp, taps, tab, total;
};
__host__ __device__ inline CompactSmem compact_smem(int P, int TS, int N, int rows, int A, int K, int nker, bool taps,
                                                    int words)
{
    auto up = [](unsigned b) { return (b + 15u) & ~15u; };
    CompactSmem s;
    const unsigned planes = static_cast<unsigned>(TS * P * rows);
    s.R = up(planes * kCS * 8u);
    unsigned r = static_cast<unsigned>(TS * P * compact_pad(rows)) * (N + 1) * 8u;
    if (TS == 2) {   // the two samples' time sums are added through R at the end
        const unsigned sum = static_cast<unsigned>(N * N) * (P == 2 ? 16u : 4u);
        r = r > sum ? r : sum;
    }
    s.es = s.R + up(r);
    s.gp = s.es + up(2u * TS * A * P * 8u);
    s.taps = s.gp + up(static_cast<unsigned>(A * P) * 8u);
    s.tab = s.taps + (nker > 1 ? (taps ? up(static_cast<unsigned>(nker * K * K) * 8u) : 0u)
                               : static_cast<unsigned>(K * (K + 1) + 1) * 8u * 16u);
    s.total = s.tab + up(static_cast<unsigned>(words) * 2u);
    return s;
}

template <int M, int Q, int P, int TS>
struct CompactShape {
    static constexpr int N = M * Q;
    static constexpr int CB = 32 / P;                          // columns per column task
    static constexpr int TASKS = TS * Q * (N / CB);            // column tasks per iteration
    static constexpr int SL = (TASKS + kFW - 1) / kFW;         // column tasks of a warp
    static constexpr int CW = P == 2 ? 128 : 64;               // TMEM columns of a task's time sums
    static constexpr int NEED = 2 * SL * CW;                   // two warps share 32 TMEM lanes
    static constexpr int COLS = NEED <= 128 ? 128 : NEED <= 256 ? 256 : 512;
    static_assert(NEED <= 512, "time sums exceed tensor memory");
    // class of a warp's k-th column task: the turned class (h = 1) in turn, so that the warps' work is even
    static __device__ __forceinline__ int cls(int task, int k) { return (task + k) % Q; }
};

// staged: bit 0 the gather lists, bit 1 the antennas' kernels (AK) are in shared memory
template <int M, int Q, int P, int TS, bool AK>
__global__ void __launch_bounds__(kCThreads, 1)
fp32_compact_kernel(const uint8_t *__restrict__ v, const float2 *__restrict__ gains, const float2 *__restrict__ kern,
                    int K, const int *__restrict__ chans, const uint16_t *__restrict__ ltab,
                    const int2 *__restrict__ lidx, const int4 *__restrict__ lchan, int A, int C, int T, int n_chan,
                    int n_tau, int rmax, int staged, float *__restrict__ partial, const float *__restrict__ dfreq,
                    const float4 *__restrict__ dtab, int *__restrict__ status, long long wait_budget)
{
    using S = CompactShape<M, Q, P, TS>;
    constexpr int N = S::N, RS = N + 1, KO = M / 8, KH = KO / P;   // outputs per group; pixels a lane keeps of it
    extern __shared__ __align__(16) unsigned char smem_c[];
    __shared__ uint32_t tmem_slot;
    // G holds a sample (gridding warps arrive); G has been read, R has been read (transform warps)
    __shared__ __align__(8) uint64_t bar_full, bar_free, bar_read;
    const int AP = A * P, KK = K * K, TPN = K * (K + 1);
    const CompactSmem L = compact_smem(P, TS, N, rmax, A, K, AK ? A : 1, (staged & 2) != 0, 0);
    float2 *G = reinterpret_cast<float2 *>(smem_c);              // [TS][P][rmax][65]
    float2 *R = reinterpret_cast<float2 *>(smem_c + L.R);        // [TS][P][rmax][N + 1]
    float2 *es = reinterpret_cast<float2 *>(smem_c + L.es);      // [2][TS][A P]
    float2 *gp = reinterpret_cast<float2 *>(smem_c + L.gp);      // [A P]
    float4 *tw2 = reinterpret_cast<float4 *>(smem_c + L.taps);   // [K (K + 1) + 1][8 copies] (one kernel)
    const float2 *tapw = staged & 2 ? reinterpret_cast<const float2 *>(smem_c + L.taps) : kern;   // [A][K K] (a kernel per antenna)
    uint16_t *stab = reinterpret_cast<uint16_t *>(smem_c + L.tab);
    const int gplane = rmax * kCS, rplane = compact_pad(rmax) * RS;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ci = blockIdx.x % n_chan, tau = blockIdx.x / n_chan;
    const int c = chans[ci];
    const int t0 = static_cast<int>(static_cast<long long>(T) * tau / n_tau);
    const int t1 = static_cast<int>(static_cast<long long>(T) * (tau + 1) / n_tau);
    const int4 ch = lchan[2 * ci];                               // (block start, block words, rows, columns)
    const int rows = ch.z, cols = ch.w;

    if (warp == 0) tc::tmem_alloc(&tmem_slot, S::COLS);
    if (tid == 0) {
        tc::mbar_init(&bar_full, kGW);
        tc::mbar_init(&bar_free, kFW);
        tc::mbar_init(&bar_read, kFW);
        tc::fence_mbar_init();
    }
    // ---- set-up: a zero G (the cells no list names stay zero), gains, taps, lists
    for (int i = tid; i < TS * P * gplane; i += kCThreads) G[i] = make_float2(0.f, 0.f);
    const int rpad = (compact_pad(rows) - rows) * RS;            // R's rows past the channel's stay zero
    for (int i = tid; i < TS * P * rpad; i += kCThreads) R[(i / rpad) * rplane + rows * RS + i % rpad] = make_float2(0.f, 0.f);
    for (int i = tid; i < AP; i += kCThreads)
        gp[i] = gains ? gains[static_cast<size_t>(c) * AP + i] : make_float2(1.f, 0.f);
    if constexpr (AK) {
        if (staged & 2)
            for (int i = tid; i < A * KK; i += kCThreads) reinterpret_cast<float2 *>(smem_c + L.taps)[i] = kern[i];
    } else {
        // tap pairs (w(dy, dxl), w(dy, dxl + 1)), zero outside the footprint row; eight interleaved
        // copies, so the eight lanes of one 16-byte request never share a bank group; the last slot
        // is zero, for the lists' empty steps
        for (int i = tid; i < 8 * (TPN + 1); i += kCThreads) {
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
        for (int i = tid; i < ch.y; i += kCThreads) stab[i] = __ldg(ltab + ch.x + i);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = tmem_slot;
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

    if (warp < kFW) {
        // ================ transforms
        const uint32_t tw0 = taddr + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + (warp >> 2) * (S::SL * S::CW);
        uint32_t z[32];
#pragma unroll
        for (int j = 0; j < 32; j++) z[j] = 0u;
        for (int cc = 0; cc < S::SL * S::CW; cc += 32) tc::tmem_st32_issue(tw0 + cc, z);
        tc::tmem_wait_st();
        const int rb = (rows * P + 31) >> 5;                     // row tasks per sample and class
        const int n_row = TS * Q * rb;
        const int last_k = (S::TASKS - 1 - warp) / kFW;          // the warp's last column task (TASKS - 1 < warp: none)
        uint32_t ph = 0;
        for (int t = t0; t < t1; t += TS, ph ^= 1u) {
            wait(bar_full, ph);                                  // G holds sample t
            if (warp >= n_row) arrive(bar_free);
            bool r_free = t == t0;
            for (int task = warp; task < n_row; task += kFW) {
                const int h = task % Q, blk = (task / Q) % rb, ts = task / (Q * rb);
                const int q = blk * 32 + lane;
                const bool ok = q < rows * P;
                const int p = ok ? q / rows : 0, y = ok ? q - p * rows : 0;
                float2 x[M];
                class_load<M, 1>(x, G + (ts * P + p) * gplane + y * kCS, (cols + 7) >> 3, h);
                if (task + kFW >= n_row) arrive(bar_free);       // this warp has read G
                class_turn<M>(x, (cols + 7) >> 3, h);
                float2 *dst = R + (ts * P + p) * rplane + y * RS + h;
                if (!r_free) {
                    wait(bar_read, ph ^ 1u);                     // the columns of the sample before have been read
                    r_free = true;
                }
                fft_groups<M>(x, [&](int k1, auto &o) {
                    if (ok) {
#pragma unroll
                        for (int k2 = 0; k2 < KO; k2++) dst[Q * (k1 + 8 * k2)] = o[k2];
                    }
                });
            }
            if (!r_free) wait(bar_read, ph ^ 1u);
            tc::named_bar_sync(kBarFFT, kFT);                    // R is complete
            if (warp >= S::TASKS) arrive(bar_read);
#pragma unroll 1
            for (int k = 0; k < S::SL; k++) {
                const int task = warp + k * kFW;
                if (task >= S::TASKS) break;
                const int h = S::cls(task, k), blk = (task / Q) % (N / S::CB), ts = task / (Q * (N / S::CB));
                const int p = lane / S::CB, col = blk * S::CB + lane % S::CB;
                float2 x[M];
                class_load<M, RS>(x, R + (ts * P + p) * rplane + col, (rows + 7) >> 3, h);
                if (k == last_k) arrive(bar_read);
                class_turn<M>(x, (rows + 7) >> 3, h);
                const uint32_t at = tw0 + k * S::CW;
                fft_groups<M>(x, [&](int k1, auto &o) {
                    if constexpr (P == 2) {
                        uint32_t s[16];
                        tc::tmem_ld16_issue(at + 16 * k1, s);
                        float bx[KH], by[KH];
#pragma unroll
                        for (int j = 0; j < KH; j++) {
                            bx[j] = __shfl_xor_sync(0xffffffffu, o[j + KH].x, 16);
                            by[j] = __shfl_xor_sync(0xffffffffu, o[j + KH].y, 16);
                        }
                        tc::tmem_wait_ld();
                        tc::reg_fence16(s);
                        // own |F|^2, the other polarisation's |F|^2, Re and Im of F_X F_Y^* (Im with the
                        // lane's sign: own F_Y on the Y lanes)
#pragma unroll
                        for (int j = 0; j < KH; j++) {
                            const float2 a = o[j];
                            const float cx = bx[j], cy = by[j];
                            s[4 * j] = __float_as_uint(fmaf(a.x, a.x, fmaf(a.y, a.y, __uint_as_float(s[4 * j]))));
                            s[4 * j + 1] = __float_as_uint(fmaf(cx, cx, fmaf(cy, cy, __uint_as_float(s[4 * j + 1]))));
                            s[4 * j + 2] = __float_as_uint(fmaf(a.x, cx, fmaf(a.y, cy, __uint_as_float(s[4 * j + 2]))));
                            s[4 * j + 3] = __float_as_uint(fmaf(a.y, cx, fmaf(-a.x, cy, __uint_as_float(s[4 * j + 3]))));
                        }
                        tc::tmem_st16_issue(at + 16 * k1, s);
                    } else {
                        uint32_t s[8];
                        tc::tmem_ld8_issue(at + 8 * k1, s);
                        tc::tmem_wait_ld();
                        tc::reg_fence8(s);
#pragma unroll
                        for (int j = 0; j < KO; j++)
                            s[j] = __float_as_uint(fmaf(o[j].x, o[j].x, fmaf(o[j].y, o[j].y, __uint_as_float(s[j]))));
                        tc::tmem_st8_issue(at + 8 * k1, s);
                    }
                });
                tc::tmem_wait_st();
            }
        }
    } else {
        // ================ unpack, calibrate, grid
        const int gt = tid - kFT, gw = warp - kFW;
        const int2 my = lidx[ci * kGW + gw];                     // (first batch, batches)
        const bool words = (AP & 3) == 0 && (reinterpret_cast<uintptr_t>(v) & 3) == 0;
        const int APW = AP >> 2;
        uint32_t pre[TS][kPreC];
        // the bytes of sample t: words gt, gt + kGT, ..; or single bytes gt, gt + kGT, .. packed four to a word
        auto prefetch = [&](int t) {
#pragma unroll
            for (int ts = 0; ts < TS; ts++) {
                const uint8_t *row = v + (static_cast<size_t>(t + ts) * C + c) * AP;
                const bool ok = t + ts < t1;
#pragma unroll
                for (int r = 0; r < kPreC; r++) {
                    pre[ts][r] = 0u;
                    if (words) {
                        const int w = gt + r * kGT;
                        if (ok && w < APW) pre[ts][r] = __ldg(reinterpret_cast<const uint32_t *>(row) + w);
                    } else {
#pragma unroll
                        for (int b = 0; b < 4; b++) {
                            const int i = gt + (4 * r + b) * kGT;
                            if (ok && i < AP) pre[ts][r] |= static_cast<uint32_t>(__ldg(row + i)) << (8 * b);
                        }
                    }
                }
            }
        };
        auto unpack = [&](int t, int buf) {
            for (int ts = 0; ts < TS; ts++) {
                float2 *dst = es + (buf * TS + ts) * AP;
                const bool ok = t + ts < t1;                     // an absent sample grids zeros
#pragma unroll
                for (int r = 0; r < kPreC; r++) {
                    const uint32_t w4 = TS == 2 && ts == 1 ? pre[TS - 1][r] : pre[0][r];
                    float2 ph = make_float2(1.f, 0.f);
#pragma unroll
                    for (int b = 0; b < 4; b++) {
                        const int i = words ? 4 * (gt + r * kGT) + b : gt + (4 * r + b) * kGT;
                        if (i >= AP) continue;
                        float2 e = cmul(gp[i], ci4_decode(w4 >> (8 * b)));
                        if (dtab) {
                            // one phase per antenna: a word holds whole antennas
                            if (!words || P == 1 || (b & 1) == 0)
                                ph = ok ? delay_phase(dtab[static_cast<size_t>(t + ts) * A + i / P], dfreq[c])
                                        : make_float2(0.f, 0.f);
                            e = cmul(e, ph);
                        }
                        dst[i] = ok ? e : make_float2(0.f, 0.f);
                    }
                }
            }
        };
        // gather of the warp's batches: [d][32 left-cell offsets, bit 15: odd row, 0xFFFF: empty lane]
        // [d x 32 entries tp << 10 | a]; empty steps name the zero tap slot
        auto gather = [&](int buf) {
            const uint16_t *bt = (staged & 1 ? stab : ltab + ch.x) + my.x;
            auto ld = [](const uint16_t *q) -> uint32_t { return *q; };   // shared or global
            const float2 *e0 = es + buf * TS * AP;
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
                float2 e[TS][P];
            };
            auto volts = [&](uint32_t en) {
                Volt x;
                const int a = static_cast<int>(en & 1023u);
#pragma unroll
                for (int ts = 0; ts < TS; ts++) {
                    if constexpr (P == 2) {
                        const float4 f = reinterpret_cast<const float4 *>(e0 + ts * AP)[a];
                        x.e[ts][0] = make_float2(f.x, f.y);
                        x.e[ts][1] = make_float2(f.z, f.w);
                    } else {
                        x.e[ts][0] = e0[ts * AP + a];
                    }
                }
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
                float2 acc[TS][P][2];
#pragma unroll
                for (int ts = 0; ts < TS; ts++)
#pragma unroll
                    for (int p = 0; p < P; p++) acc[ts][p][0] = acc[ts][p][1] = make_float2(0.f, 0.f);
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
                    for (int ts = 0; ts < TS; ts++)
#pragma unroll
                        for (int p = 0; p < P; p++)
#pragma unroll
                            for (int u = 0; u < 2; u++) {
                                const float2 e = ee.e[ts][p];
                                float2 &o = acc[ts][p][u];
                                o.x = fmaf(-wi[u], e.y, fmaf(wr[u], e.x, o.x));
                                o.y = fmaf(wi[u], e.x, fmaf(wr[u], e.y, o.y));
                            }
                    ww = wwn;
                    ee = een;
                    en1 = en2;
                }
                if (off != kNoCell) {
                    float2 *cell = G + (off & 0x7FFFu);
                    const float sg = P == 2 && (off & kOddRow) ? -1.f : 1.f;   // (-1)^y on Y
#pragma unroll
                    for (int ts = 0; ts < TS; ts++)
#pragma unroll
                        for (int p = 0; p < P; p++)
#pragma unroll
                            for (int u = 0; u < 2; u++)
                                cell[(ts * P + p) * gplane + u] = p == 1 ? cscale(acc[ts][p][u], sg) : acc[ts][p][u];
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
            unpack(t0, 0);
            prefetch(t0 + TS);
            tc::named_bar_sync(kBarGrid, kGT);
            gather(0);
            arrive(bar_full);
        }
        uint32_t ph = 0;
        for (int t = t0; t + TS < t1; t += TS, ph ^= 1u) {
            buf ^= 1;
            unpack(t + TS, buf);
            prefetch(t + 2 * TS);
            tc::named_bar_sync(kBarGrid, kGT);                   // the sample's voltages are complete
            wait(bar_free, ph);                                  // the row transforms hold G(t)
            gather(buf);
            arrive(bar_full);
        }
    }

    // ---- partial image: [tau][channel item of class (hy, hx)][my M + mx]
    __syncthreads();
    float4 *sum4 = reinterpret_cast<float4 *>(R);
    float *sum1 = reinterpret_cast<float *>(R);
    for (int pass = TS - 1; pass >= 0; pass--) {             // TS == 2: the second sample's sums first, through R
        if (warp < kFW) {
            const uint32_t tw0 = taddr + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + (warp >> 2) * (S::SL * S::CW);
            for (int k = 0; k < S::SL; k++) {
                const int task = warp + k * kFW;
                if (task >= S::TASKS) break;
                const int h = S::cls(task, k), blk = (task / Q) % (N / S::CB), ts = task / (Q * (N / S::CB));
                if (ts != pass) continue;
                const int p = lane / S::CB, col = blk * S::CB + lane % S::CB;
                const int hx = col % Q, mx = col / Q;
                const size_t item = static_cast<size_t>(tau) * (n_chan * Q * Q) + ci * Q * Q + h * Q + hx;
                const int slot = (task % (Q * (N / S::CB))) * 8;   // the pair of tasks of two samples share it
#pragma unroll
                for (int k1 = 0; k1 < 8; k1++) {
                    if constexpr (P == 2) {
                        uint32_t s[16];
                        tc::tmem_ld16_issue(tw0 + k * S::CW + 16 * k1, s);
                        tc::tmem_wait_ld();
                        tc::reg_fence16(s);
                        float4 *dst = reinterpret_cast<float4 *>(partial) + item * (M * M) + mx;
#pragma unroll
                        for (int j = 0; j < KH; j++) {
                            const float a = __uint_as_float(s[4 * j]), b = __uint_as_float(s[4 * j + 1]);
                            const float re = __uint_as_float(s[4 * j + 2]), im = __uint_as_float(s[4 * j + 3]);
                            float4 f = p ? make_float4(b, a, re, -im) : make_float4(a, b, re, im);
                            float4 *sl = sum4 + ((slot + k1) * KH + j) * 32 + lane;
                            if (TS == 2 && pass == 1) {
                                *sl = f;
                                continue;
                            }
                            if (TS == 2) {
                                const float4 o = *sl;
                                f = make_float4(f.x + o.x, f.y + o.y, f.z + o.z, f.w + o.w);
                            }
                            dst[(k1 + 8 * (j + p * KH)) * M] = f;
                        }
                    } else {
                        uint32_t s[8];
                        tc::tmem_ld8_issue(tw0 + k * S::CW + 8 * k1, s);
                        tc::tmem_wait_ld();
                        tc::reg_fence8(s);
                        float *dst = partial + item * (M * M) + mx;
#pragma unroll
                        for (int j = 0; j < KO; j++) {
                            float f = __uint_as_float(s[j]);
                            float *sl = sum1 + ((slot + k1) * KO + j) * 32 + lane;
                            if (TS == 2 && pass == 1) {
                                *sl = f;
                                continue;
                            }
                            if (TS == 2) f += *sl;
                            dst[(k1 + 8 * j) * M] = f;
                        }
                    }
                }
            }
        }
        if (TS == 2) __syncthreads();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(taddr, S::COLS);
}

template <int V>
using IC = std::integral_constant<int, V>;

// The instantiation that serves a group: grid side, polarisations, samples per iteration.
template <class F>
int compact_dispatch(const GroupCfg &g, int P, F &&f)
{
    auto with_p = [&](auto p_) {
        if (g.N == 128) return f(IC<64>{}, IC<2>{}, p_, IC<1>{});
        if (g.N == 96) return f(IC<48>{}, IC<2>{}, p_, IC<1>{});
        return f(IC<64>{}, IC<1>{}, p_, IC<2>{});
    };
    return P == 2 ? with_p(IC<2>{}) : with_p(IC<1>{});
}

template <int M, int Q, int P, int TS, bool AK>
int launch_compact_t(epic_plan_s *plan, const GroupCfg &g, const uint8_t *v, const float2 *gains, int T, int n_tau,
                     cudaStream_t stream)
{
    const CompactSmem L = compact_smem(P, TS, g.N, g.crows, plan->A, plan->K, plan->nker, g.ctaps, g.cstage ? g.cwords : 0);
    fp32_compact_kernel<M, Q, P, TS, AK><<<static_cast<unsigned>(g.n_chan * n_tau), kCThreads, L.total, stream>>>(
        v, gains, plan->d_kernel, plan->K, g.d_chans, g.d_ltab, g.d_lidx, g.d_lchan, plan->A, plan->C, T, g.n_chan, n_tau,
        g.crows, (g.cstage ? 1 : 0) | (g.ctaps ? 2 : 0), g.d_partial, plan->d_dfreq, plan->delays ? plan->d_dtab : nullptr, plan->d_status,
        plan->wait_budget);
    return cudaGetLastError() == cudaSuccess ? EPIC_OK : EPIC_ERR_CUDA;
}

}  // namespace

// The gather lists of the compact kernel: the FP32 gather table (build_gather_table) of the
// same channels with the cells moved to the compact array's corner, its batches dealt again to
// the gridding warps (longest first, each to the warp with the least work; a batch costs 4 d + 6)
// and written in 16-bit words.  Per channel two int4: (block start, block words, rows, columns),
// (first occupied column, first occupied row, 0, 0); idx[ci * kCompactGatherWarps + w] = (offset
// of the warp's first batch in the block, batches).  EPIC_ERR_UNSUPPORTED when a channel's
// footprints span more than 64 cells on an axis, when A > 1024, or when K (K + 1) > 63.
int build_compact_lists(const std::vector<short2> &cells, int A, int K, int P, const std::vector<int> &chans,
                        std::vector<uint16_t> &tab, std::vector<int2> &idx, std::vector<int4> &chan)
{
    constexpr int M = 64, W32 = 8, W = kCompactGatherWarps;
    static_assert(M + 1 == kCS, "the gather table's row stride is G's");
    if (A > 1024 || K * (K + 1) > 62) return EPIC_ERR_UNSUPPORTED;
    const int nc = static_cast<int>(chans.size()), h = (K - 1) / 2;
    std::vector<short2> moved(cells);
    chan.assign(2 * static_cast<size_t>(nc), make_int4(0, 0, 0, 0));
    for (int ci = 0; ci < nc; ci++) {
        int x0 = 1 << 20, x1 = -1, y0 = 1 << 20, y1 = -1;
        short2 *cc = moved.data() + static_cast<size_t>(chans[ci]) * A;
        for (int a = 0; a < A; a++) {
            x0 = std::min(x0, cc[a].x - h);
            x1 = std::max(x1, cc[a].x + h);
            y0 = std::min(y0, cc[a].y - h);
            y1 = std::max(y1, cc[a].y + h);
        }
        if (x1 - x0 >= M || y1 - y0 >= M) return EPIC_ERR_UNSUPPORTED;
        for (int a = 0; a < A; a++) cc[a] = make_short2(static_cast<short>(cc[a].x - x0), static_cast<short>(cc[a].y - y0));
        chan[2 * ci] = make_int4(0, 0, y1 - y0 + 1, x1 - x0 + 1);
        chan[2 * ci + 1] = make_int4(x0, y0, 0, 0);
    }
    std::vector<uint32_t> tab32;
    std::vector<int4> idx32;
    std::vector<int2> chan32;
    std::vector<unsigned long long> rows32;
    if (const int rc = build_gather_table(moved, A, K, M, P, chans, tab32, idx32, chan32, rows32); rc != EPIC_OK) return rc;
    tab.clear();
    idx.assign(static_cast<size_t>(nc) * W, make_int2(0, 0));
    const uint32_t empty_tp = static_cast<uint32_t>(K * (K + 1));
    for (int ci = 0; ci < nc; ci++) {
        const uint32_t *blk = tab32.data() + chan32[ci].x;
        std::vector<std::pair<int, int>> bat;                    // (length, offset)
        for (int w = 0; w < W32; w++) {
            const int4 i32 = idx32[static_cast<size_t>(ci) * W32 + w];
            int at = i32.z;
            for (int b = 0; b < i32.w; b++) {
                const int d = static_cast<int>(blk[at]);
                bat.push_back({d, at});
                at += 33 + 32 * d;
            }
        }
        std::stable_sort(bat.begin(), bat.end(), [](const auto &u, const auto &v) { return u.first > v.first; });
        std::vector<std::vector<int>> per(W);
        std::vector<long long> load(W, 0);
        for (const auto &b : bat) {
            const int w = static_cast<int>(std::min_element(load.begin(), load.end()) - load.begin());
            per[w].push_back(b.second);
            load[w] += 4LL * b.first + 6;
        }
        const size_t start = tab.size();
        for (int w = 0; w < W; w++) {
            idx[static_cast<size_t>(ci) * W + w] = make_int2(static_cast<int>(tab.size() - start), static_cast<int>(per[w].size()));
            for (int at : per[w]) {
                const int d = static_cast<int>(blk[at]);
                tab.push_back(static_cast<uint16_t>(d));
                for (int l = 0; l < 32; l++) {
                    const uint32_t cw = blk[at + 1 + l];
                    tab.push_back(cw == ~0u ? kNoCell : static_cast<uint16_t>(cw | ((cw / kCS) & 1u ? kOddRow : 0u)));
                }
                for (int j = 0; j < d; j++) {
                    const uint32_t *en = blk + at + 33 + 32 * j;
                    // an empty step loads an antenna its 8-lane group loads anyway (its tap pair is zero)
                    for (int l = 0; l < 32; l++) {
                        uint32_t a = 0, tp = empty_tp;
                        if (en[l] != ~0u) {
                            a = en[l] >> 8;
                            tp = en[l] & 0xFFu;
                        } else {
                            for (int u = l & ~7; u < (l & ~7) + 8; u++)
                                if (en[u] != ~0u) {
                                    a = en[u] >> 8;
                                    break;
                                }
                        }
                        tab.push_back(static_cast<uint16_t>((tp << 10) | a));
                    }
                }
            }
        }
        if (tab.size() > 0x7FFFFFFFull) return EPIC_ERR_UNSUPPORTED;
        chan[2 * ci].x = static_cast<int>(start);
        chan[2 * ci].y = static_cast<int>(tab.size() - start);
    }
    if (tab.empty()) tab.push_back(0);
    return EPIC_OK;
}

// Whether images of a side are faster here than in the per-class kernel.  At side 64 there is one
// class, so nothing is gridded twice there: its gather uses all warps between the transforms, this
// kernel's four warps run beside them, but with a single polarisation only half of the transform warps
// have work.  What decides is the gather, as footprint cells a row (batches get longer, not more, where
// footprints overlap).  One GB300, us per class / compact, 300 spectra of 32 channels: one polarisation,
// footprints over 56 x 56 cells, 64 antennas 5 x 5 (29 cells a row) 129 / 153, 64 of 7 x 7 (56) 143 / 150;
// over 15 x 15, 64 of 3 x 3 (38) 129 / 145, 32 of 5 x 5 (50) 141 / 144, 64 of 5 x 5 (100) 162 / 146; two
// polarisations over 14 x 14, 16 antennas 1 x 1 (1) 166 / 172, 32 of 3 x 3 (19) 187 / 177; over 56 x 56,
// 16 of 1 x 1 (0.3) 166 / 183.
bool compact_pays(int N, int P, int A, int K, int rows, int cols)
{
    const double per_row = static_cast<double>(A) * K * K / std::sqrt(static_cast<double>(rows) * cols);
    return N != 64 || per_row > (P == 2 ? 5.0 : 60.0);
}

// The same against the shared-memory kernel, where n_ant n_pol is not a multiple of 4: its atomics cost
// little for one tap.  Side 64, one polarisation, us there / here: 34 antennas, 1 x 1, 60 channels x 74 spectra
// 76 / 90, 32 x 300 139 / 147, 255 antennas 82 / 92 and 152 / 150; 17 antennas, 3 x 3 92 / 90.
bool compact_pays_odd(int N, int P, int K) { return !(N == 64 && P == 1 && K == 1); }

size_t compact_smem_bytes(int N, int P, int rows, int A, int K, int nker, bool taps, int words)
{
    return compact_smem(P, N == 64 ? 2 : 1, N, rows, A, K, nker, taps, words).total;
}

int prepare_compact(const epic_plan_s *plan, const GroupCfg &g)
{
    const size_t need = compact_smem_bytes(g.N, plan->P, g.crows, plan->A, plan->K, plan->nker, g.ctaps, g.cstage ? g.cwords : 0);
    return compact_dispatch(g, plan->P, [&](auto m_, auto q_, auto p_, auto ts_) {
        constexpr int M = decltype(m_)::value, Q = decltype(q_)::value, P = decltype(p_)::value, TS = decltype(ts_)::value;
        return plan->nker > 1 ? raise_dyn_smem_cap(reinterpret_cast<const void *>(fp32_compact_kernel<M, Q, P, TS, true>), need)
                              : raise_dyn_smem_cap(reinterpret_cast<const void *>(fp32_compact_kernel<M, Q, P, TS, false>), need);
    });
}

int launch_compact(epic_plan_s *plan, const GroupCfg &g, const uint8_t *v, const float2 *gains, int T, int *n_tau_out,
                   cudaStream_t stream)
{
    const int n_tau = choose_tau(plan, g, T);
    *n_tau_out = n_tau;
    return compact_dispatch(g, plan->P, [&](auto m_, auto q_, auto p_, auto ts_) {
        constexpr int M = decltype(m_)::value, Q = decltype(q_)::value, P = decltype(p_)::value, TS = decltype(ts_)::value;
        return plan->nker > 1 ? launch_compact_t<M, Q, P, TS, true>(plan, g, v, gains, T, n_tau, stream)
                              : launch_compact_t<M, Q, P, TS, false>(plan, g, v, gains, T, n_tau, stream);
    });
}

}  // namespace epic
