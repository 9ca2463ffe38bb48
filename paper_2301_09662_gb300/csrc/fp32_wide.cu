// FP32 form for grid sides 256 and 512 (dual polarisation) whose aperture occupies at
// most 128 x 128 cells: rows first, columns second, each sample gridded once.
//
// The occupied cells form a compact array whose corner is the first occupied
// cell (the common unit factor this takes out of F cancels in every product).
// With l = Q m + h, N = 64 Q, an N-point transform of at most 128 inputs is, for each class h < Q,
// one 64-point transform of x(i) + w_Q^h x(i + 64) turned by w_N^{i h}.
//
//  * wide_rows_kernel: a block owns a channel, a band of 64 rows and a run of
//    samples; it calibrates and gathers each sample into the band (both
//    polarisations) and transforms the rows to all N columns, written to
//    workspace as [channel][sample][class hx][polarisation][m][row].
//  * wide_cols_kernel: a block owns 32 columns of a channel (half a class hx) and
//    all N of their rows; per sample one bulk copy a polarisation brings its
//    inputs, each warp transforms 16 columns of both polarisations for one class
//    hy at a time, forms the products from registers and adds them to time sums
//    in tensor memory (32 N pixels of 4 floats: all 512 columns at side 512).
//
// What this replaces at side 512: gridding once and folding into 64 class grids
// of 64 x 64, 4 MB a channel and sample written and read through HBM, and a row
// and column transform of each; here 1 MB, a quarter of the row transforms and
// half of the column transforms' loads.  At side 256 the per-class kernel grids
// every sample 16 times.  64 channels of 512 x 512, 2048 antennas, 7 x 7 kernel,
// 100 spectra: 20.40 -> 6.96 ms (rows 2.5, columns 4.0); 32 channels of 256 x
// 256, 1024 antennas 2.90 -> 1.21 ms.  Columns: FMA pipe 59 % active, HBM 19 %;
// rows: shared-memory and list latency between barriers, FMA 28 %.
//
// The workspace's row order within a column is turned by the column (16-byte units, unit u of column
// m at u ^ (m mod 8)): a warp's columns then read distinct banks, and a column's
// 128-byte segments stay whole for the writer.
#include <algorithm>
#include <atomic>
#include <thread>
#include <type_traits>

#include "epic_internal.cuh"
#include "fft_class.cuh"
#include "tc_ptx.cuh"

namespace epic {
namespace {

constexpr int kRowsThreads = 384, kRowsWarps = 12, kBand = 64;
constexpr int kWS = 129;                     // row stride of the band (float2)
constexpr int kColWarps = 8, kColThreads = 32 * kColWarps;   // 8 warps: a ninth would cap all at 168 registers
constexpr int kTileCols = 32;
constexpr uint32_t kNoCellW = ~0u;

// w_N^{i h}, i < 64, h < Q, of N = 64 Q
template <int Q>
struct WideTwiddle {
    float2 w[Q][64];
};
template <int Q>
constexpr WideTwiddle<Q> make_wide_twiddle()
{
    WideTwiddle<Q> t{};
    for (int h = 0; h < Q; h++)
        for (int i = 0; i < 64; i++) t.w[h][i] = ce_w(i * h, 64 * Q);
    return t;
}
__constant__ const WideTwiddle<4> c_wide4 = make_wide_twiddle<4>();
__constant__ const WideTwiddle<8> c_wide8 = make_wide_twiddle<8>();

template <int Q>
__device__ __forceinline__ float2 wide_tw(int h, int i)
{
    if constexpr (Q == 4) return c_wide4.w[h][i];
    else return c_wide8.w[h][i];
}
// w_Q^h = w_N^{64 h}
template <int Q>
__device__ __forceinline__ float2 wide_fold(int h)
{
    const float s = kSqrtHalf;
    const int e = h * (8 / Q);               // eighths of a turn
    const float re = (e & 1) ? ((e + 1) & 4 ? -s : s) : (e == 0 ? 1.f : e == 4 ? -1.f : 0.f);
    const float im = (e & 1) ? (e & 4 ? -s : s) : (e == 2 ? 1.f : e == 6 ? -1.f : 0.f);
    return make_float2(re, im);
}

// x(i) for i = 0 .. 63: x += g y packed, (re, im) pairs
__device__ __forceinline__ float2 wide_mac(float2 x, float2 y, float2 grr, float2 gni)
{
    return pfma(pswap(y), gni, pfma(y, grr, x));
}

// dynamic shared memory of the row kernel: G [2][64][129], es [A] (X re, im, Y re, im), tap pairs [8 copies]
size_t wide_rows_smem(int A, int K)
{
    return sizeof(float2) * 2 * kBand * kWS + sizeof(float4) * static_cast<size_t>(A) +
           sizeof(float4) * 8 * (static_cast<size_t>(K) * (K + 1) + 1);
}
// with the gains [A] (X re, im, Y re, im) behind them where they fit
size_t wide_rows_smem(int A, int K, bool gains) { return wide_rows_smem(A, K) + (gains ? sizeof(float4) * static_cast<size_t>(A) : 0); }

// grid: time chunk fastest, then band, then channel of the batch.  Samples tb0 .. tb0 + nb of the batch.
template <int Q>
__global__ void __launch_bounds__(kRowsThreads, 1)
wide_rows_kernel(const uint8_t *__restrict__ v, const float2 *__restrict__ gains, const float2 *__restrict__ kern, int K,
                 const int *__restrict__ chans, const uint32_t *__restrict__ ltab, const int2 *__restrict__ lidx,
                 const int4 *__restrict__ lchan, int A, int C, int ci0, int bands, int tb0, int nb, int n_chunk, int rpad, int staged,
                 const float *__restrict__ dfreq, const float4 *__restrict__ dtab, float2 *__restrict__ ws)
{
    extern __shared__ __align__(16) unsigned char smem_w[];
    float2 *G = reinterpret_cast<float2 *>(smem_w);              // [2][64][129]
    float4 *es = reinterpret_cast<float4 *>(G + 2 * kBand * kWS);
    float4 *tw2 = es + A;
    constexpr int GP = kBand * kWS;
    const int TPN = K * (K + 1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int chunk = blockIdx.x % n_chunk, band = (blockIdx.x / n_chunk) % bands, cb = blockIdx.x / (n_chunk * bands);
    const int ci = ci0 + cb, c = chans[ci];
    const int b0 = static_cast<int>(static_cast<long long>(nb) * chunk / n_chunk);
    const int b1 = static_cast<int>(static_cast<long long>(nb) * (chunk + 1) / n_chunk);
    const int4 ch = lchan[ci];                                   // (rows, columns, 0, 0)
    const int nbx = (ch.y + 7) >> 3;
    const int2 my = lidx[(static_cast<size_t>(ci) * bands + band) * kRowsWarps + warp];   // (first batch, batches)

    for (int i = tid; i < 2 * GP; i += kRowsThreads) G[i] = make_float2(0.f, 0.f);
    for (int i = tid; i < 8 * (TPN + 1); i += kRowsThreads) {    // tap pairs, eight copies; the last slot zero
        const int tp = i >> 3, dyi = tp / (K + 1), j = tp % (K + 1);
        float2 w[2];
        for (int u = 0; u < 2; u++) {
            const int dx = j - 1 + u;
            w[u] = (tp < TPN && dx >= 0 && dx < K) ? kern[dyi * K + dx] : make_float2(0.f, 0.f);
        }
        tw2[i] = make_float4(w[0].x, w[0].y, w[1].x, w[1].y);
    }
    float4 *gs = tw2 + 8 * (TPN + 1);        // staged gains
    if (staged)
        for (int a = tid; a < A; a += kRowsThreads) {
            const float2 *gg = gains ? gains + (static_cast<size_t>(c) * A + a) * 2 : nullptr;
            gs[a] = gg ? make_float4(gg[0].x, gg[0].y, gg[1].x, gg[1].y) : make_float4(1.f, 0.f, 1.f, 0.f);
        }
    const bool two = (reinterpret_cast<uintptr_t>(v) & 1) == 0;
    const uint32_t empty = static_cast<uint32_t>(TPN);
    const float4 *tw8 = tw2 + (lane & 7);

    for (int bt = b0; bt < b1; bt++) {
        const int t = tb0 + bt;
        const uint8_t *row = v + (static_cast<size_t>(t) * C + c) * A * 2;
        for (int a = tid; a < A; a += kRowsThreads) {
            const uint32_t b = two ? __ldg(reinterpret_cast<const uint16_t *>(row) + a)
                                   : __ldg(row + 2 * a) | static_cast<uint32_t>(__ldg(row + 2 * a + 1)) << 8;
            float2 ex = ci4_decode(b), ey = ci4_decode(b >> 8);
            if (staged) {                    // (this thread's own entries)
                const float4 gv = gs[a];
                ex = cmul(make_float2(gv.x, gv.y), ex);
                ey = cmul(make_float2(gv.z, gv.w), ey);
            } else if (gains) {
                const float2 *gg = gains + (static_cast<size_t>(c) * A + a) * 2;
                ex = cmul(__ldg(gg), ex);
                ey = cmul(__ldg(gg + 1), ey);
            }
            if (dtab) {
                const float2 ph = delay_phase(dtab[static_cast<size_t>(t) * A + a], dfreq[c]);
                ex = cmul(ex, ph);
                ey = cmul(ey, ph);
            }
            es[a] = make_float4(ex.x, ex.y, ey.x, ey.y);
        }
        __syncthreads();   // voltages complete; the band's rows of the sample before have been read

        // ---- gather: [d][32 left-cell offsets][d x 32 entries a << 8 | tp], two steps at a time (an odd last
        // step's second half names the zero tap slot).  The lists come from L2: the next batch's header
        // and first entries are loaded a batch ahead, entries four steps ahead, taps and voltages two.
        {
            const uint32_t *bp = ltab + my.x;
            int d = my.y > 0 ? static_cast<int>(__ldg(bp)) : 0;
            uint32_t off = __ldg(bp + 1 + lane), q[4];
#pragma unroll
            for (int i = 0; i < 4; i++) q[i] = __ldg(bp + 33 + i * 32 + lane);   // the table ends with spare words
            for (int b = 0; b < my.y; b++) {
                const uint32_t *ent = bp + 33 + lane, *np = bp + 33 + 32 * d;
                const int dn = static_cast<int>(__ldg(np));
                const uint32_t offn = __ldg(np + 1 + lane);
                uint32_t qn[4];
#pragma unroll
                for (int i = 0; i < 4; i++) qn[i] = __ldg(np + 33 + i * 32 + lane);
#pragma unroll
                for (int i = 1; i < 4; i++) q[i] = i < d ? q[i] : empty;
                float2 acc[2][2];
                acc[0][0] = acc[0][1] = acc[1][0] = acc[1][1] = make_float2(0.f, 0.f);
                float4 ww[2], ee[2];
#pragma unroll
                for (int i = 0; i < 2; i++) {
                    ww[i] = tw8[(q[i] & 255u) << 3];
                    ee[i] = es[q[i] >> 8];
                }
#pragma unroll 2
                for (int j = 0; j < d; j += 2) {
                    const float4 w0 = ww[0], w1 = ww[1], e0 = ee[0], e1 = ee[1];
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        ww[i] = tw8[(q[2 + i] & 255u) << 3];
                        ee[i] = es[q[2 + i] >> 8];
                        q[2 + i] = j + 4 + i < d ? __ldg(ent + (j + 4 + i) * 32) : empty;
                    }
                    auto add = [&](const float4 &w, const float4 &e) {
                        const float wr[2] = {w.x, w.z}, wi[2] = {w.y, w.w};
#pragma unroll
                        for (int u = 0; u < 2; u++) {
                            acc[0][u].x = fmaf(-wi[u], e.y, fmaf(wr[u], e.x, acc[0][u].x));
                            acc[0][u].y = fmaf(wi[u], e.x, fmaf(wr[u], e.y, acc[0][u].y));
                            acc[1][u].x = fmaf(-wi[u], e.w, fmaf(wr[u], e.z, acc[1][u].x));
                            acc[1][u].y = fmaf(wi[u], e.z, fmaf(wr[u], e.w, acc[1][u].y));
                        }
                    };
                    add(w0, e0);
                    add(w1, e1);
                }
                if (off != kNoCellW) {
                    // Y rows take (-1)^y, which moves Y's column outputs by 32 of 64 (wide_cols_kernel)
                    const float sg = (off >> 31) ? -1.f : 1.f;
                    float2 *cell = G + (off & 0x7FFFFFFFu);
                    cell[0] = acc[0][0];
                    cell[1] = acc[0][1];
                    cell[GP] = cscale(acc[1][0], sg);
                    cell[GP + 1] = cscale(acc[1][1], sg);
                }
                bp = np;
                d = dn;
                off = offn;
#pragma unroll
                for (int i = 0; i < 4; i++) q[i] = qn[i];
            }
        }
        __syncthreads();

        // ---- rows: lane = row of the band and polarisation, one class at a time
        for (int task = warp; task < 4 * Q; task += kRowsWarps) {
            const int h = task % Q, blk = task / Q, p = blk >> 1, y = (blk & 1) * 32 + lane, gy = band * kBand + y;
            const float2 *line = G + p * GP + y * kWS;
            const float2 g = wide_fold<Q>(h);
            const float2 grr = make_float2(g.x, g.x), gni = make_float2(-g.y, g.y);
            float2 x[64];
#pragma unroll
            for (int b = 0; b < 8; b++) {
                if (b < nbx) {
#pragma unroll
                    for (int i = 8 * b; i < 8 * b + 8; i++) x[i] = line[i];
                } else {
#pragma unroll
                    for (int i = 8 * b; i < 8 * b + 8; i++) x[i] = make_float2(0.f, 0.f);
                }
                if (b + 8 < nbx) {
#pragma unroll
                    for (int i = 8 * b; i < 8 * b + 8; i++) x[i] = wide_mac(x[i], line[i + 64], grr, gni);
                }
            }
            if (h) {
#pragma unroll
                for (int i = 1; i < 64; i++) x[i] = cmul(x[i], wide_tw<Q>(h, i));
            }
            // column m = k1 + 8 k2 of the class: unit (row / 2) ^ (m mod 8) of 16 bytes
            float2 *dst = ws + (((static_cast<size_t>(cb) * nb + bt) * Q + h) * 2 + p) * 64 * rpad;
            const bool ok = gy < rpad;
            fft_groups<64>(x, [&](int k1, auto &o) {
                float2 *at = dst + static_cast<size_t>(k1) * rpad + ((((gy >> 1) ^ k1) << 1) | (gy & 1));
                if (ok) {
#pragma unroll
                    for (int k2 = 0; k2 < 8; k2++) at[static_cast<size_t>(8 * k2) * rpad] = o[k2];
                }
            });
        }
    }
}

// grid: tile (class hx, half of its columns) fastest, then channel of the batch, then time chunk: chunk
// tau of n_sub takes its share of the batch's nb samples into partial slot tau
template <int Q>
__global__ void __launch_bounds__(kColThreads, 1)
wide_cols_kernel(const float2 *__restrict__ ws, int nb, int nc, int n_sub, int ci0, int rpad, int stages, int accumulate,
                 float4 *__restrict__ partial, size_t slot, int *__restrict__ status, long long wait_budget)
{
    constexpr int SL = 2 * Q / kColWarps;                        // column tasks of a warp: 16 columns, one class
    constexpr int COLS = 256 * SL;                               // tensor memory columns: 128 a task, two warps share lanes
    extern __shared__ __align__(128) unsigned char smem_w[];     // [stages][2][32][rpad] float2
    __shared__ __align__(8) uint64_t full[4], empty[4];
    __shared__ uint32_t tmem_slot;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.x % (2 * Q), cb = (blockIdx.x / (2 * Q)) % nc, hx = tile >> 1, m0 = (tile & 1) * kTileCols;
    const int ci = ci0 + cb, tau = blockIdx.x / (2 * Q * nc);
    const int b0 = static_cast<int>(static_cast<long long>(nb) * tau / n_sub);
    const int n = static_cast<int>(static_cast<long long>(nb) * (tau + 1) / n_sub) - b0;   // samples of this block
    partial += slot * tau;
    const uint32_t bytes = static_cast<uint32_t>(kTileCols * rpad) * 8u;   // of one polarisation
    if (warp == 0) tc::tmem_alloc(&tmem_slot, COLS);
    if (tid == 0) {
        for (int s = 0; s < stages; s++) {
            tc::mbar_init(&full[s], 1);
            tc::mbar_init(&empty[s], kColWarps);
        }
        tc::fence_mbar_init();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t taddr = tmem_slot;
    bool dead = false;                       // bounded waits: record a timeout, wait no more, end
    auto wait = [&](uint64_t &bar, uint32_t parity) {
        if (!dead && !tc::mbar_wait(&bar, parity, wait_budget)) {
            dead = true;
            atomicOr(status, kStatusTimeout);
        }
    };
    const uint32_t tw0 = taddr + (static_cast<uint32_t>(32 * (warp & 3)) << 16) + (warp >> 2) * (SL * 128);
    const int p = lane >> 4, cl = lane & 15;
    // pixel (ly, lx) of this lane's column lx = Q (m0 + ..) + hx in the partial image
    auto pix = [&](int h, int blk, int m) {
        return ((static_cast<size_t>(ci) * Q * Q + h * Q + hx) * 64 + m) * 64 + m0 + blk * 16 + cl;
    };

    // sample q's tile into its buffer, one bulk copy a polarisation (warp 0)
    int fetched = 0;
    auto fetch = [&](int q) {
        const int s = q % stages, use = q / stages;
        if (use > 0) wait(empty[s], (use - 1) & 1);
        if (!dead) fetched = q + 1;
        if (lane == 0 && !dead) {
            tc::mbar_expect_tx(&full[s], 2 * bytes);
            const float2 *src = ws + ((static_cast<size_t>(cb) * nb + b0 + q) * Q + hx) * 2 * 64 * rpad + static_cast<size_t>(m0) * rpad;
            unsigned char *dst = smem_w + static_cast<size_t>(s) * 2 * bytes;
            tc::bulk_g2s(dst, src, bytes, &full[s]);
            tc::bulk_g2s(dst + bytes, src + static_cast<size_t>(64) * rpad, bytes, &full[s]);
        }
        __syncwarp();
    };
    if (warp == 0)
        for (int q = 0; q < stages - 1 && q < n; q++) fetch(q);
    {
        // ---- time sums: zero, or the batches before
        for (int k = 0; k < SL; k++) {
            const int task = warp + k * kColWarps, h = task % Q, blk = task / Q;
#pragma unroll
            for (int k1 = 0; k1 < 8; k1++) {
                uint32_t s[16];
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    float4 f = accumulate ? partial[pix(h, blk, k1 + 8 * j + 32 * p)] : make_float4(0.f, 0.f, 0.f, 0.f);
                    if (p) f = make_float4(f.y, f.x, f.z, -f.w);
                    s[4 * j] = __float_as_uint(f.x);
                    s[4 * j + 1] = __float_as_uint(f.y);
                    s[4 * j + 2] = __float_as_uint(f.z);
                    s[4 * j + 3] = __float_as_uint(f.w);
                }
                tc::tmem_st16_issue(tw0 + k * 128 + 16 * k1, s);
            }
        }
        tc::tmem_wait_st();
        const int nby = rpad >> 4;           // blocks of 16 rows
        for (int bt = 0; bt < n; bt++) {
            const int st = bt % stages;
            wait(full[st], (bt / stages) & 1);
            const unsigned char *base = smem_w + static_cast<size_t>(st) * 2 * bytes + p * bytes;
#pragma unroll 1
            for (int k = 0; k < SL; k++) {
                const int task = warp + k * kColWarps, h = task % Q, blk = task / Q;
                const int col = blk * 16 + cl;
                const unsigned char *line = base + static_cast<size_t>(col) * rpad * 8;
                const int sw = col & 7;
                // rows 2 u, 2 u + 1
                auto ld = [&](int u) {
                    return *reinterpret_cast<const float4 *>(line + ((((u & 7) ^ sw) << 4) + ((u & ~7) << 4)));
                };
                const float2 g = wide_fold<Q>(h);
                const float2 grr = make_float2(g.x, g.x), gni = make_float2(-g.y, g.y);
                float2 x[64];
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    if (b < nby) {
#pragma unroll
                        for (int u = 8 * b; u < 8 * b + 8; u++) {
                            const float4 f = ld(u);
                            x[2 * u] = make_float2(f.x, f.y);
                            x[2 * u + 1] = make_float2(f.z, f.w);
                        }
                    } else {
#pragma unroll
                        for (int u = 8 * b; u < 8 * b + 8; u++) x[2 * u] = x[2 * u + 1] = make_float2(0.f, 0.f);
                    }
                    if (b + 4 < nby) {
#pragma unroll
                        for (int u = 8 * b; u < 8 * b + 8; u++) {
                            const float4 f = ld(u + 32);
                            x[2 * u] = wide_mac(x[2 * u], make_float2(f.x, f.y), grr, gni);
                            x[2 * u + 1] = wide_mac(x[2 * u + 1], make_float2(f.z, f.w), grr, gni);
                        }
                    }
                }
                if (k == SL - 1) {           // this warp has read the tile; warp 0 refills the buffer before it
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&empty[st]);
                    if (warp == 0 && bt + stages - 1 < n) fetch(bt + stages - 1);
                }
                if (h) {
#pragma unroll
                    for (int i = 1; i < 64; i++) x[i] = cmul(x[i], wide_tw<Q>(h, i));
                }
                const uint32_t at = tw0 + k * 128;
                fft_groups<64>(x, [&](int k1, auto &o) {
                    uint32_t s[16];
                    tc::tmem_ld16_issue(at + 16 * k1, s);
                    float bx[4], by[4];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        bx[j] = __shfl_xor_sync(0xffffffffu, o[j + 4].x, 16);
                        by[j] = __shfl_xor_sync(0xffffffffu, o[j + 4].y, 16);
                    }
                    tc::tmem_wait_ld();
                    tc::reg_fence16(s);
                    // own |F|^2, the other polarisation's |F|^2, Re and Im of F_X F_Y^* (Im with the
                    // lane's sign); Y's outputs are moved by 32, so both lanes keep the first half
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const float2 a = o[j];
                        const float cx = bx[j], cy = by[j];
                        s[4 * j] = __float_as_uint(fmaf(a.x, a.x, fmaf(a.y, a.y, __uint_as_float(s[4 * j]))));
                        s[4 * j + 1] = __float_as_uint(fmaf(cx, cx, fmaf(cy, cy, __uint_as_float(s[4 * j + 1]))));
                        s[4 * j + 2] = __float_as_uint(fmaf(a.x, cx, fmaf(a.y, cy, __uint_as_float(s[4 * j + 2]))));
                        s[4 * j + 3] = __float_as_uint(fmaf(a.y, cx, fmaf(-a.x, cy, __uint_as_float(s[4 * j + 3]))));
                    }
                    tc::tmem_st16_issue(at + 16 * k1, s);
                });
                tc::tmem_wait_st();
            }
        }
        for (int k = 0; k < SL; k++) {
            const int task = warp + k * kColWarps, h = task % Q, blk = task / Q;
#pragma unroll
            for (int k1 = 0; k1 < 8; k1++) {
                uint32_t s[16];
                tc::tmem_ld16_issue(tw0 + k * 128 + 16 * k1, s);
                tc::tmem_wait_ld();
                tc::reg_fence16(s);
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float a = __uint_as_float(s[4 * j]), b = __uint_as_float(s[4 * j + 1]);
                    const float re = __uint_as_float(s[4 * j + 2]), im = __uint_as_float(s[4 * j + 3]);
                    partial[pix(h, blk, k1 + 8 * j + 32 * p)] = p ? make_float4(b, a, re, -im) : make_float4(a, b, re, im);
                }
            }
        }
    }
    if (tid == 0 && dead)                // copies still in flight land before the block's memory is another's
        for (int q = max(0, fetched - stages); q < fetched; q++) tc::mbar_wait(&full[q % stages], (q / stages) & 1, wait_budget);
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(taddr, COLS);
}

size_t wide_cols_smem(int rpad, int stages) { return static_cast<size_t>(stages) * 2 * kTileCols * rpad * 8; }

}  // namespace

// Gather lists of the row kernel: per (channel, band of 64 rows) the pairs of horizontally adjacent
// cells (2 xp, 2 xp + 1) of the compact array with their (antenna, tap pair) entries, as in
// build_gather_table; pairs sorted by list length, batches of 32 lanes, within each 8-lane group (one
// 16-byte voltage request) a step order whose antennas fall in distinct banks (a mod 8) where the
// lists allow; batches dealt longest first to the warp with the least work.  Words: [d][32 cell
// offsets y 129 + x, bit 31: odd row, or ~0][d x 32 entries a << 8 | tp], an empty step naming the
// zero tap slot K (K + 1).  chan[ci] = (rows, columns, 0, 0); idx[(ci bands + band) 12 + warp] =
// (offset of the warp's first batch, batches).  EPIC_ERR_UNSUPPORTED when a channel's footprints
// span more than 128 cells on an axis.
int build_wide_lists(const std::vector<short2> &cells, int A, int K, const std::vector<int> &chans, int &bands,
                     std::vector<uint32_t> &tab, std::vector<int2> &idx, std::vector<int4> &chan, int threads)
{
    constexpr int W = kRowsWarps;
    const int nc = static_cast<int>(chans.size()), h = (K - 1) / 2;
    const uint32_t empty = static_cast<uint32_t>(K * (K + 1));
    if (A > 4096 || K * (K + 1) > 255) return EPIC_ERR_UNSUPPORTED;
    chan.assign(nc, make_int4(0, 0, 0, 0));
    std::vector<short2> org(nc);
    int rmax = 0;
    for (int ci = 0; ci < nc; ci++) {
        int x0 = 1 << 20, x1 = -1, y0 = 1 << 20, y1 = -1;
        const short2 *cc = cells.data() + static_cast<size_t>(chans[ci]) * A;
        for (int a = 0; a < A; a++) {
            x0 = std::min(x0, cc[a].x - h);
            x1 = std::max(x1, cc[a].x + h);
            y0 = std::min(y0, cc[a].y - h);
            y1 = std::max(y1, cc[a].y + h);
        }
        if (x1 - x0 >= 128 || y1 - y0 >= 128) return EPIC_ERR_UNSUPPORTED;
        chan[ci] = make_int4(y1 - y0 + 1, x1 - x0 + 1, 0, 0);
        org[ci] = make_short2(static_cast<short>(x0), static_cast<short>(y0));
        rmax = std::max(rmax, y1 - y0 + 1);
    }
    bands = (rmax + kBand - 1) / kBand;
    const int nbl = nc * bands;
    idx.assign(static_cast<size_t>(nbl) * W, make_int2(0, 0));
    std::vector<std::vector<uint32_t>> blocks(nbl);
    auto build = [&](int bi) {
        const int ci = bi / bands, band = bi % bands;
        const short2 *cc = cells.data() + static_cast<size_t>(chans[ci]) * A;
        std::vector<std::vector<uint32_t>> list(kBand * 64);     // [row of the band][pair]
        for (int a = 0; a < A; a++)
            for (int dyi = 0; dyi < K; dyi++) {
                const int y = cc[a].y + dyi - h - org[ci].y - band * kBand;
                if (y < 0 || y >= kBand) continue;
                const int xl = cc[a].x - h - org[ci].x;          // first covered column
                for (int xp = xl >> 1; 2 * xp < xl + K; xp++)
                    list[y * 64 + xp].push_back((static_cast<uint32_t>(a) << 8) |
                                                static_cast<uint32_t>(dyi * (K + 1) + (2 * xp - xl) + 1));
            }
        std::vector<int> used;
        for (int i = 0; i < kBand * 64; i++)
            if (!list[i].empty()) used.push_back(i);
        std::stable_sort(used.begin(), used.end(), [&](int u, int w) { return list[u].size() > list[w].size(); });
        std::vector<std::vector<uint32_t>> batches;
        for (size_t q0 = 0; q0 < used.size(); q0 += 32) {
            const int nl = static_cast<int>(std::min<size_t>(32, used.size() - q0));
            const int d = static_cast<int>(list[used[q0]].size());
            std::vector<uint32_t> wd(33 + 32 * static_cast<size_t>(d), empty);
            wd[0] = static_cast<uint32_t>(d);
            for (int l = 0; l < 32; l++) wd[1 + l] = kNoCellW;
            for (int l = 0; l < nl; l++) {
                const int y = used[q0 + l] / 64, xp = used[q0 + l] % 64;
                wd[1 + l] = static_cast<uint32_t>(y * kWS + 2 * xp) | (static_cast<uint32_t>(y & 1) << 31);
            }
            for (int g0 = 0; g0 < 32; g0 += 8) {
                std::vector<uint32_t> rem[8];
                for (int l = 0; l < 8; l++)
                    if (g0 + l < nl) rem[l] = list[used[q0 + g0 + l]];
                for (int j = 0; j < d; j++) {
                    int slot[8] = {-1, -1, -1, -1, -1, -1, -1, -1}, first = -1;
                    for (int l = 0; l < 8; l++) {
                        auto &r = rem[l];
                        if (r.empty()) continue;
                        int pick = -1;
                        for (size_t q = 0; q < r.size() && pick < 0; q++) {
                            const int a = static_cast<int>(r[q] >> 8);
                            if (slot[a & 7] < 0 || slot[a & 7] == a) pick = static_cast<int>(q);
                        }
                        if (pick < 0 && static_cast<int>(r.size()) >= d - j) pick = 0;
                        if (pick < 0) continue;
                        const uint32_t e = r[pick];
                        r.erase(r.begin() + pick);
                        slot[(e >> 8) & 7] = static_cast<int>(e >> 8);
                        first = static_cast<int>(e >> 8);
                        wd[33 + 32 * static_cast<size_t>(j) + g0 + l] = e;
                    }
                    for (int l = 0; l < 8 && first >= 0; l++) {  // empty steps load an antenna the group loads anyway
                        uint32_t &e = wd[33 + 32 * static_cast<size_t>(j) + g0 + l];
                        if (e == empty) e = (static_cast<uint32_t>(first) << 8) | empty;
                    }
                }
            }
            batches.push_back(std::move(wd));
        }
        std::vector<std::vector<int>> per(W);
        std::vector<long long> load(W, 0);
        for (size_t b = 0; b < batches.size(); b++) {            // longest first already
            const int w = static_cast<int>(std::min_element(load.begin(), load.end()) - load.begin());
            per[w].push_back(static_cast<int>(b));
            load[w] += 4LL * batches[b][0] + 6;
        }
        auto &blk = blocks[bi];
        for (int w = 0; w < W; w++) {
            idx[static_cast<size_t>(bi) * W + w] = make_int2(static_cast<int>(blk.size()), static_cast<int>(per[w].size()));
            for (int b : per[w]) blk.insert(blk.end(), batches[b].begin(), batches[b].end());
        }
    };
    std::atomic<int> next{0};
    std::atomic<bool> nomem{false};
    auto worker = [&]() {
        for (int bi; !nomem && (bi = next++) < nbl;) {
            try {
                build(bi);
            } catch (const std::bad_alloc &) {
                nomem = true;
            }
        }
    };
    const int nt = threads > 0 ? std::min(nbl, threads)
                               : std::max(1, std::min({nbl, 16, static_cast<int>(std::thread::hardware_concurrency())}));
    std::vector<std::thread> pool;
    for (int i = 1; i < nt; i++) {
        try {
            pool.emplace_back(worker);
        } catch (...) {
            break;   // fewer threads: the calling thread takes the rest
        }
    }
    worker();
    for (auto &th : pool) th.join();
    if (nomem) return EPIC_ERR_NOMEM;
    tab.clear();
    for (int bi = 0; bi < nbl; bi++) {
        if (tab.size() + blocks[bi].size() > 0x7FFFFFFFull) return EPIC_ERR_UNSUPPORTED;
        for (int w = 0; w < W; w++) idx[static_cast<size_t>(bi) * W + w].x += static_cast<int>(tab.size());
        tab.insert(tab.end(), blocks[bi].begin(), blocks[bi].end());
        std::vector<uint32_t>().swap(blocks[bi]);
    }
    tab.resize(tab.size() + 33 + 4 * 32, 0u);   // spare words: the kernel loads a header and entries past a warp's last batch
    return EPIC_OK;
}

// Shared memory of the two kernels (row kernel, column kernel with the stages that fit); 0 stages: does not fit
size_t wide_rows_smem_bytes(int A, int K, bool gains) { return wide_rows_smem(A, K, gains); }
int wide_stages(int rpad, size_t smem_optin)
{
    int s = 3;
    while (s > 0 && wide_cols_smem(rpad, s) + 256 > smem_optin) s--;
    return s >= 2 ? s : 0;
}

// How an integration of T spectra in groups of cb channels runs: batches of at most tb spectra, each in
// n_sub chunks side by side, batch b adding to the partial images of round b mod rounds (n_sub rounds
// slots in all, every one of them written).  The fewest samples on the busiest SM, a chunk costing two
// more, one that continues earlier sums three, and a batch's launches four.  At side 256 no slot sums more spectra than a chunk of
// the per-class kernel (at side 512 the fold path adds all of them into one).
WideSplit wide_split(int N, int n_items, int cb, int tb, int slots, int T, int sms)
{
    const int blocks = cb * 2 * (N / 64), need = std::max(1, (T + tb - 1) / tb);
    const int n_min = N == 512 ? 1 : std::max(1, std::min(slots, fp32_pick_tau(n_items, T, sms)));
    WideSplit best{need, 1, 1, 1e300};
    for (int n = 1; n <= slots; n++) {
        const int rounds = need == 1 ? 1 : (n_min + n - 1) / n;
        if (rounds * n < n_min || rounds * n > slots) continue;
        WideSplit s{rounds * ((need + rounds - 1) / rounds), n, rounds, 0};
        const int nb = (T + s.batches - 1) / s.batches;
        if (n > 1 && n > nb) break;
        const long long waves = (static_cast<long long>(blocks) * n + sms - 1) / sms;
        s.cost = s.batches * (waves * ((nb + n - 1) / n + (s.batches > rounds ? 3.0 : 2.0)) + 4.0);
        if (s.cost < best.cost - 1e-9) best = s;
    }
    return best;
}

// Channels and spectra of a batch and the partial images of a plan: the workspace holds cb x tb channel
// samples within 4 GiB, the partial images stay within 2 GiB (or the tau_class of the per-class kernel).
// Few channels at a time leave SMs idle, many make short batches, so the cheapest split over the whole
// call decides.  16 channels, 300 antennas, side 512, 5000 spectra: in batches of 2500 of one channel with
// one chunk each 488 ms, in 19 chunks 72.9 (fold path 143); side 256, 9000 spectra 412, 46.0 (per class 58).
WideLayout wide_layout(int N, int n_chan, int rpad, int max_spectra, int cap_tb, int tau_class, int sms)
{
    constexpr size_t kWork = size_t(4) << 30, kSums = size_t(2) << 30;
    const size_t per = static_cast<size_t>(N) * 2 * rpad * sizeof(float2);
    const size_t slot = static_cast<size_t>(n_chan) * N * N * sizeof(float4);
    const int room = static_cast<int>(std::max<size_t>(1, kWork / per));   // channel samples
    const int n_items = n_chan * (N / 64) * (N / 64);
    const int slots = std::max(tau_class, static_cast<int>(std::max<size_t>(1, std::min<size_t>(kMaxTau, kSums / slot))));
    WideLayout best{1, 1, tau_class};
    double best_cost = 1e300;
    int last = 0;
    for (int groups = 1; groups <= n_chan; groups++) {
        const int cb = (n_chan + groups - 1) / groups;
        if (cb == last || cb > room) continue;
        last = cb;
        int tb = std::min(max_spectra, room / cb);
        if (cap_tb > 0) tb = std::min(tb, cap_tb);
        const WideSplit s = wide_split(N, n_items, cb, tb, slots, max_spectra, sms);
        double cost = s.cost * (n_chan / cb);
        if (n_chan % cb) cost += wide_split(N, n_items, n_chan % cb, tb, slots, max_spectra, sms).cost;
        if (cost < best_cost - 1e-9) {
            best_cost = cost;
            best = WideLayout{cb, tb, std::max(tau_class, s.n_sub * s.rounds)};
        }
    }
    return best;
}

// Whether an integration of T spectra is worth the two launches: for the smallest the per-class
// kernel's single launch is shorter.  Its time goes as the classes times transform and gridding, a
// footprint cell weighing three times the arithmetic's share (lists and shared-memory reads).  One
// GB300, us wide / per class: side 256, 300 antennas, 5 x 5, 2 channels x 16 spectra 40 / 34, 4 x 16
// 46 / 50; 2048 antennas, 7 x 7, 1 x 8 45 / 63; side 512, 2048 antennas, 7 x 7, 1 x 2 59 / 65, 1 x 4
// 60 / 107; 1000 antennas, 7 x 7, 1 x 4 54 / 47, 1 x 8 58 / 72; 300 antennas, 5 x 5, 1 x 16 60 / 54,
// 2 x 16 77 / 83; 64 antennas, 3 x 3, 2 x 16 109 / 97, 4 x 12 106 / 105.  (1 x 2 of 2048 antennas, 4.1e7
// by this count, lies on the wrong side; 1 x 4 of 1000, 4.2e7, asks for the line above both.)  At side 512
// the calls below the line went to the fold path before there were wide kernels: 84 us for 2048 antennas, 1 x 1
// (63 per class now), 66 for 1000, 1 x 2 (45), 92 for 300, 1 x 16 (51).
bool wide_pays(const epic_plan_s *plan, const GroupCfg &g, int T)
{
    const double work = static_cast<double>(g.n_items) * T * (3.0 * plan->A * plan->K * plan->K + 16384.0);
    return g.wforce || work >= (g.N == 512 ? 5.5e7 : 3e7);
}
int prepare_wide(const epic_plan_s *plan, const GroupCfg &g)
{
    const size_t rows = wide_rows_smem(plan->A, plan->K, g.wgains), cols = wide_cols_smem(g.wrpad, g.wstages);
    const bool big = g.N == 512;
    const int rc = raise_dyn_smem_cap(big ? reinterpret_cast<const void *>(wide_rows_kernel<8>)
                                          : reinterpret_cast<const void *>(wide_rows_kernel<4>), rows);
    return rc != EPIC_OK ? rc
                         : raise_dyn_smem_cap(big ? reinterpret_cast<const void *>(wide_cols_kernel<8>)
                                                  : reinterpret_cast<const void *>(wide_cols_kernel<4>), cols);
}

template <int Q>
static int launch_wide_t(epic_plan_s *plan, const GroupCfg &g, const uint8_t *v, const float2 *gains, int T, int *n_tau,
                         cudaStream_t stream)
{
    const size_t sm_rows = wide_rows_smem(plan->A, plan->K, g.wgains), sm_cols = wide_cols_smem(g.wrpad, g.wstages);
    const WideSplit split = wide_split(g.N, g.n_items, std::min(g.wcb, g.n_chan), g.wtb, g.tau_cap, T, plan->sm_count);
    *n_tau = split.n_sub * split.rounds;
    const size_t slot = static_cast<size_t>(g.n_items) * 64 * 64;
    for (int c0 = 0; c0 < g.n_chan; c0 += g.wcb) {
        const int nc = std::min(g.wcb, g.n_chan - c0);
        for (int b = 0; b < split.batches; b++) {
            const int tb0 = static_cast<int>(static_cast<long long>(T) * b / split.batches);
            const int nb = static_cast<int>(static_cast<long long>(T) * (b + 1) / split.batches) - tb0;
            const int s = b % split.rounds * split.n_sub;
            const int chunks = fp32_pick_tau(nc * g.wbands, nb, plan->sm_count);
            wide_rows_kernel<Q><<<static_cast<unsigned>(nc * g.wbands * chunks), kRowsThreads, sm_rows, stream>>>(
                v, gains, plan->d_kernel, plan->K, g.d_chans, g.d_wtab, g.d_widx, g.d_wchan, plan->A, plan->C, c0, g.wbands,
                tb0, nb, chunks, g.wrpad, g.wgains ? 1 : 0, plan->d_dfreq, plan->delays ? plan->d_dtab : nullptr, g.d_wws);
            wide_cols_kernel<Q><<<static_cast<unsigned>(nc * 2 * Q * split.n_sub), kColThreads, sm_cols, stream>>>(
                g.d_wws, nb, nc, split.n_sub, c0, g.wrpad, g.wstages, b >= split.rounds ? 1 : 0,
                reinterpret_cast<float4 *>(g.d_partial) + slot * s, slot, plan->d_status, plan->wait_budget);
            if (cudaGetLastError() != cudaSuccess) return EPIC_ERR_CUDA;
        }
    }
    return EPIC_OK;
}

int launch_wide(epic_plan_s *plan, const GroupCfg &g, const uint8_t *v, const float2 *gains, int T, int *n_tau,
                cudaStream_t stream)
{
    return g.N == 512 ? launch_wide_t<8>(plan, g, v, gains, T, n_tau, stream)
                      : launch_wide_t<4>(plan, g, v, gains, T, n_tau, stream);
}

}  // namespace epic
