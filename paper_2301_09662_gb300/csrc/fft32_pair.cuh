// 32-point DFTs of two signals at once, X[k] = sum_n x[n] exp(+2 pi i n k / 32), and
// the N = 32 Q point transforms built from them.
//
// The two signals (the two polarisations, or two samples of one) sit in the
// halves of packed FP32 pairs, real parts in one pair and imaginary parts in
// another: xr = (re a, re b), xi = (im a, im b).  Every operation is then one
// packed instruction for both, a turn by +-i is a choice of registers, and no
// lane is ever exchanged (with (re, im) pairs a turn or a twiddle needs two
// moves besides its two packed instructions: about a fifth of all instructions).
//
// With l = Q m + h, F(Q m + h) = sum_i w_32^{i m} [w_N^{i h} sum_q w_Q^{q h} x(i + 32 q)]: class h
// of the outputs is one 32-point transform of the inputs folded to 32 and turned
// by w_N^{i h}; inputs at 64 positions or fewer fold at most once.
#pragma once

#include "fft_class.cuh"

namespace epic {

// Twiddles as pairs for both signals: (re, re), (im, im), (-im, -im)
struct PairTwiddle {
    float2 re[32], im[32], ni[32];
};
constexpr PairTwiddle make_pair_twiddle(int num, int n)   // w_n^{num j}
{
    PairTwiddle t{};
    for (int j = 0; j < 32; j++) {
        const float2 w = ce_w(num * j, n);
        t.re[j] = float2{w.x, w.x};
        t.im[j] = float2{w.y, w.y};
        t.ni[j] = float2{-w.y, -w.y};
    }
    return t;
}
struct PairClassTwiddle {
    PairTwiddle h[4];
};
constexpr PairClassTwiddle make_pair_class_twiddle(int Q)
{
    PairClassTwiddle t{};
    for (int h = 0; h < 4; h++) t.h[h] = make_pair_twiddle(h, 32 * Q);
    return t;
}
__constant__ const PairTwiddle c_pw32 = make_pair_twiddle(1, 32);
__constant__ const PairClassTwiddle c_cls2 = make_pair_class_twiddle(2);
__constant__ const PairClassTwiddle c_cls3 = make_pair_class_twiddle(3);
__constant__ const PairClassTwiddle c_cls4 = make_pair_class_twiddle(4);

// (r, i) *= w, both signals
__device__ __forceinline__ void pair_mul(float2 &r, float2 &i, float2 wr, float2 wi, float2 wn)
{
    const float2 t = pfma(i, wn, pmul(r, wr));
    i = pfma(r, wi, pmul(i, wr));
    r = t;
}

__device__ __forceinline__ void pair_dft4(float2 (&r)[4], float2 (&i)[4])
{
    const float2 sr = padd(r[0], r[2]), si = padd(i[0], i[2]), dr = psub(r[0], r[2]), di = psub(i[0], i[2]);
    const float2 tr = padd(r[1], r[3]), ti = padd(i[1], i[3]), ur = psub(r[1], r[3]), ui = psub(i[1], i[3]);
    r[0] = padd(sr, tr);
    i[0] = padd(si, ti);
    r[2] = psub(sr, tr);
    i[2] = psub(si, ti);
    r[1] = psub(dr, ui);              // d + i u
    i[1] = padd(di, ur);
    r[3] = padd(dr, ui);              // d - i u
    i[3] = psub(di, ur);
}

__device__ __forceinline__ void pair_dft8(float2 (&r)[8], float2 (&i)[8])
{
    const float2 H = make_float2(kSqrtHalf, kSqrtHalf), NH = make_float2(-kSqrtHalf, -kSqrtHalf);
    float2 er[4] = {r[0], r[2], r[4], r[6]}, ei[4] = {i[0], i[2], i[4], i[6]};
    float2 o_r[4] = {r[1], r[3], r[5], r[7]}, o_i[4] = {i[1], i[3], i[5], i[7]};
    pair_dft4(er, ei);
    pair_dft4(o_r, o_i);
    r[0] = padd(er[0], o_r[0]);
    i[0] = padd(ei[0], o_i[0]);
    r[4] = psub(er[0], o_r[0]);
    i[4] = psub(ei[0], o_i[0]);
    const float2 v1r = psub(o_r[1], o_i[1]), v1i = padd(o_r[1], o_i[1]);   // w8 o / sqrt(1/2)
    r[1] = pfma(v1r, H, er[1]);
    i[1] = pfma(v1i, H, ei[1]);
    r[5] = pfma(v1r, NH, er[1]);
    i[5] = pfma(v1i, NH, ei[1]);
    r[2] = psub(er[2], o_i[2]);
    i[2] = padd(ei[2], o_r[2]);
    r[6] = padd(er[2], o_i[2]);
    i[6] = psub(ei[2], o_r[2]);
    const float2 v3r = padd(o_r[3], o_i[3]), v3i = psub(o_i[3], o_r[3]);   // -w8^3 o / sqrt(1/2)
    r[3] = pfma(v3r, NH, er[3]);
    i[3] = pfma(v3i, NH, ei[3]);
    r[7] = pfma(v3r, H, er[3]);
    i[7] = pfma(v3i, H, ei[3]);
}

// x(i), i < 8 nb (nb <= 8, the same in every lane; positions past the last occupied one are zeros in
// memory), from line[i * STRIDE] = (re a, re b, im a, im b), folded to 32 for class h of Q.  Whole
// blocks of eight: a test per position took as many instructions as the loads.
template <int Q, int STRIDE>
__device__ __forceinline__ void pair_load(float2 (&xr)[32], float2 (&xi)[32], const float4 *line, int nb, int h)
{
    static_assert(Q >= 1 && Q <= 4, "sides 32 to 128");
#pragma unroll
    for (int b = 0; b < 4; b++) {
        if (b < nb) {
#pragma unroll
            for (int i = 8 * b; i < 8 * b + 8; i++) {
                const float4 v = line[i * STRIDE];
                xr[i] = make_float2(v.x, v.y);
                xi[i] = make_float2(v.z, v.w);
            }
        } else {
#pragma unroll
            for (int i = 8 * b; i < 8 * b + 8; i++) xr[i] = xi[i] = make_float2(0.f, 0.f);
        }
    }
    if constexpr (Q > 1) {
        // + w_Q^h x(i + 32)
        const float2 gr = Q == 3 ? (h ? make_float2(-0.5f, -0.5f) : make_float2(1.f, 1.f))
                                 : (h & (Q / 2) ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f));
        const float2 gi = Q == 3 ? (h == 0   ? make_float2(0.f, 0.f)
                                    : h == 1 ? make_float2(kSin60, kSin60)
                                             : make_float2(-kSin60, -kSin60))
                                 : (h == 1 ? make_float2(1.f, 1.f) : make_float2(-1.f, -1.f));
        const float2 gn = make_float2(-gi.x, -gi.y);
#pragma unroll
        for (int b = 0; b < 4; b++) {
            if (b + 4 < nb) {
                if (Q == 4 && (h & 1)) {             // +-i
#pragma unroll
                    for (int i = 8 * b; i < 8 * b + 8; i++) {
                        const float4 v = line[(i + 32) * STRIDE];
                        xr[i] = pfma(make_float2(v.z, v.w), gn, xr[i]);
                        xi[i] = pfma(make_float2(v.x, v.y), gi, xi[i]);
                    }
                } else {
#pragma unroll
                    for (int i = 8 * b; i < 8 * b + 8; i++) {
                        const float4 v = line[(i + 32) * STRIDE];
                        const float2 vr = make_float2(v.x, v.y), vi = make_float2(v.z, v.w);
                        xr[i] = pfma(vr, gr, xr[i]);
                        xi[i] = pfma(vi, gr, xi[i]);
                        if constexpr (Q == 3) {
                            xr[i] = pfma(vi, gn, xr[i]);
                            xi[i] = pfma(vr, gi, xi[i]);
                        }
                    }
                }
            }
        }
    }
}

template <int Q, int H>
__device__ __forceinline__ void pair_turn_h(float2 (&xr)[32], float2 (&xi)[32], int nb)
{
    const PairClassTwiddle &c = Q == 2 ? c_cls2 : Q == 3 ? c_cls3 : c_cls4;
#pragma unroll
    for (int b = 0; b < 4; b++) {
        if (b < nb) {
#pragma unroll
            for (int i = b ? 8 * b : 1; i < 8 * b + 8; i++) pair_mul(xr[i], xi[i], c.h[H].re[i], c.h[H].im[i], c.h[H].ni[i]);
        }
    }
}
// the class turn w_N^{i h}
template <int Q>
__device__ __forceinline__ void pair_turn(float2 (&xr)[32], float2 (&xi)[32], int nb, int h)
{
    if (Q > 1 && h == 1) pair_turn_h<Q, 1>(xr, xi, nb);
    if (Q > 2 && h == 2) pair_turn_h<Q, 2>(xr, xi, nb);
    if (Q > 3 && h == 3) pair_turn_h<Q, 3>(xr, xi, nb);
}

// The 32-point transforms as 8 x 4, in eight groups: group(k1, r, i) receives X[k1 + 8 k2], k2 < 4
template <class Group>
__device__ __forceinline__ void pair_fft32(float2 (&xr)[32], float2 (&xi)[32], Group &&group)
{
#pragma unroll
    for (int n2 = 0; n2 < 4; n2++) {
        float2 r[8], i[8];
#pragma unroll
        for (int n1 = 0; n1 < 8; n1++) {
            r[n1] = xr[n2 + 4 * n1];
            i[n1] = xi[n2 + 4 * n1];
        }
        pair_dft8(r, i);
#pragma unroll
        for (int k1 = 0; k1 < 8; k1++) {
            const int j = n2 * k1;
            if (j == 8) {                            // i
                xr[n2 + 4 * k1] = make_float2(-i[k1].x, -i[k1].y);
                xi[n2 + 4 * k1] = r[k1];
                continue;
            }
            if (j) pair_mul(r[k1], i[k1], c_pw32.re[j], c_pw32.im[j], c_pw32.ni[j]);
            xr[n2 + 4 * k1] = r[k1];
            xi[n2 + 4 * k1] = i[k1];
        }
    }
#pragma unroll
    for (int k1 = 0; k1 < 8; k1++) {
        float2 r[4], i[4];
#pragma unroll
        for (int n2 = 0; n2 < 4; n2++) {
            r[n2] = xr[n2 + 4 * k1];
            i[n2] = xi[n2 + 4 * k1];
        }
        pair_dft4(r, i);
        group(k1, r, i);
    }
}

}  // namespace epic
