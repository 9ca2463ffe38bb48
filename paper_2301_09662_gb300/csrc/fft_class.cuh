// Pixel-class form of an N-point DFT whose input occupies at most 64 positions:
// with l = Q m + h, F(Q m + h) = sum_i w_M^{i m} [w_N^{i h} x(i)], M = N / Q, so each
// class h is one M-point register transform of the same inputs, turned by
// w_N^{i h} (and, at M = 48, folded from 64 to 48 positions).
#pragma once

#include "fft48.cuh"

namespace epic {

// exp(+2 pi i j / n), n a multiple of 8, with exact reduction on the integer j
constexpr float2 ce_w(int j, int n)
{
    j = ((j % n) + n) % n;
    const int q = j / (n / 4), r = j % (n / 4);
    const double step = 2.0 * 3.14159265358979323846 / n;
    double c = 0, s = 0;
    if (8 * r <= n) {
        c = ce_cos_q(r * step);
        s = ce_sin_q(r * step);
    } else {
        c = ce_sin_q((n / 4 - r) * step);
        s = ce_cos_q((n / 4 - r) * step);
    }
    double re = c, im = s;
    for (int i = 0; i < q; i++) {
        const double t = re;
        re = -im;
        im = t;
    }
    return float2{static_cast<float>(re), static_cast<float>(im)};
}

// w_N^i for the odd class of N = 2 M, as lane pairs (re, re) and (-im, im)
template <int M>
struct ClassTwiddle {
    float2 rr[M], ni[M];
};
template <int M>
constexpr ClassTwiddle<M> make_class_twiddle()
{
    ClassTwiddle<M> t{};
    for (int i = 0; i < M; i++) {
        const float2 w = ce_w(i, 2 * M);
        t.rr[i] = float2{w.x, w.x};
        t.ni[i] = float2{-w.y, w.y};
    }
    return t;
}
__constant__ const ClassTwiddle<64> c_cls64 = make_class_twiddle<64>();
__constant__ const ClassTwiddle<48> c_cls48 = make_class_twiddle<48>();

// x(i), i < 8 nb (nb <= 8, the same in every lane; the positions past the last occupied one are
// zeros in memory), from line[i * STRIDE], folded to M for class h.  Whole blocks of eight: a test
// per position took as many instructions as the loads.
template <int M, int STRIDE>
__device__ __forceinline__ void class_load(float2 (&x)[M], const float2 *line, int nb, int h)
{
#pragma unroll
    for (int b = 0; b < M / 8; b++) {
        if (b < nb) {
#pragma unroll
            for (int i = 8 * b; i < 8 * b + 8; i++) x[i] = line[i * STRIDE];
        } else {
#pragma unroll
            for (int i = 8 * b; i < 8 * b + 8; i++) x[i] = make_float2(0.f, 0.f);
        }
    }
    if constexpr (M == 48) {
        // w_96^{(i + 48) h} = (-1)^h w_96^{i h}
        const float2 sg = h ? make_float2(-1.f, -1.f) : make_float2(1.f, 1.f);
#pragma unroll
        for (int b = 0; b < 2; b++) {
            if (b + 6 < nb) {
#pragma unroll
                for (int i = 8 * b; i < 8 * b + 8; i++) x[i] = pfma(line[(i + 48) * STRIDE], sg, x[i]);
            }
        }
    }
}

template <int M>
__device__ __forceinline__ void class_turn(float2 (&x)[M], int nb, int h)
{
    if (h) {
#pragma unroll
        for (int b = 0; b < M / 8; b++) {
            if (b < nb) {
#pragma unroll
                for (int i = b ? 8 * b : 1; i < 8 * b + 8; i++) {
                    if constexpr (M == 64) x[i] = pfma(pswap(x[i]), c_cls64.ni[i], pmul(x[i], c_cls64.rr[i]));
                    else x[i] = pfma(pswap(x[i]), c_cls48.ni[i], pmul(x[i], c_cls48.rr[i]));
                }
            }
        }
    }
}

// The M-point transform in eight groups: group(k1, t) receives t[k2] = X[k1 + 8 k2], k2 < M / 8
template <int M, class Group>
__device__ __forceinline__ void fft_groups(float2 (&x)[M], Group &&group)
{
    if constexpr (M == 64) {
        fft64p_stage1(x);
#pragma unroll
        for (int k1 = 0; k1 < 8; k1++) {
            float2 t[8];
#pragma unroll
            for (int n2 = 0; n2 < 8; n2++) t[n2] = x[n2 + 8 * k1];
            dft8p(t);
            group(k1, t);
        }
    } else {
        fft48p_stage1(x);
#pragma unroll
        for (int k1 = 0; k1 < 8; k1++) {
            float2 t[6];
#pragma unroll
            for (int n2 = 0; n2 < 6; n2++) t[n2] = x[6 * k1 + n2];
            dft6p(t);
            group(k1, t);
        }
    }
}

}  // namespace epic
