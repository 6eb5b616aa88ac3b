// Complex values in pairs: the register DFTs of the L = 4096 filter.
//
// The spread segment is zero at every odd cell, so the inverse transform of
// length L splits into two of length L/2 that run through the same steps: one
// gives the even cells (on X (G[f] + G[f + L/2])), one the odd cells (on X
// (G[f] - G[f + L/2]) times a twiddle the bank holds).  A thread keeps point f
// of both side by side: `re` and `im` each hold (even, odd) in an aligned
// register pair, so every butterfly and every twiddle product is packed FP32
// (add/sub/mul/fma .f32x2), a rotation by +-i only renames registers, and one
// instruction serves two points.  Sign +1 (inverse) throughout.
#pragma once

#include "fft.cuh"

namespace jerk {

struct cpair {
    float2 re, im;
};

__device__ __forceinline__ cpair operator+(cpair a, cpair b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ cpair operator-(cpair a, cpair b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a + i b and a - i b
__device__ __forceinline__ cpair add_i(cpair a, cpair b) { return {sub2(a.re, b.im), add2(a.im, b.re)}; }
__device__ __forceinline__ cpair sub_i(cpair a, cpair b) { return {add2(a.re, b.im), sub2(a.im, b.re)}; }
// a + k q, k real
__device__ __forceinline__ cpair axpy(float k, cpair q, cpair a) { return {fma2k(k, q.re, a.re), fma2k(k, q.im, a.im)}; }
// a times w, each lane its own or (broadcast) the same
__device__ __forceinline__ cpair mul(cpair a, float2 wr, float2 wi) {
    return {sub2(mul2(a.re, wr), mul2(a.im, wi)), fma2(a.re, wi, mul2(a.im, wr))};
}
// a times the constant c + i s
__device__ __forceinline__ cpair mulc(cpair a, float c, float s) {
    return {fma2k(-s, a.im, mul2(a.re, make_float2(c, c))), fma2k(s, a.re, mul2(a.im, make_float2(c, c)))};
}
// (u, v) with exp(2 pi i / 8) b = (u + i v) / sqrt 2
__device__ __forceinline__ cpair eighth1(cpair b) { return {sub2(b.re, b.im), add2(b.im, b.re)}; }

__device__ __forceinline__ void dft4(cpair &a0, cpair &a1, cpair &a2, cpair &a3) {
    const cpair s02 = a0 + a2, d02 = a0 - a2, s13 = a1 + a3, e13 = a1 - a3;
    a0 = s02 + s13;
    a2 = s02 - s13;
    a1 = add_i(d02, e13);
    a3 = sub_i(d02, e13);
}

// y_r = sum_k a_k exp(2 pi i k r / 8), natural order: the split of dft8 in fft.cuh
__device__ __forceinline__ void dft8(cpair &a0, cpair &a1, cpair &a2, cpair &a3, cpair &a4, cpair &a5, cpair &a6,
                                     cpair &a7) {
    dft4(a0, a2, a4, a6);
    dft4(a1, a3, a5, a7);
    const cpair c0 = a0, c1 = a2, c2 = a4, c3 = a6;            // even k: outputs 0..3
    const cpair o0 = a1, o1 = a3, o2 = a5, o3 = a7;
    a0 = c0 + o0;
    a4 = c0 - o0;
    const cpair q1 = eighth1(o1);
    a1 = axpy(kRsqrt2, q1, c1);
    a5 = axpy(-kRsqrt2, q1, c1);
    a2 = add_i(c2, o2);
    a6 = sub_i(c2, o2);
    const cpair s = {add2(o3.re, o3.im), sub2(o3.im, o3.re)};  // -(u, v) of exp(6 pi i / 8) o3
    a3 = axpy(-kRsqrt2, s, c3);
    a7 = axpy(kRsqrt2, s, c3);
}

// y_r = sum_k a_k exp(2 pi i k r / 16): the 4 x 4 split of dft16 in fft.cuh, after its
// first stage (dft4 of a[k1], a[k1 + 4], a[k1 + 8], a[k1 + 12] for k1 = 0 .. 3)
__device__ __forceinline__ void dft16_rest(cpair (&a)[16]) {
    constexpr float C1 = 0.92387953251128674f, S1 = 0.38268343236508977f;
    cpair y[16];
    {
        cpair x0 = a[0], x1 = a[1], x2 = a[2], x3 = a[3];
        dft4(x0, x1, x2, x3);
        y[0] = x0;
        y[4] = x1;
        y[8] = x2;
        y[12] = x3;
    }
    {
        const cpair q = eighth1(a[6]);
        const cpair s02 = axpy(kRsqrt2, q, a[4]), d02 = axpy(-kRsqrt2, q, a[4]);
        const cpair x1 = mulc(a[5], C1, S1), x3 = mulc(a[7], S1, C1);
        const cpair s13 = x1 + x3, e13 = x1 - x3;
        y[1] = s02 + s13;
        y[9] = s02 - s13;
        y[5] = add_i(d02, e13);
        y[13] = sub_i(d02, e13);
    }
    {
        const cpair s02 = add_i(a[8], a[10]), d02 = sub_i(a[8], a[10]);
        const cpair e = add_i(a[9], a[11]), f = sub_i(a[9], a[11]);   // x1 + x3 = w^2 e, x1 - x3 = w^2 f
        const cpair qe = eighth1(e), qf = eighth1(f);
        y[2] = axpy(kRsqrt2, qe, s02);
        y[10] = axpy(-kRsqrt2, qe, s02);
        // +- i w^2 f = +- (-qf.im, qf.re) / sqrt 2
        y[6] = {fma2k(-kRsqrt2, qf.im, d02.re), fma2k(kRsqrt2, qf.re, d02.im)};
        y[14] = {fma2k(kRsqrt2, qf.im, d02.re), fma2k(-kRsqrt2, qf.re, d02.im)};
    }
    {
        const cpair s = {add2(a[14].re, a[14].im), sub2(a[14].im, a[14].re)};   // -(u, v) of exp(6 pi i / 8) a[14]
        const cpair s02 = axpy(-kRsqrt2, s, a[12]), d02 = axpy(kRsqrt2, s, a[12]);
        const cpair x1 = mulc(a[13], S1, C1), x3 = mulc(a[15], -C1, -S1);
        const cpair s13 = x1 + x3, e13 = x1 - x3;
        y[3] = s02 + s13;
        y[11] = s02 - s13;
        y[7] = add_i(d02, e13);
        y[15] = sub_i(d02, e13);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) a[i] = y[i];
}

__device__ __forceinline__ void dft16(cpair (&a)[16]) {
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) dft4(a[k1], a[k1 + 4], a[k1 + 8], a[k1 + 12]);
    dft16_rest(a);
}

}  // namespace jerk
