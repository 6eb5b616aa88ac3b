// FP64 template generation on the GPU (off the timed path).
//
// Sec. 2: "each filter fits a specific Fourier response for a given first
// frequency derivative z = fdot T^2 and second frequency derivative
// w = fddot T^3".  The response of a unit signal whose frequency,
// fdot T^2 and fddot T^3 at mid-observation are (r, z, w), at frequency
// offset q bins, is
//     rho(q; z, w) = int_{-1/2}^{1/2} exp(2 pi i (-q u + z u^2/2 + w u^3/6)) du
// and the matched-filter taps are c_d = conj(rho(d/b; z, w)), |d| <= b m(z, w).
//
// The integral is evaluated by composite 64-node Gauss-Legendre quadrature
// with J equal panels, J fixed by the widest template of the bank so that no
// panel holds more than 20 cycles of the integrand (64 nodes integrate 20
// cycles to 1e-24, 24 to 1e-14: far below FP64 rounding).  With u = a_j + s_i,
// a_j = -1/2 + j/J, s_i = (x_i + 1)/(2J), and q = d/2,
//     rho(d/2) = i^d sum_i exp(-pi i d s_i) A_i(d),
//     A_i(d) = sum_j c_{j,i} exp(-pi i d j/J),
// c_{j,i} = W_i/(2J) exp(2 pi i (z u^2/2 + w u^3/6)).  A_i has period 2J in d,
// so a template needs 64 x 2J sums of J terms once and then 64 terms per tap
// instead of 64 J; the nodes +-x_i share their factors: with theta = pi d x_i/(2J),
//     exp(-i theta) A_{+} + exp(i theta) A_{-} = cos theta S_i - i sin theta D_i,
// S = A_+ + A_-, D = A_+ - A_- (half the products), and cos, sin of every (i, |d|)
// come from a table made once per bank.
//
// Conjugation and reversal of the integral give rho(q; -z, w) = conj rho(q; z, w)
// and rho(q; z, -w) = rho(-q; z, w), so jerk_templates evaluates only the
// templates with z, w >= 0 and writes up to four bank rows from each FP64
// transform: with Ghat[f] = (1/L) sum_d c_d exp(2 pi i f d/L) the rows of
// (-z, w), (z, -w) and (-z, -w) are conj Ghat[-f], Ghat[-f] and conj Ghat[f],
// each times exp(2 pi i f bM/L), bM its own group's tap offset, in FP64 before
// the one rounding to FP32.  Bank of 12 261 templates at L = 4096 (201 x 61,
// 765 taps): 173.2 ms -> 3.95 ms, of which the FP64 pipe needs about 3.
#include <cmath>
#include <vector>

#include "jerk_internal.h"

namespace jerk {

// Gauss-Legendre nodes/weights on [-1, 1] by Newton iteration on P_n.
void gauss_legendre(int n, std::vector<double> &x, std::vector<double> &w) {
    x.assign(n, 0.0);
    w.assign(n, 0.0);
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < (n + 1) / 2; ++i) {
        double z = std::cos(pi * (i + 0.75) / (n + 0.5));
        double dp = 0.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = p2;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            const double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        // recompute the derivative at the converged root
        double p0 = 1.0, p1 = z;
        for (int k = 2; k <= n; ++k) {
            const double p2 = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
            p0 = p1;
            p1 = p2;
        }
        dp = n * (z * p1 - p0) / (z * z - 1.0);
        x[i] = -z;
        x[n - 1 - i] = z;
        w[i] = w[n - 1 - i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

constexpr int kGL = 64;            // nodes per panel
constexpr int kPairs = kGL / 2;    // node pairs +-x
constexpr double kCyclesPerPanel = 20.0;

__device__ __forceinline__ int halfwidth_dev(int z, int w, int pad) {
    return (4 * abs(z) + abs(w) + 7) / 8 + pad;
}

// panels for a bank of half-width M = bM / b (|z|/2 + |w|/8 <= M - pad, |q| <= M)
static int tap_panels(int M, int pad) { return (int)std::ceil((2.0 * M - pad) / kCyclesPerPanel) + 1; }

// tab[i][d], i < 32: (cos, sin) of pi d x_i / (2J), x_i the positive nodes;
// tab[32][d]: i^d exp(-pi i d / (2J)); d = 0 .. bM
__global__ void tap_table_kernel(double2 *tab, const double2 *gl, int J, int bM) {
    const int d = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (d > bM) return;
    double s, c;
    if (i < kPairs)
        sincospi((double)d * gl[kPairs + i].x / (2.0 * J), &s, &c);
    else
        // d/2 - d/(2J) half turns, reduced exactly: d (J - 1) mod 4J over 2J
        sincospi((double)(((int64_t)d * (J - 1)) % (4 * J)) / (2.0 * J), &s, &c);
    tab[(int64_t)i * (bM + 1) + d] = make_double2(c, s);
}

// One CTA per template.  What bounds it is the FP64 pipe (about 2 fused
// multiply-adds per clock and SM): 64 J phases, 256 J^2 of them for S and D and
// 128 K for the K taps, 0.3 M at J = 20, K = 765, where summing every panel at
// every tap took 18 M.  `ib` node pairs at a time sit in shared memory (all 32
// unless J is very large); later ones add to the taps stored before.
__global__ void __launch_bounds__(256) taps_kernel(const int32_t *__restrict__ zt, const int32_t *__restrict__ wt,
                                                   const int32_t *__restrict__ tlist, int32_t t0, int b, int pad,
                                                   int bM, int J, int ib, const double2 *__restrict__ gl,
                                                   const double2 *__restrict__ tab, double2 *__restrict__ out) {
    extern __shared__ double2 sm[];
    double2 *root = sm;                       // [2J] exp(-pi i k / J)
    double2 *chirp = root + 2 * J;            // [2 ib][J]: node pair p at rows 2p (x > 0) and 2p + 1 (x < 0)
    double2 *S = chirp + 2 * ib * J;          // [ib][2J]
    double2 *D = S + 2 * ib * J;              // [ib][2J]
    const int t = tlist ? tlist[blockIdx.x] : t0 + (int)blockIdx.x;
    const int K = 2 * bM + 1;
    double2 *dst = out + (int64_t)blockIdx.x * K;
    const int zi = zt[t], wi = wt[t];
    const double z = zi, w = wi;
    const int reach = b * halfwidth_dev(zi, wi, pad);
    const double h = 1.0 / J;
    for (int k = threadIdx.x; k < 2 * J; k += blockDim.x) {
        double s, c;
        sincospi(-(double)k / J, &s, &c);
        root[k] = make_double2(c, s);
    }
    for (int p0 = 0; p0 < kPairs; p0 += ib) {
        __syncthreads();                      // (the previous pairs' S and D are read)
        for (int n = threadIdx.x; n < 2 * ib * J; n += blockDim.x) {
            const int row = n / J, j = n - row * J, p = p0 + (row >> 1);
            const double2 g = gl[(row & 1) ? kPairs - 1 - p : kPairs + p];
            // u = (2j + 1 - J + x) / (2J) and its rounding error ul: at up to
            // |z|/2 + |w|/8 cycles per unit of u the error would be the phase's largest
            // (taps of z, w up to 200, 600: 1.0e-14 of their norm off, 2.3e-15 with it)
            const double m = 2 * j + 1 - J, nu = m + g.x, nl = g.x - (nu - m);   // (exact for m = 0 too)
            const double u = nu * (0.5 * h), ul = (fma(-u, 2.0 * J, nu) + nl) * (0.5 * h);
            double ph = z * u * u / 2.0 + w * u * u * u / 6.0;     // cycles
            ph -= rint(ph);
            ph = fma(ul, u * (z + 0.5 * w * u), ph);
            double s, c;
            sincospi(2.0 * ph, &s, &c);
            const double wt_ = g.y * 0.5 * h;
            chirp[n] = make_double2(wt_ * c, wt_ * s);
        }
        __syncthreads();
        // A(e) and A(e + J) = (even j) +- (odd j), for both nodes of a pair
        for (int n = threadIdx.x; n < ib * J; n += blockDim.x) {
            const int p = n / J, e = n - p * J;
            const double2 *cp = chirp + 2 * p * J, *cm = cp + J;
            double pr[2] = {0.0, 0.0}, pi[2] = {0.0, 0.0}, mr[2] = {0.0, 0.0}, mi[2] = {0.0, 0.0};
            int k = 0;                        // e j mod 2J
            for (int j = 0; j < J; j += 2) {
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    if (j + o < J) {
                        const double2 r = root[k], x = cp[j + o], y = cm[j + o];
                        pr[o] = fma(x.x, r.x, fma(-x.y, r.y, pr[o]));
                        pi[o] = fma(x.x, r.y, fma(x.y, r.x, pi[o]));
                        mr[o] = fma(y.x, r.x, fma(-y.y, r.y, mr[o]));
                        mi[o] = fma(y.x, r.y, fma(y.y, r.x, mi[o]));
                        k += e;
                        if (k >= 2 * J) k -= 2 * J;
                    }
                }
            }
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const double f = o ? -1.0 : 1.0;
                const double ar = fma(f, pr[1], pr[0]), ai = fma(f, pi[1], pi[0]);
                const double br = fma(f, mr[1], mr[0]), bi = fma(f, mi[1], mi[0]);
                S[p * 2 * J + e + o * J] = make_double2(ar + br, ai + bi);
                D[p * 2 * J + e + o * J] = make_double2(ar - br, ai - bi);
            }
        }
        __syncthreads();
        for (int d = -bM + (int)threadIdx.x; d <= bM; d += blockDim.x) {
            double2 res = make_double2(0.0, 0.0);
            if (abs(d) <= reach) {
                int e = d % (2 * J);
                if (e < 0) e += 2 * J;
                const double2 *tb = tab + (int64_t)p0 * (bM + 1) + abs(d);
                double xr = 0.0, xi = 0.0, yr = 0.0, yi = 0.0;
                for (int p = 0; p < ib; ++p) {
                    const double2 cs = __ldg(tb + (int64_t)p * (bM + 1));
                    const double2 s = S[p * 2 * J + e], v = D[p * 2 * J + e];
                    xr = fma(cs.x, s.x, xr);
                    xi = fma(cs.x, s.y, xi);
                    yr = fma(cs.y, v.y, yr);
                    yi = fma(cs.y, v.x, yi);
                }
                // cos S - i sin D; sin is odd in d
                const double re = d < 0 ? xr - yr : xr + yr, im = d < 0 ? xi + yi : xi - yi;
                const double2 ph = __ldg(tab + (int64_t)kPairs * (bM + 1) + abs(d));
                const double py = d < 0 ? -ph.y : ph.y;
                res = make_double2(re * ph.x - im * py, -(re * py + im * ph.x));   // c_d = conj(rho(d/b))
                if (p0 > 0) {
                    res.x += dst[d + bM].x;
                    res.y += dst[d + bM].y;
                }
            }
            dst[d + bM] = res;
        }
    }
}

// tw[i] = exp(+2 pi i i / L), i < L
__global__ void twiddle64_kernel(double2 *tw, int L) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < L) {
        double s, c;
        sincospi(2.0 * i / L, &s, &c);
        tw[i] = make_double2(c, s);
    }
}

__device__ __forceinline__ double2 cmul64(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// The bank rows of the templates (+-z, +-w) from the taps of (z, w): the
// centred transform Ghat (header comment) by radix-4 passes in shared memory
// (one radix-2 pass first when log2 L is odd), then each row's symmetry, its
// group's offset phase and its stored form.  dest[4 i + q] is the bank row of
// the template with z negated (q & 1) and w negated (q & 2), or -1, and
// offs[4 i + q] the tap offset bM of its group; bm the bank-wide offset of `taps`.
//
// fold_r0 > 0 stores a row in the folded form the FP32 filter multiplies
// with (its inverse transform's first pass has radix R0 = fold_r0 over the
// elements f = j + (L/16)(i + (16/R0) k)): the spread segment has zeros at
// every odd cell, so its spectrum X has period L/2, and that pass splits
// into two DFTs of R0/2 points on, for f < L/2,
//   Ge[f] = G[f] + G[f + L/2],
//   Go[f] = (G[f] - G[f + L/2]) exp(+2 pi i k / R0),  k = (f / (L/16)) / (16 / R0),
// both computed in FP64 before the one rounding to FP32 and stored
// interleaved, row[2 f] = Ge[f], row[2 f + 1] = Go[f], so that one 16-byte
// shared-memory load gives a thread both factors of its spectrum value X[f].
// fold_r0 < 0 stores the paired form of the tensor-core filter: values f and
// f + P (P = -fold_r0, bit log2 P of f clear) side by side as (Re f, Re f+P)
// (Im f, Im f+P) at float2 slots 2 q and 2 q + 1, q = f with that bit removed,
// so that one 16-byte load feeds a packed product of two values.
// *cmax receives the maximum of |Re| and |Im| over what is stored.
__global__ void __launch_bounds__(512) template_fft_kernel(const double2 *__restrict__ taps,
                                                           const int32_t *__restrict__ dest,
                                                           const int32_t *__restrict__ offs, int bm, int L,
                                                           int log2L, const double2 *__restrict__ tw, int fold_r0,
                                                           float2 *__restrict__ bank, int *__restrict__ cmax) {
    extern __shared__ double2 buf[];   // [L]
    const double2 *c = taps + (int64_t)blockIdx.x * (2 * bm + 1) + bm;
    const double inv = 1.0 / L;
    for (int m = threadIdx.x; m < L; m += blockDim.x) {
        const int d = m < L / 2 ? m : m - L;
        double2 v = make_double2(0.0, 0.0);
        if (abs(d) <= bm) v = make_double2(c[d].x * inv, c[d].y * inv);
        buf[__brev(m) >> (32 - log2L)] = v;
    }
    __syncthreads();
    int len = 1;                       // length of the sub-transforms done
    if (log2L & 1) {
        for (int i = threadIdx.x; i < L / 2; i += blockDim.x) {
            const double2 x = buf[2 * i], y = buf[2 * i + 1];
            buf[2 * i] = make_double2(x.x + y.x, x.y + y.y);
            buf[2 * i + 1] = make_double2(x.x - y.x, x.y - y.y);
        }
        len = 2;
        __syncthreads();
    }
    for (; len < L; len <<= 2) {
        // four sub-transforms of len points, bit-reversed order (0, 2, 1, 3), into one of 4 len
        const int step = L / (4 * len);
        for (int i = threadIdx.x; i < L / 4; i += blockDim.x) {
            const int k = i & (len - 1), i0 = ((i - k) << 2) + k;
            double2 x0 = buf[i0], x2 = buf[i0 + len], x1 = buf[i0 + 2 * len], x3 = buf[i0 + 3 * len];
            if (len > 1) {
                x1 = cmul64(x1, __ldg(tw + k * step));
                x2 = cmul64(x2, __ldg(tw + 2 * k * step));
                x3 = cmul64(x3, __ldg(tw + 3 * k * step));
            }
            const double2 s02 = make_double2(x0.x + x2.x, x0.y + x2.y), d02 = make_double2(x0.x - x2.x, x0.y - x2.y);
            const double2 s13 = make_double2(x1.x + x3.x, x1.y + x3.y), d13 = make_double2(x1.x - x3.x, x1.y - x3.y);
            buf[i0] = make_double2(s02.x + s13.x, s02.y + s13.y);
            buf[i0 + len] = make_double2(d02.x - d13.y, d02.y + d13.x);
            buf[i0 + 2 * len] = make_double2(s02.x - s13.x, s02.y - s13.y);
            buf[i0 + 3 * len] = make_double2(d02.x + d13.y, d02.y - d13.x);
        }
        __syncthreads();
    }
    float top = 0.f;
    for (int q = 0; q < 4; ++q) {
        const int row = dest[4 * blockIdx.x + q];
        if (row < 0) continue;
        const int off = offs[4 * blockIdx.x + q];
        const bool mirror = q == 1 || q == 2, conj = q & 1;
        auto value = [&](int f) {
            double2 v = buf[mirror ? (L - f) & (L - 1) : f];
            if (conj) v.y = -v.y;
            return cmul64(v, __ldg(tw + (int)(((int64_t)f * off) & (L - 1))));
        };
        float4 *dst = reinterpret_cast<float4 *>(bank + (int64_t)row * L);
        for (int i = threadIdx.x; i < L / 2; i += blockDim.x) {
            float4 o;
            if (fold_r0 > 0) {
                const double2 u = value(i), v = value(i + L / 2);
                const int k = (i / (L / 16)) / (16 / fold_r0);
                const double2 d = cmul64(make_double2(u.x - v.x, u.y - v.y), __ldg(tw + k * (L / fold_r0)));
                o = make_float4((float)(u.x + v.x), (float)(u.y + v.y), (float)d.x, (float)d.y);
            } else if (fold_r0 < 0) {
                const int P = -fold_r0, f = (i & (P - 1)) | ((i & ~(P - 1)) << 1);
                const double2 u = value(f), v = value(f + P);
                o = make_float4((float)u.x, (float)v.x, (float)u.y, (float)v.y);
            } else {
                const double2 u = value(2 * i), v = value(2 * i + 1);
                o = make_float4((float)u.x, (float)u.y, (float)v.x, (float)v.y);
            }
            dst[i] = o;
            top = fmaxf(fmaxf(top, fmaxf(fabsf(o.x), fabsf(o.y))), fmaxf(fabsf(o.z), fabsf(o.w)));
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    if ((threadIdx.x & 31) == 0) atomicMax(cmax, __float_as_int(top));   // non-negative floats compare as ints
}

size_t tap_table_elems(int bM) { return (size_t)(kPairs + 1) * (bM + 1); }

cudaError_t launch_tap_table(double2 *tab, const double2 *gl, int b, int bM, int pad, cudaStream_t st) {
    const dim3 grid((bM + 256) / 256, kPairs + 1);
    tap_table_kernel<<<grid, 256, 0, st>>>(tab, gl, tap_panels(bM / b, pad), bM);
    return cudaGetLastError();
}

cudaError_t launch_taps(const int32_t *zt, const int32_t *wt, const int32_t *tlist, int32_t t0, int32_t nt, int b,
                        int pad, int bM, const double2 *gl, const double2 *tab, double2 *out, cudaStream_t st) {
    if (b != 2) return cudaErrorInvalidValue;     // the period 2J of the panel sums is that of half-bin steps
    const int J = tap_panels(bM / b, pad);
    // node pairs at a time: all 32 below 96 KB of shared memory (two CTAs per SM), fewer for very wide banks
    int ib = kPairs;
    auto bytes = [&] { return (size_t)(2 * J + 6 * ib * J) * sizeof(double2); };
    while (ib > 4 && bytes() > (96u << 10)) ib /= 2;
    cudaError_t e = cudaFuncSetAttribute(taps_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes());
    if (e != cudaSuccess) return e;
    taps_kernel<<<nt, 256, bytes(), st>>>(zt, wt, tlist, t0, b, pad, bM, J, ib, gl, tab, out);
    return cudaGetLastError();
}

cudaError_t launch_twiddles64(double2 *tw, int L, cudaStream_t st) {
    twiddle64_kernel<<<(L + 255) / 256, 256, 0, st>>>(tw, L);
    return cudaGetLastError();
}

cudaError_t launch_template_fft(const double2 *taps, const int32_t *dest, const int32_t *offs, int32_t n, int bM,
                                int L, const double2 *tw, int fold_r0, float2 *bank, float *cmax, cudaStream_t st) {
    int log2L = 0;
    while ((1 << log2L) < L) ++log2L;
    const size_t sm = (size_t)L * sizeof(double2);
    cudaError_t e =
        cudaFuncSetAttribute(template_fft_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    template_fft_kernel<<<n, 512, sm, st>>>(taps, dest, offs, bM, L, log2L, tw, fold_r0, bank,
                                            reinterpret_cast<int *>(cmax));
    return cudaGetLastError();
}

}  // namespace jerk
