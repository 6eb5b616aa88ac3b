// Matched-filter power at arbitrary points of the continuous (r, z, w)
// space: the response of Sec. 2 off the search grid, for refining candidates
// and for testing them against their 26 neighbours.
//
//   P(r, z, w) = |A|^2,  A = sum_k F_k conj(rho(k - r; z, w)),  |k - r| <= m(z, w),
//   rho(q; z, w) = int_{-1/2}^{1/2} exp(2 pi i (-q u + z u^2/2 + w u^3/6)) du,
//
// F the normalised spectrum (bins outside [0, N) zero), m(z, w) =
// ceil(|z|/2 + |w|/8) + P.  On the grid (r = p / b, integer z, w) this is the
// plane value P(p, z, w) the filter kernels compute.
//
// The integral is the template bank's quadrature (64-node Gauss-Legendre
// panels of at most 20 cycles; J equal panels, a class of J per range of
// half-widths), and the same periodicity makes it cheap: with k = k0 + kappa,
// delta = k0 - r and u = -1/2 + j/J + (1 + x_i)/(2J),
//   rho = (-1)^kappa e^{-pi i kappa/J} sum_i e^{-pi i kappa x_i/J} A_i(kappa),
//   A_i(kappa) = sum_j c_{j,i} e^{-2 pi i kappa j/J},
//   c_{j,i} = W_i/(2J) e^{2 pi i (z u^2/2 + w u^3/6 - delta u)},
// A_i of period J in kappa, and the nodes +-x_i combined as
// cos theta S_i - i sin theta D_i (see templates.cu), cos and sin from a table
// per class of J.  One CTA per point.  Summing every node at every bin (64 J x
// nk exponentials by recurrence) took 9 M operations per point at z = 200,
// w = 600; this takes 0.16 M: 0.06 M for the nodes' phases, 0.05 M for S and D,
// 0.05 M for the bins.  All in FP32 but the panels' phases, whose large part is
// reduced in FP64 once per panel; the product of slope and offset inside a
// panel (up to 10 cycles) is kept as an exact pair.  Bins are summed as exact
// pairs.  Where the power sits in one or two bins nothing averages the roundings
// of a bin: at J = 2 and 4 a bin's node pairs are summed in four chains and its
// products' errors kept, above in two chains.  40 candidates x 175 points (z = 200,
// w = 600 bank, 2^18 bins), host included: 2.69 -> 0.50 ms.  Relative error of a
// strong signal's power against FP64, RMS, in 1e-7:
//   (z, w)                            (0, 0)  (0, 20)  (4, 0)  (20, 60)  (50, 300)  (200, 600)
//   every node summed at every bin      1.1     2.5     2.5     1.0        0.8        0.9
//   one chain, plain products           2.1     2.4     1.4     0.9        0.9        0.7
//   this                                0.8     1.0     0.6     0.5        0.7        0.6
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "jerk_internal.h"
#include "twosum.cuh"

namespace jerk {
namespace {

constexpr int kThreads = 128;
constexpr int kPairs = 32;                 // node pairs +-x of a panel's 64 Gauss-Legendre nodes (the bank's rule)
constexpr double kCyclesPerPanel = 20.0;
constexpr int kMaxWindow = 24000;          // bins per point
constexpr int kClasses = 24;               // classes of J: 2, 4, 6, 8, 12, 16, 24, ...
constexpr int kRun = 4;                    // bins of one residue class mod J a thread sums at a time

__device__ __host__ inline int halfwidth_at(double z, double w, int pad) {
    return (int)ceil(fabs(z) / 2.0 + fabs(w) / 8.0) + pad;
}

// the class of a point and its panels: the first J that holds its cycles
__device__ __host__ inline int panel_class(double z, double w, int pad, int *J) {
    const double cyc = halfwidth_at(z, w, pad) + 1 + fabs(z) / 2.0 + fabs(w) / 8.0;
    const int need = (int)ceil(cyc / kCyclesPerPanel) + 1;
    int c = 0, j = 2;
    while (j < need) {
        j = j == 2 ? 4 : (j & (j - 1)) == 0 ? j / 2 * 3 : j / 3 * 4;
        ++c;
    }
    *J = j;
    return c;
}

// per class: its J (0: no point of it), the offset of its table (float2) and the row length (bins)
struct ClassTables {
    int64_t off[kClasses];
    int32_t J[kClasses], len[kClasses];
};

// The tables of every class in use (grid plane z: the z-th), one launch: a call for
// few points is its launches.  Rows i < 32: (cos, sin) of pi kappa x_i / J, x_i the
// positive nodes; row 32: (-1)^kappa e^{-pi i kappa / J}
__global__ void window_table_kernel(float2 *tables, ClassTables ct, const double2 *__restrict__ gl) {
    int cls = 0;
    for (int z = (int)blockIdx.z; ct.J[cls] == 0 || z-- > 0;) ++cls;
    const int J = ct.J[cls], len = ct.len[cls];
    float2 *tab = tables + ct.off[cls];
    const int k = blockIdx.x * blockDim.x + threadIdx.x, i = blockIdx.y;
    if (k >= len) return;
    double s, c;
    if (i < kPairs)
        sincospi((double)k * gl[kPairs + i].x / J, &s, &c);
    else
        sincospi((double)(((int64_t)k * (J - 1)) % (2 * J)) / J, &s, &c);
    tab[(int64_t)i * len + k] = make_float2((float)c, (float)s);
}

// add y to the unevaluated pair (s, c): s the rounded sum, c the sum of its exact errors
__device__ __forceinline__ void pair_add(float &s, float &c, float y) { c = __fadd_rn(c, two_sum(s, y)); }
// the same of the product x y, whose rounding error is exact too
__device__ __forceinline__ void pair_add_product(float &s, float &c, float x, float y) {
    const float t = __fmul_rn(x, y);
    pair_add(s, c, t);
    c = __fadd_rn(c, __fmaf_rn(x, y, -t));
}

__global__ void __launch_bounds__(kThreads) power_at_kernel(const float2 *__restrict__ F, int64_t N,
                                                            const double *__restrict__ rzw, int pad, ClassTables ct,
                                                            int smem_float2, const double2 *__restrict__ gl,
                                                            const float2 *__restrict__ tables,
                                                            float *__restrict__ out) {
    extern __shared__ __align__(16) float2 sm[];
    __shared__ float2 node[2 * kPairs];    // offset x_i / (2J) as a pair (hi, lo)
    __shared__ float weight[kPairs];       // W_i / (2J)
    __shared__ double red[2][kThreads / 32];
    const double r = rzw[3 * blockIdx.x], z = rzw[3 * blockIdx.x + 1], w = rzw[3 * blockIdx.x + 2];
    const int m = halfwidth_at(z, w, pad);
    const int64_t k0 = max((int64_t)0, (int64_t)ceil(r - m));
    const int64_t k1 = min(N - 1, (int64_t)floor(r + m));
    const int nk = k1 >= k0 ? (int)(k1 - k0 + 1) : 0;
    int J;
    const int cls = panel_class(z, w, pad, &J);
    const float2 *tab = tables + ct.off[cls];
    const int len = ct.len[cls];
    const int hJ = J / 2;
    // shared: roots e^{-2 pi i k / J} [J] | panel phases float4 [J] | nodes' chirps [2 ib][J] | S [ib][J] | D [ib][J]
    float2 *root = sm;
    float4 *panel = reinterpret_cast<float4 *>(sm + J);          // (J is even)
    float2 *chirp = sm + 3 * J;
    int ib = kPairs;
    while (ib > 2 && 3 * J + 4 * ib * J > smem_float2) ib >>= 1;     // (two chains below: at least two)
    float2 *S = chirp + 2 * ib * J, *D = S + ib * J;
    const float w6 = (float)(w / 6.0);
    for (int k = threadIdx.x; k < J; k += kThreads) {
        float s, c;
        sincospif(-2.0f * (float)k / (float)J, &s, &c);
        root[k] = make_float2(c, s);
        // phase (cycles) at the panel's centre a and its derivatives there
        const double a = -0.5 + (k + 0.5) / J, dl = (double)k0 - r;
        double p0 = a * (a * (z / 2.0 + w * a / 6.0) - dl);
        p0 -= rint(p0);
        const double p1 = a * (z + w * a / 2.0) - dl;
        const float h1 = (float)p1;
        panel[k] = make_float4((float)p0, h1, (float)(p1 - (double)h1), (float)((z + w * a) / 2.0));
    }
    for (int i = threadIdx.x; i < 2 * kPairs; i += kThreads) {
        const double2 g = gl[i];
        const double x = g.x * 0.5 / J;
        const float xh = (float)x;
        node[i] = make_float2(xh, (float)(x - (double)xh));
        if (i >= kPairs) weight[i - kPairs] = (float)(g.y * 0.5 / J);
    }
    float ar = 0.f, er = 0.f, ai = 0.f, ei = 0.f;
    for (int q0 = 0; q0 < kPairs; q0 += ib) {
        __syncthreads();
        for (int n = threadIdx.x; n < 2 * ib * J; n += kThreads) {
            const int row = n / J, j = n - row * J, q = q0 + (row >> 1);
            const float2 x = node[(row & 1) ? kPairs - 1 - q : kPairs + q];
            const float4 p = panel[j];
            // slope x offset as an exact pair, its whole cycles dropped
            const float t = p.y * x.x;
            float lo = fmaf(p.y, x.x, -t);
            lo = fmaf(p.y, x.y, lo);
            lo = fmaf(p.z, x.x, lo);
            lo = fmaf(x.x * x.x, fmaf(w6, x.x, p.w), lo);
            float ph = (t - rintf(t)) + (p.x + lo);
            ph -= rintf(ph);
            float s, c;
            sincospif(2.0f * ph, &s, &c);
            const float wt = weight[q];
            chirp[n] = make_float2(wt * c, wt * s);
        }
        __syncthreads();
        // A(e) and A(e + J/2) = (even j) +- (odd j), for both nodes of a pair
        for (int n = threadIdx.x; n < ib * hJ; n += kThreads) {
            const int p = n / hJ, e = n - p * hJ;
            const float2 *cp = chirp + 2 * p * J, *cm = cp + J;
            float pr[2] = {0.f, 0.f}, pi[2] = {0.f, 0.f}, mr[2] = {0.f, 0.f}, mi[2] = {0.f, 0.f};
            int k = 0;                     // e j mod J
            for (int j = 0; j < J; j += 2) {
#pragma unroll
                for (int o = 0; o < 2; ++o) {
                    const float2 t = root[k], x = cp[j + o], y = cm[j + o];
                    pr[o] = fmaf(x.x, t.x, fmaf(-x.y, t.y, pr[o]));
                    pi[o] = fmaf(x.x, t.y, fmaf(x.y, t.x, pi[o]));
                    mr[o] = fmaf(y.x, t.x, fmaf(-y.y, t.y, mr[o]));
                    mi[o] = fmaf(y.x, t.y, fmaf(y.y, t.x, mi[o]));
                    k += e;
                    if (k >= J) k -= J;
                }
            }
#pragma unroll
            for (int o = 0; o < 2; ++o) {
                const float f = o ? -1.f : 1.f;
                const float xr = fmaf(f, pr[1], pr[0]), xi = fmaf(f, pi[1], pi[0]);
                const float yr = fmaf(f, mr[1], mr[0]), yi = fmaf(f, mi[1], mi[0]);
                S[p * J + e + o * hJ] = make_float2(xr + yr, xi + yi);
                D[p * J + e + o * hJ] = make_float2(xr - yr, xi - yi);
            }
        }
        __syncthreads();
        // bins of one residue e mod J share S and D: kRun of them per thread and step
        const int runs = (nk + kRun * J - 1) / (kRun * J);
        auto bins = [&](auto chains) {                           // chains divide ib, a power of two
            constexpr int CH = decltype(chains)::value;
            for (int n = threadIdx.x; n < runs * J; n += kThreads) {
                const int b = n / J, e = n - b * J;
                const int kap = e + b * kRun * J;
                float cr[kRun][CH], ci[kRun][CH];
                int at[kRun];
#pragma unroll
                for (int v = 0; v < kRun; ++v) {
#pragma unroll
                    for (int u = 0; u < CH; ++u) cr[v][u] = ci[v][u] = 0.f;
                    at[v] = min(kap + v * J, nk - 1);
                }
                for (int p0 = 0; p0 < ib; p0 += CH) {
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        const float2 s = S[(p0 + u) * J + e], d = D[(p0 + u) * J + e];
                        const float2 *row = tab + (int64_t)(q0 + p0 + u) * len;
#pragma unroll
                        for (int v = 0; v < kRun; ++v) {
                            const float2 cs = __ldg(row + at[v]);
                            cr[v][u] = fmaf(cs.x, s.x, fmaf(cs.y, d.y, cr[v][u]));
                            ci[v][u] = fmaf(cs.x, s.y, fmaf(-cs.y, d.x, ci[v][u]));
                        }
                    }
                }
#pragma unroll
                for (int v = 0; v < kRun; ++v) {
                    if (kap + v * J >= nk) continue;
                    const float2 ph = __ldg(tab + (int64_t)kPairs * len + at[v]);
                    const float2 f = F[k0 + at[v]];
                    float rr = cr[v][0], ri = ci[v][0];
                    if constexpr (CH == 2) rr += cr[v][1], ri += ci[v][1];
                    if constexpr (CH == 4) {
                        rr = (cr[v][0] + cr[v][1]) + (cr[v][2] + cr[v][3]);
                        ri = (ci[v][0] + ci[v][1]) + (ci[v][2] + ci[v][3]);
                    }
                    const float xr = fmaf(rr, ph.x, -ri * ph.y), xi = fmaf(rr, ph.y, ri * ph.x);
                    if constexpr (CH == 4) {                         // F conj(rho)
                        pair_add_product(ar, er, f.x, xr);
                        pair_add_product(ar, er, f.y, xi);
                        pair_add_product(ai, ei, f.y, xr);
                        pair_add_product(ai, ei, -f.x, xi);
                    } else {
                        pair_add(ar, er, fmaf(f.x, xr, f.y * xi));
                        pair_add(ai, ei, fmaf(f.y, xr, -f.x * xi));
                    }
                }
            }
        };
        // (classes of J = 2 and 4: the power sits in one or two bins)
        if (J <= 4)
            bins(std::integral_constant<int, 4>{});
        else
            bins(std::integral_constant<int, 2>{});
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float yr = __shfl_xor_sync(0xffffffffu, ar, o), cr = __shfl_xor_sync(0xffffffffu, er, o);
        const float yi = __shfl_xor_sync(0xffffffffu, ai, o), ci = __shfl_xor_sync(0xffffffffu, ei, o);
        pair_add(ar, er, yr);
        pair_add(ai, ei, yi);
        er += cr;
        ei += ci;
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = (double)ar + (double)er;
        red[1][threadIdx.x >> 5] = (double)ai + (double)ei;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sr = 0.0, si = 0.0;
        for (int i = 0; i < kThreads / 32; ++i) {
            sr += red[0][i];
            si += red[1][i];
        }
        out[blockIdx.x] = (float)(sr * sr + si * si);
    }
}

}  // namespace
}  // namespace jerk

using namespace jerk;

namespace {

jerk_status from_cuda_r(cudaError_t e) {
    if (e == cudaSuccess) return JERK_OK;
    if (e == cudaErrorMemoryAllocation) return JERK_ENOMEM;
    return JERK_ECUDA;
}

#define RCHECK(x)                                      \
    do {                                               \
        cudaError_t e_ = (x);                          \
        if (e_ != cudaSuccess) return from_cuda_r(e_); \
    } while (0)

// normalise d_spec into the plan's workspace (after the plan's previous work)
jerk_status stage_spectrum(jerk_plan pl, const void *d_spec, int64_t n, cudaStream_t st, const float2 **out) {
    RCHECK(cudaStreamWaitEvent(st, pl->done, 0));
    if (pl->prm.norm_block > 0) {
        RCHECK(launch_normalise((const float2 *)d_spec, pl->d_spec_norm, n, pl->prm.norm_block, st));
        *out = pl->d_spec_norm;
    } else {
        *out = (const float2 *)d_spec;
    }
    return JERK_OK;
}

jerk_status power_at_host(jerk_plan pl, const float2 *F, int64_t n, const std::vector<double> &pts, float *h_out,
                          cudaStream_t st) {
    const int64_t count = (int64_t)pts.size() / 3;
    if (count == 0) return JERK_OK;
    ClassTables ct;
    for (int c = 0; c < kClasses; ++c) ct.off[c] = ct.J[c] = ct.len[c] = 0;
    for (int64_t i = 0; i < count; ++i) {
        const double z = pts[3 * i + 1], w = pts[3 * i + 2];
        if (!std::isfinite(pts[3 * i]) || !std::isfinite(z) || !std::isfinite(w)) return JERK_EINVAL;
        if (std::fabs(z) > 8192.0 || std::fabs(w) > 65536.0) return JERK_EINVAL;
        const int win = 2 * halfwidth_at(z, w, pl->prm.pad_bins) + 2;
        if (win > kMaxWindow) return JERK_EINVAL;
        int J;
        const int c = panel_class(z, w, pl->prm.pad_bins, &J);
        if (c >= kClasses) return JERK_EINVAL;
        ct.J[c] = J;
        ct.len[c] = std::max(ct.len[c], win);
    }
    int64_t tab = 0;
    int jmax = 2, classes = 0, longest = 0;
    for (int c = 0; c < kClasses; ++c) {
        if (!ct.J[c]) continue;
        ct.off[c] = tab;
        tab += (int64_t)(kPairs + 1) * ct.len[c];
        jmax = std::max(jmax, ct.J[c]);
        longest = std::max(longest, ct.len[c]);
        ++classes;
    }
    // shared memory: all node pairs at once up to 96 KB (J = 64), then fewer at a time, two
    // at least (J = 1536, the most: 132 KB)
    const int all = (3 + 4 * kPairs) * jmax, cap = (96 << 10) / (int)sizeof(float2);
    const int smem_float2 = std::max(std::min(all, cap), 11 * jmax);
    const size_t smem = (size_t)smem_float2 * sizeof(float2);
    // one buffer: points | tables | powers
    const size_t b_pts = (sizeof(double) * pts.size() + 255) & ~(size_t)255;
    const size_t b_tab = (sizeof(float2) * (size_t)tab + 255) & ~(size_t)255;
    char *buf = nullptr;
    RCHECK(cudaMallocAsync((void **)&buf, b_pts + b_tab + sizeof(float) * count, st));
    double *d_pts = (double *)buf;
    float2 *d_tab = (float2 *)(buf + b_pts);
    float *d_out = (float *)(buf + b_pts + b_tab);
    cudaError_t e = cudaMemcpyAsync(d_pts, pts.data(), sizeof(double) * pts.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        const dim3 grid((unsigned)((longest + 127) / 128), kPairs + 1, (unsigned)classes);
        window_table_kernel<<<grid, 128, 0, st>>>(d_tab, ct, pl->d_gl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(power_at_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    for (int64_t b0 = 0; b0 < count && e == cudaSuccess; b0 += 1 << 30) {
        const unsigned nb = (unsigned)std::min<int64_t>(1 << 30, count - b0);
        power_at_kernel<<<nb, kThreads, smem, st>>>(F, n, d_pts + 3 * b0, pl->prm.pad_bins, ct, smem_float2, pl->d_gl,
                                                    d_tab, d_out + b0);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_out, d_out, sizeof(float) * count, cudaMemcpyDeviceToHost, st);
    cudaFreeAsync(buf, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = cudaEventRecord(pl->done, st);
    return from_cuda_r(e);
}

}  // namespace

extern "C" {

jerk_status jerk_power_at(jerk_plan pl, const void *d_spec, int64_t n, const double *h_rzw, int64_t count,
                          float *h_power, void *stream) {
    if (!pl || !d_spec || n < 1 || n > pl->prm.max_bins || count < 0 || (count > 0 && (!h_rzw || !h_power)))
        return JERK_EINVAL;
    if (!pl->share) return JERK_ESTATE;
    RCHECK(cudaSetDevice(pl->device));
    cudaStream_t st = (cudaStream_t)stream;
    const float2 *F = nullptr;
    jerk_status s = stage_spectrum(pl, d_spec, n, st, &F);
    if (s != JERK_OK) return s;
    std::vector<double> pts(h_rzw, h_rzw + 3 * count);
    return power_at_host(pl, F, n, pts, h_power, st);
}

jerk_status jerk_refine(jerk_plan pl, const void *d_spec, int64_t n, const jerk_candidate *h_cands, int32_t count,
                        const double *h_step, const int32_t *h_half, jerk_refined *h_out, void *stream) {
    if (!pl || !d_spec || n < 1 || n > pl->prm.max_bins || count < 0 || !h_step || !h_half) return JERK_EINVAL;
    if (count > 0 && (!h_cands || !h_out)) return JERK_EINVAL;
    for (int i = 0; i < 3; ++i)
        if (h_half[i] < 0 || h_half[i] > 64 || !std::isfinite(h_step[i]) || h_step[i] < 0.0) return JERK_EINVAL;
    if (!pl->share) return JERK_ESTATE;
    RCHECK(cudaSetDevice(pl->device));
    cudaStream_t st = (cudaStream_t)stream;
    const int nr = 2 * h_half[0] + 1, nzf = 2 * h_half[1] + 1, nwf = 2 * h_half[2] + 1;
    const int64_t G = (int64_t)nr * nzf * nwf;
    if ((int64_t)count * G > ((int64_t)1 << 26)) return JERK_EINVAL;
    std::vector<double> pts((size_t)(3 * count * G));
    for (int c = 0; c < count; ++c) {
        int64_t g = 0;
        for (int i = -h_half[0]; i <= h_half[0]; ++i)
            for (int j = -h_half[1]; j <= h_half[1]; ++j)
                for (int l = -h_half[2]; l <= h_half[2]; ++l, ++g) {
                    double *p = &pts[3 * ((size_t)c * G + g)];
                    p[0] = h_cands[c].r + i * h_step[0];
                    p[1] = (double)h_cands[c].z + j * h_step[1];
                    p[2] = (double)h_cands[c].w + l * h_step[2];
                }
    }
    const float2 *F = nullptr;
    jerk_status s = stage_spectrum(pl, d_spec, n, st, &F);
    if (s != JERK_OK) return s;
    std::vector<float> P((size_t)(count * G));
    s = power_at_host(pl, F, n, pts, P.data(), st);
    if (s != JERK_OK) return s;
    const int64_t centre = (G - 1) / 2;    // (i, j, l) = (0, 0, 0)
    for (int c = 0; c < count; ++c) {
        const float *pc = P.data() + (size_t)c * G;
        int64_t best = 0;
        for (int64_t g = 1; g < G; ++g)
            if (pc[g] > pc[best]) best = g;
        const double *p = &pts[3 * ((size_t)c * G + best)];
        jerk_refined &o = h_out[c];
        o.r = p[0];
        o.z = (float)p[1];
        o.w = (float)p[2];
        o.power = pc[best];
        o.power_in = pc[centre];
        o.is_peak = pc[centre] >= pc[best] ? 1 : 0;
        o.reserved = 0;
    }
    return JERK_OK;
}

}  // extern "C"
