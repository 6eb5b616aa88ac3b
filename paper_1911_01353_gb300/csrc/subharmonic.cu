// Harmonic sums indexed by the highest harmonic (the sub-harmonic form).
//
// For a top harmonic at cell q of template t = (z, w):
//   S'_H(q, t) = sum_{h=1..H} P(round(h q / H), z_h, w_h),
// with (z_h, w_h) the grid point nearest to (h z / H, h w / H) and halves
// rounded away from zero.  Every template and every cell is a possible top
// harmonic, so the form needs the whole power plane; it serves banks whose
// plane fits on the device (the plane comes from jerk_plane).  Sec. 3 names
// the harmonic sum; this indexing is the one of the method's lineage (the
// fundamental-indexed sum of the main path adds the same terms where the
// rounding is exact).
//
// A block takes 32 consecutive cells: each of its eight warps walks an eighth
// of the templates for them and the partial (max, argmax) are combined in
// ascending t (lowest t on equal sums).  The H template indices of every t are
// a table in shared memory.  A plane of 77 MB is read through L2 at 4 H bytes
// per sum; with the table, 64-bit divisions no longer come before each load,
// and eight warps share a cell, so that 2^14 cells already fill the chip.  2^16
// bins, 147 templates, H = 1..4 with the plane and the peaks: 2.54 -> 0.88 ms
// (one cell per thread and FP64 sums before).
#include "jerk_internal.h"
#include "twosum.cuh"

namespace jerk {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kTable = 1024;         // templates whose harmonic indices are in shared memory at a time
constexpr int kAhead = 4;            // templates whose loads are in flight together
constexpr int kFlush = 32;           // sums between two additions to the FP64 statistics

// a h / H to the nearest integer, halves away from zero
__device__ __forceinline__ int64_t round_ratio(int64_t a, int h, int H) {
    const int64_t m = (a < 0 ? -a : a) * h;
    const int64_t q = (2 * m + H) / (2 * H);
    return a < 0 ? -q : q;
}
__device__ __forceinline__ int round_ratio32(int a, int h, int H) {
    const int q = (2 * abs(a) * h + H) / (2 * H);
    return a < 0 ? -q : q;
}

// Sums of non-negative FP32 values and of their squares as unevaluated FP32 sums, s
// the rounded one, c the sum of its exact errors: FP64 additions run at 1/64 of the
// FP32 rate here and were the longest part.  The FP64 totals keep s and the rest
// apart: sums of s are exact there (24-bit values of nearly one size).  A square is
// its rounded value and r, what that left; squares of 24-bit numbers end in binary
// 00 or 01, so wherever their last bits are rounded off, as by FP64 sums in turn,
// the total leans down.  The r of four squares are added first (three exact sums,
// the last but for a bit), then to a pair (r, d) of their own.  Relative error of
// sum S^2 at H = 2, 4, 8, 32 000 cells x 147 templates: FP64 additions in turn
// 0.9e-15, r added to c 1.6, 2.0 and 2.3e-15, this 0.1 to 0.2e-15.
struct ValueSum {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void add(float y) {
        const float hi = fmaxf(s, y), lo = fminf(s, y);      // (the larger first: three operations for the error)
        s = __fadd_rn(hi, lo);
        c = __fadd_rn(c, __fsub_rn(lo, __fsub_rn(s, hi)));
    }
    __device__ __forceinline__ void flush(double &sum, double &rest) {
        sum += (double)s;
        rest += (double)c;
        s = c = 0.f;
    }
};
struct SquareSum {
    ValueSum v;
    float r = 0.f, d = 0.f;
    __device__ __forceinline__ float add(float x) {           // returns what the square's rounding left
        const float sq = __fmul_rn(x, x);
        v.add(sq);
        return __fmaf_rn(x, x, -sq);
    }
    __device__ __forceinline__ void add_rest(float y) { d = __fadd_rn(d, two_sum(r, y)); }
    __device__ __forceinline__ void flush(double &sum, double &rest) {
        v.flush(sum, rest);
        rest += (double)r + (double)d;
        r = d = 0.f;
    }
};

struct SubArgs {
    const float *plane;          // [T][bN]
    int64_t bN;
    int32_t T, H, nz, zc, wc;    // zc = zmax / dz, wc = wmax / dw
    unsigned long long *M;       // [bN] packed max-projection
    double *part;                // [gridDim.x][2] statistics partials
};

template <int H>
__global__ void __launch_bounds__(kThreads) subharmonic_kernel(SubArgs a) {
    __shared__ int32_t row[kTable][H];
    __shared__ float smax[kWarps][32];
    __shared__ int sarg[kWarps][32];
    __shared__ double r1[kWarps], r2[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double s1 = 0.0, s2 = 0.0, e2 = 0.0;     // totals; e2: what the sums of squares left
    ValueSum p1;
    SquareSum p2;
    int k = 0;                               // sums in p1, p2
    auto flush = [&] {
        p1.flush(s1, s1);
        p2.flush(s2, e2);
        k = 0;
    };
    for (int64_t q0 = 32 * (int64_t)blockIdx.x; q0 < a.bN; q0 += 32 * (int64_t)gridDim.x) {
        const int64_t q = q0 + lane;
        const bool in = q < a.bN;
        const float *col[H];
#pragma unroll
        for (int h = 1; h <= H; ++h) col[h - 1] = a.plane + (in ? round_ratio(q, h, H) : 0);
        float best = -1.0f;
        int bt = 0;
        for (int tb = 0; tb < a.T; tb += kTable) {
            const int n = min(kTable, a.T - tb);
            if (a.T > kTable || q0 == 32 * (int64_t)blockIdx.x) {   // one table serves every cell when it holds all
                __syncthreads();
                for (int i = threadIdx.x; i < n; i += kThreads) {
                    const int t = tb + i, zi = t % a.nz - a.zc, wi = t / a.nz - a.wc;
#pragma unroll
                    for (int h = 1; h <= H; ++h)
                        row[i][h - 1] = (round_ratio32(wi, h, H) + a.wc) * a.nz + (round_ratio32(zi, h, H) + a.zc);
                }
                __syncthreads();
            }
            // this warp's part, ascending; parts and tables ascend too.  kAhead
            // templates at a time, their loads issued before the first is used
            const int i1 = (int)((int64_t)n * (warp + 1) / kWarps);
            float pb = -1.0f;
            int pt = 0;
            for (int i = (int)((int64_t)n * warp / kWarps); i < i1; i += kAhead) {
                float S[kAhead];
                const int u1 = min(kAhead, i1 - i);
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    const int e = i + min(u, u1 - 1);
                    S[u] = 0.0f;
#pragma unroll
                    for (int h = 0; h < H; ++h) S[u] += __ldg(col[h] + (int64_t)row[e][h] * a.bN);
                }
                float top = S[0], low = S[0];
                bool nan = false;
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    if (u < u1 && S[u] > pb) {
                        pb = S[u];
                        pt = tb + i + u;
                    }
                    top = fmaxf(top, S[u]);
                    low = fminf(low, S[u]);
                    nan = nan || !(S[u] == S[u]);
                }
                // S and S^2 as FP32 sums in the range where both are normal numbers, else in FP64
                if (low >= 1e-12f && top <= 1e15f && !nan) {
                    float left[kAhead];
#pragma unroll
                    for (int u = 0; u < kAhead; ++u) {
                        const float x = u < u1 && in ? S[u] : 0.f;
                        p1.add(x);
                        left[u] = p2.add(x);
                    }
                    p2.add_rest((left[0] + left[1]) + (left[2] + left[3]));
                    k += kAhead;
                } else if (in) {
                    for (int u = 0; u < u1; ++u) {
                        const double x = u == 0 ? S[0] : u == 1 ? S[1] : u == 2 ? S[2] : S[3];
                        s1 += x;
                        s2 += x * x;
                    }
                }
                if (k >= kFlush) flush();
            }
            smax[warp][lane] = pb;
            sarg[warp][lane] = pt;
            __syncthreads();
            if (warp == 0) {
#pragma unroll
                for (int w = 0; w < kWarps; ++w)
                    if (smax[w][lane] > best) {
                        best = smax[w][lane];
                        bt = sarg[w][lane];
                    }
            }
            __syncthreads();
        }
        if (warp == 0 && in)
            a.M[q] = ((unsigned long long)__float_as_uint(best) << 32) |
                     (unsigned long long)(0xFFFFFFFFu - (unsigned)bt);
    }
    flush();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        e2 += __shfl_xor_sync(0xffffffffu, e2, o);
    }
    if (lane == 0) {
        r1[warp] = s1;
        r2[warp] = s2 + e2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double x1 = 0.0, x2 = 0.0;
        for (int w = 0; w < kWarps; ++w) {
            x1 += r1[w];
            x2 += r2[w];
        }
        a.part[2 * blockIdx.x] = x1;
        a.part[2 * blockIdx.x + 1] = x2;
    }
}

// the partials in a fixed order (deterministic) into sums[0..1]
__global__ void __launch_bounds__(kThreads) sum_partials_kernel(const double *part, int n, double *sums) {
    __shared__ double r[2][kWarps];
    double x1 = 0.0, x2 = 0.0;
    for (int i = threadIdx.x; i < n; i += kThreads) {
        x1 += part[2 * i];
        x2 += part[2 * i + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x1 += __shfl_xor_sync(0xffffffffu, x1, o);
        x2 += __shfl_xor_sync(0xffffffffu, x2, o);
    }
    if ((threadIdx.x & 31) == 0) {
        r[0][threadIdx.x >> 5] = x1;
        r[1][threadIdx.x >> 5] = x2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double x = 0.0;
        for (int w = 0; w < kWarps; ++w) x += r[threadIdx.x][w];
        sums[threadIdx.x] = x;
    }
}

cudaError_t launch_subharmonic(const SubArgs &a, int nblk, cudaStream_t st) {
    switch (a.H) {
        case 1: subharmonic_kernel<1><<<nblk, kThreads, 0, st>>>(a); break;
        case 2: subharmonic_kernel<2><<<nblk, kThreads, 0, st>>>(a); break;
        case 3: subharmonic_kernel<3><<<nblk, kThreads, 0, st>>>(a); break;
        case 4: subharmonic_kernel<4><<<nblk, kThreads, 0, st>>>(a); break;
        case 5: subharmonic_kernel<5><<<nblk, kThreads, 0, st>>>(a); break;
        case 6: subharmonic_kernel<6><<<nblk, kThreads, 0, st>>>(a); break;
        case 7: subharmonic_kernel<7><<<nblk, kThreads, 0, st>>>(a); break;
        default: subharmonic_kernel<8><<<nblk, kThreads, 0, st>>>(a); break;
    }
    return cudaGetLastError();
}

}  // namespace
}  // namespace jerk

extern "C" jerk_status jerk_subharmonic(jerk_plan pl, const float *d_plane, int64_t n, int32_t H,
                                        uint64_t *d_maxproj, double *d_sums, void *stream) {
    using namespace jerk;
    if (!pl || !d_plane || !d_maxproj || !d_sums || n < 1 || n > pl->prm.max_bins) return JERK_EINVAL;
    if (H < 1 || H > JERK_MAX_HARMONIC) return JERK_EINVAL;
    if (cudaSetDevice(pl->device) != cudaSuccess) return JERK_ECUDA;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaStreamWaitEvent(st, pl->done, 0) != cudaSuccess) return JERK_ECUDA;
    SubArgs a;
    a.plane = d_plane;
    a.bN = (int64_t)pl->b * n;
    a.T = pl->T;
    a.H = H;
    a.nz = pl->nz;
    a.zc = pl->prm.zmax / pl->prm.dz;
    a.wc = pl->prm.wmax / pl->prm.dw;
    a.M = (unsigned long long *)d_maxproj;
    a.part = pl->d_stat_part;
    int64_t nblk = (a.bN + 31) / 32;
    nblk = std::min<int64_t>(nblk, (int64_t)pl->sms * 8);
    nblk = std::min<int64_t>(nblk, pl->stat_part_cap / 2);
    if (nblk < 1) return JERK_ENOMEM;
    if (launch_subharmonic(a, (int)nblk, st) != cudaSuccess) return JERK_ECUDA;
    sum_partials_kernel<<<1, kThreads, 0, st>>>(pl->d_stat_part, (int)nblk, d_sums);
    if (cudaGetLastError() != cudaSuccess) return JERK_ECUDA;
    if (cudaEventRecord(pl->done, st) != cudaSuccess) return JERK_ECUDA;
    return JERK_OK;
}
