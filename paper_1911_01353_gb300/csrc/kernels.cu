// Normalisation, harmonic sum, statistics and peak finding.
#include <cfloat>

#include "device_sync.cuh"
#include "jerk_internal.h"

namespace jerk {

// ---------------------------------------------------------------------------
// Power normalisation (the paper is silent; reading): for each block of B
// bins, med = element of rank floor((n-1)/2) of |F_k|^2 (FP64, exact for
// FP32 input), F_k <- F_k (med / ln 2)^(-1/2).
//
// Each block's powers are formed in FP32 (at most 2^-22 off, relatively) and
// kept in registers; bisecting their bit patterns by counting (one compare per
// bin and step, one warp reduction) closes in on the FP32 median v.  The FP64
// median then lies within a few units in the last place of v: the FP64 powers
// of the bins that close decide, one or two bins as a rule.  Bins are scaled by
// the FP64 factor as a pair of floats, with the FP64 product where the pair
// cannot decide the rounding, so that the result is the FP64 one bit for bit.
// FP64 instructions run at 1/64 of the FP32 rate, and sorting all FP64 powers
// (55 barriers), then keying and scaling all bins in FP64, were the longest
// parts: 2^16 bins 24 -> 10 us, 2^21 bins 170 -> 39 us, a batch of 24 spectra of
// 2^13-2^16 bins 555 -> 34 us.  Blocks that are too small or too large for FP32
// powers take the FP64 powers rounded to FP32, which keep the order.  One warp
// per block of up to 1024 bins (four above, or where there are few blocks);
// one launch normalises up to kNormItems spectra.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long power_key(float2 f) {
    const double re = f.x, im = f.y;
    return (unsigned long long)__double_as_longlong(re * re + im * im);   // non-negative: integer order = value order
}

// (float)((double)f * scale), scale = sh + sl to 2^-48 from 2^-100 up (below, sl
// and then sh are subnormal and keep fewer bits).  The product as a pair p + e
// is good to 2^-46 of it; it decides the rounding unless what is left after
// rounding lies within 2^-18 of half a unit in the last place, the result is a
// power of two (the unit changes there) or out of the normal range.
__device__ __forceinline__ float scaled(float f, double scale, float sh, float sl) {
    const float p = __fmul_rn(f, sh);
    const float e = __fmaf_rn(f, sl, __fmaf_rn(f, sh, -p));
    const float r = __fadd_rn(p, e);
    const float left = fabsf(__fadd_rn(__fsub_rn(p, r), e));
    const unsigned bits = __float_as_uint(r);
    const float half = __uint_as_float(bits & 0x7f800000u) * 5.9604644775390625e-8f;   // 2^-24 of r's power of two
    const float a = fabsf(r);
    if (fabsf(left - half) > half * 3.8e-6f && (bits & 0x007fffffu) != 0u && a >= 1e-28f && a <= 1e28f &&
        sh >= 0x1p-100f)
        return r;
    return (float)((double)f * scale);
}

// sums and extrema over the W warps of a block of bins
template <int W>
struct BlockOf {
    static __device__ __forceinline__ void sync() {
        if constexpr (W > 1) __syncthreads(); else __syncwarp();
    }
    static __device__ __forceinline__ unsigned add(unsigned x) {
        x = __reduce_add_sync(0xffffffffu, x);
        if constexpr (W > 1) x = across(x, [](unsigned a, unsigned b) { return a + b; });
        return x;
    }
    static __device__ __forceinline__ unsigned low(unsigned x) {
        x = __reduce_min_sync(0xffffffffu, x);
        if constexpr (W > 1) x = across(x, [](unsigned a, unsigned b) { return a < b ? a : b; });
        return x;
    }
    static __device__ __forceinline__ unsigned high(unsigned x) {
        x = __reduce_max_sync(0xffffffffu, x);
        if constexpr (W > 1) x = across(x, [](unsigned a, unsigned b) { return a > b ? a : b; });
        return x;
    }
    template <class Op>
    static __device__ __forceinline__ unsigned across(unsigned x, Op op) {
        __shared__ unsigned part[W];
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = x;
        __syncthreads();
        unsigned r = part[0];
#pragma unroll
        for (int w = 1; w < W; ++w) r = op(r, part[w]);
        __syncthreads();
        return r;
    }
    // a 64-bit minimum or maximum, high word first
    static __device__ __forceinline__ unsigned long long low64(unsigned long long x) {
        const unsigned h = low((unsigned)(x >> 32));
        const unsigned l = low((unsigned)(x >> 32) == h ? (unsigned)x : ~0u);
        return ((unsigned long long)h << 32) | l;
    }
    static __device__ __forceinline__ unsigned long long high64(unsigned long long x) { return ~low64(~x); }
};

// KPT bins per thread, W warps per block of at most 32 W KPT bins
template <int KPT, int W>
__global__ void __launch_bounds__(32 * W) normalise_kernel(NormArgs a, int B) {
    constexpr int NT = 32 * W;
    int item = 0;
    while (item + 1 < a.count && (int)blockIdx.x >= a.blk0[item + 1]) ++item;
    const int64_t s0 = (int64_t)((int)blockIdx.x - a.blk0[item]) * B, n = a.n[item];
    const int nb = (int)((n - s0) < B ? (n - s0) : B);
    const float2 *in = a.in[item] + s0;
    float2 *out = a.out[item] + s0;
    const int tid = threadIdx.x;
    unsigned key[KPT];
    const unsigned rank = (unsigned)(nb - 1) / 2;
    unsigned lo, hi, n_lo;
    // pass 0: FP32 powers; pass 1, where those are too small or too large: FP64
    // powers rounded to FP32, which keeps their order
    for (int pass = 0;; ++pass) {
        lo = ~0u;
        hi = 0u;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            const int k = tid + NT * i;
            key[i] = ~0u;                                     // above every power: never counted
            if (k < nb) {
                const float2 f = in[k];
                key[i] = __float_as_uint(fmaf(f.x, f.x, f.y * f.y));
                if (pass) key[i] = __float_as_uint((float)__longlong_as_double((long long)power_key(f)));
                lo = min(lo, key[i]);
                hi = max(hi, key[i]);
            }
        }
        lo = BlockOf<W>::low(lo);
        hi = BlockOf<W>::high(hi);
        // the key of that rank is one of the n_hi - n_lo in [lo, hi]
        unsigned n_hi = (unsigned)nb;
        n_lo = 0;
        while (lo < hi && n_hi - n_lo > 1) {
            const unsigned mid = lo + (hi - lo) / 2;
            unsigned c0 = 0, c1 = 0, c2 = 0, c3 = 0;          // four counts: short chains
#pragma unroll
            for (int i = 0; i < KPT; i += 4) {
                c0 += key[i] <= mid ? 1u : 0u;
                c1 += key[i + 1] <= mid ? 1u : 0u;
                c2 += key[i + 2] <= mid ? 1u : 0u;
                c3 += key[i + 3] <= mid ? 1u : 0u;
            }
            const unsigned c = BlockOf<W>::add((c0 + c1) + (c2 + c3));
            if (c > rank) {
                hi = mid;
                n_hi = c;
            } else {
                lo = mid + 1;
                n_lo = c;
            }
        }
        if (pass) break;
        // the one key of that rank: the smallest in [lo, hi]
        unsigned v = ~0u;
#pragma unroll
        for (int i = 0; i < KPT; ++i)
            if (key[i] >= lo && key[i] <= hi) v = min(v, key[i]);
        v = BlockOf<W>::low(v);
        const float fv = __uint_as_float(v);
        if (fv >= 1e-30f && fv <= 1e30f) {
            // |FP32 power - FP64 power| <= 2^-22 of it, so is the median's distance from v: a bin
            // 8 units in the last place (2^-21 or more of v) below v is below the median
            lo = v - 8;
            hi = v + 8;
            unsigned c = 0;
#pragma unroll
            for (int i = 0; i < KPT; ++i) c += key[i] < lo ? 1u : 0u;
            n_lo = BlockOf<W>::add(c);
            break;
        }
    }
    // among the bins in [lo, hi], listed, by their FP64 powers: the one with at
    // most rank - n_lo others below it and more than that not above it
    constexpr int LIST = 64;
    __shared__ unsigned long long list[LIST], med64;
    __shared__ int listed;
    if (tid == 0) listed = 0;
    BlockOf<W>::sync();
#pragma unroll
    for (int i = 0; i < KPT; ++i)
        if (key[i] >= lo && key[i] <= hi) {
            const int at = atomicAdd(&listed, 1);
            if (at < LIST) list[at] = power_key(in[tid + NT * i]);
        }
    BlockOf<W>::sync();
    const int n_list = listed;
    unsigned long long lo64;
    if (n_list <= LIST) {
        for (int i = tid; i < n_list; i += NT) {
            unsigned below = 0, equal = 0;
            for (int q = 0; q < n_list; ++q) {
                below += list[q] < list[i] ? 1u : 0u;
                equal += list[q] == list[i] ? 1u : 0u;
            }
            if (below <= rank - n_lo && rank - n_lo < below + equal) med64 = list[i];
        }
        BlockOf<W>::sync();
        lo64 = med64;
    } else {
        // many equal FP32 powers: bisect the FP64 ones
        unsigned long long hi64 = 0ull;
        lo64 = ~0ull;
#pragma unroll
        for (int i = 0; i < KPT; ++i) {
            if (key[i] >= lo && key[i] <= hi) {
                const unsigned long long v = power_key(in[tid + NT * i]);
                lo64 = v < lo64 ? v : lo64;
                hi64 = v > hi64 ? v : hi64;
            }
        }
        lo64 = BlockOf<W>::low64(lo64);
        hi64 = BlockOf<W>::high64(hi64);
        while (lo64 < hi64) {
            const unsigned long long mid = lo64 + (hi64 - lo64) / 2;
            unsigned c = 0;
#pragma unroll
            for (int i = 0; i < KPT; ++i)
                if (key[i] >= lo && key[i] <= hi) c += power_key(in[tid + NT * i]) <= mid ? 1u : 0u;
            c = BlockOf<W>::add(c);
            if (c > rank - n_lo)
                hi64 = mid;
            else
                lo64 = mid + 1;
        }
    }
    const double med = __longlong_as_double((long long)lo64);
    const double scale = med > 0.0 ? 1.0 / sqrt(med / 0.69314718055994530942) : 1.0;
    const float sh = (float)scale, sl = (float)(scale - (double)sh);
#pragma unroll
    for (int i = 0; i < KPT; ++i) {
        const int k = tid + NT * i;
        if (k < nb) {
            const float2 f = in[k];
            out[k] = make_float2(scaled(f.x, scale, sh, sl), scaled(f.y, scale, sh, sl));
        }
    }
}

cudaError_t launch_normalise(const float2 *const *in, float2 *const *out, const int64_t *n, int count, int B,
                             cudaStream_t st) {
    const int64_t sms = current_device_sms();
    for (int i0 = 0; i0 < count; i0 += kNormItems) {
        NormArgs a;
        a.count = count - i0 < kNormItems ? count - i0 : kNormItems;
        int64_t blk = 0;
        for (int i = 0; i < a.count; ++i) {
            a.in[i] = in[i0 + i];
            a.out[i] = out[i0 + i];
            a.n[i] = n[i0 + i];
            a.blk0[i] = (int32_t)blk;
            blk += (n[i0 + i] + B - 1) / B;
        }
        if (blk > INT32_MAX) return cudaErrorInvalidValue;
        if (B <= 256)
            normalise_kernel<8, 1><<<(unsigned)blk, 32, 0, st>>>(a, B);
        else if (B <= 1024 && blk <= sms)
            normalise_kernel<8, 4><<<(unsigned)blk, 128, 0, st>>>(a, B);
        else if (B <= 1024)
            normalise_kernel<32, 1><<<(unsigned)blk, 32, 0, st>>>(a, B);
        else
            normalise_kernel<32, 4><<<(unsigned)blk, 128, 0, st>>>(a, B);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_normalise(const float2 *in, float2 *out, int64_t n, int B, cudaStream_t st) {
    return launch_normalise(&in, &out, &n, 1, B, st);
}

// ---------------------------------------------------------------------------
// Harmonic sum (Sec. 3 names it; S_H(p, z, w) = sum_{h=1..H} P(h p, h z, h w)
// is the reading) and the stage-H max-projection over (z, w).  The harmonic
// rows P(h p, h z, h w) were written by the fused kernel into per-(h,
// fundamental) slots indexed by p (128-byte aligned).  A block covers
// HC_CELLS consecutive fundamental cells: HC_THREADS consumer threads own
// HC_PT cells each, and one producer warp streams the block's chunk of every
// row it needs (fundamentals in ascending t, h ascending) from HBM into a
// ring of HR shared-memory slots with bulk copies (cp.async.bulk +
// mbarrier), so HR x 8 KB are in flight per block whatever the consumers
// do.  The producer stages 32 table entries at a time in shared memory and
// one lane issues the copies, writing each slot's (t, top stage) beside it.
// Consumers sum their cells of each row in fixed h order (FP32), keep
// (max, argmax) per stage (lowest t on ties) and the statistics partials,
// and release each slot per warp.  One launch serves every spectrum of a
// batch (24 spectra of 2^13-2^16 bins: 727 -> 68 us); a spectrum's fundamentals
// are split over several blocks (harm_ny, chosen where the plan lays out its
// launches) that meet in an atomic maximum (2^16 bins, 33 fundamentals: 31 -> 14 us).  Every wait is bounded (about one
// second); on expiry the block sets the error flag and leaves after its
// copies in flight have landed.
// ---------------------------------------------------------------------------
constexpr int HC_THREADS = 256;                 // consumer threads
constexpr int HC_PT = 8;                        // cells per consumer thread (two float4)
constexpr int HC_CELLS = HC_PT * HC_THREADS;    // fundamental cells per block
constexpr int HR = 11;                          // ring slots, one row chunk (HC_CELLS floats) each:
                                                // two blocks (ring + statics) fit an SM's shared memory

struct HarmEntry {                              // a table entry as the producer stages it
    int64_t off[JERK_MAX_HARMONIC];
    int t, st;
};

template <int NS>
__global__ void __launch_bounds__(HC_THREADS + 32, 2) harmonic_kernel(const __grid_constant__ HarmArgs a, bool stats) {
    extern __shared__ __align__(128) float4 ring[];   // [HR][HC_CELLS / 4]
    __shared__ __align__(8) uint64_t full[HR];        // row chunk landed
    __shared__ __align__(8) uint64_t empty[HR];       // every consumer warp done with the slot
    __shared__ int2 meta[HR];                         // (t, top stage) of the slot's fundamental
    __shared__ HarmEntry tab[32];                     // the producer's current table entries
    __shared__ double red[JERK_MAX_STAGES][2][HC_THREADS / 32];
    __shared__ double dacc[NS - 1][2][HC_THREADS];    // per-thread FP64 statistics of stages 1.. (kept out of registers)
    constexpr int Q = HC_CELLS / 4;                   // float4 per slot
    const int tid = threadIdx.x;
    // the item of this block, and its cells and fundamentals
    int lo = 0, hi = a.n_items - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((int64_t)blockIdx.x >= __ldg(&a.items[mid].harm0)) lo = mid; else hi = mid - 1;
    }
    const ItemDesc *itm = a.items + lo;
    const int local = (int)((int64_t)blockIdx.x - __ldg(&itm->harm0));
    const int nx = __ldg(&itm->harm_nx), ny = __ldg(&itm->harm_ny);
    const int64_t c0 = (int64_t)(local % nx) * HC_CELLS;
    __shared__ int64_t n_cells[NS];
    if (tid < NS) n_cells[tid] = __ldg(&itm->n_cells[tid]);
    __syncthreads();
    int topb = 0;   // highest stage index with cells in this block
#pragma unroll
    for (int si = 1; si < NS; ++si)
        if (c0 < n_cells[si]) topb = si;
    int hlo[NS], hhi[NS];
#pragma unroll
    for (int si = 1; si < NS; ++si) {
        hlo[si] = si == 1 ? 1 : a.stages[si - 1] + 1;
        hhi[si] = a.stages[si];
    }
    if (tid < HR) {
        mbar_init(&full[tid], 1);
        mbar_init(&empty[tid], HC_THREADS / 32);
    }
    __syncthreads();
    const int n_fund = __ldg(&itm->n_fund);
    const int part = local / nx;
    const int f0 = (int)((int64_t)n_fund * part / ny), f1 = (int)((int64_t)n_fund * (part + 1) / ny);
    const FundEntry *fund = reinterpret_cast<const FundEntry *>(
        __ldg(reinterpret_cast<const unsigned long long *>(&itm->fund)));

    if (tid >= HC_THREADS) {
        // ---- producer warp ----
        const int plane = tid - HC_THREADS;
        uint32_t bytes[NS];   // chunk bytes of a stage-si row: rows hold n_cells[si] cells, padded to 32
#pragma unroll
        for (int si = 1; si < NS; ++si) {
            const int64_t avail = ((n_cells[si] + 3) & ~(int64_t)3) - c0;
            bytes[si] = (uint32_t)(4 * (avail < HC_CELLS ? (avail > 0 ? avail : 0) : HC_CELLS));
        }
        int slot = 0, round = 0, issued = 0;
        bool good = topb > 0;
        for (int fb = f0; fb < f1 && good; fb += 32) {
            const int f = fb + plane;
            if (f < f1) {
                const FundEntry *fe = fund + f;
                const int st = min(__ldg(&fe->top_stage), topb);
                const int H = a.stages[st];
                tab[plane].t = __ldg(&fe->t);
                tab[plane].st = st;
#pragma unroll
                for (int h = 0; h < JERK_MAX_HARMONIC; ++h)
                    if (h < H) tab[plane].off[h] = __ldg(&fe->off[h]);
            }
            __syncwarp();
            if (plane == 0) {
                const int nb = min(32, f1 - fb);
                for (int k = 0; k < nb && good; ++k) {
                    const int t = tab[k].t, st = tab[k].st;
#pragma unroll
                    for (int si = 1; si < NS; ++si) {
                        if (si <= st) {
                            for (int h = hlo[si]; h <= hhi[si] && good; ++h) {
                                if (round > 0 && !mbar_wait_bounded(&empty[slot], (uint32_t)(round - 1) & 1u)) {
                                    good = false;
                                    break;
                                }
                                meta[slot] = make_int2(t, st);
                                const int64_t src = tab[k].off[h - 1] + c0;
                                // a skipped copy would leave the consumers waiting: give up
                                // (bounded) like an expired wait
                                if (!JERK_CHECK(src >= 0 && src + bytes[si] / 4 <= a.slot_cap, a.chk, kChkHarmCopy)) {
                                    good = false;
                                    break;
                                }
                                bulk_load(ring + slot * Q, a.slots + src, bytes[si], &full[slot]);
                                ++issued;
                                if (++slot == HR) {
                                    slot = 0;
                                    ++round;
                                }
                            }
                        }
                    }
                }
            }
            good = __shfl_sync(0xffffffffu, good, 0);
            __syncwarp();   // lane 0 done reading `tab`
        }
        if (plane == 0) {
            if (topb > 0 && !good) atomicExch(a.err, 1);
            // never leave with a copy still writing into this block's shared memory:
            // the last phase of each slot in use
            const int last = issued < HR ? issued : HR;
            for (int k = 0; k < last; ++k) {
                const int i = issued - 1 - k;
                mbar_wait_bounded(&full[i % HR], (uint32_t)(i / HR) & 1u);
            }
        }
    } else {
        // ---- consumers: thread tid owns cells p0 + 4u + c, u = 0..HC_PT/4-1 ----
        constexpr int U = HC_PT / 4;
        const int lane = tid & 31;
        const int64_t p0 = c0 + 4 * tid;
        float mx[NS][HC_PT];
        int am[NS][HC_PT];
        float c1[NS], c2[NS];
#pragma unroll
        for (int si = 0; si < NS; ++si) {
#pragma unroll
            for (int c = 0; c < HC_PT; ++c) {
                mx[si][c] = -1.0f;
                am[si][c] = 0;
            }
            if (si > 0) dacc[si - 1][0][tid] = dacc[si - 1][1][tid] = 0.0;
            c1[si] = c2[si] = 0.f;
        }
        // cell of (u, c): p0 + 4 HC_THREADS u + c
        auto cell_ok = [&](int si, int k) { return p0 + 4 * HC_THREADS * (k >> 2) + (k & 3) < n_cells[si]; };
        if (topb > 0) {
            int slot = 0, cnt = 0;
            uint32_t phase = 0;
            bool good = true;
            // every table entry has a top stage >= 1, so every fundamental has rows
            for (int f = f0; f < f1 && good; ++f) {
                // the fundamental's first row carries its (t, top stage)
                if (!mbar_wait_bounded(&full[slot], phase)) {
                    good = false;
                    break;
                }
                const int2 tm = meta[slot];
                const int t = tm.x, st = tm.y;
                float sv[HC_PT];
#pragma unroll
                for (int c = 0; c < HC_PT; ++c) sv[c] = 0.f;
#pragma unroll
                for (int si = 1; si < NS; ++si) {
                    if (si <= st && good) {
                        for (int h = hlo[si]; h <= hhi[si]; ++h) {
                            if (!mbar_wait_bounded(&full[slot], phase)) {
                                good = false;
                                break;
                            }
                            float4 v[U];
#pragma unroll
                            for (int u = 0; u < U; ++u) v[u] = ring[slot * Q + u * HC_THREADS + tid];
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&empty[slot]);
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                sv[4 * u] += v[u].x;
                                sv[4 * u + 1] += v[u].y;
                                sv[4 * u + 2] += v[u].z;
                                sv[4 * u + 3] += v[u].w;
                            }
                            if (++slot == HR) {
                                slot = 0;
                                phase ^= 1u;
                            }
                        }
                        if (!good) break;
#pragma unroll
                        for (int c = 0; c < HC_PT; ++c) {
                            const bool ok = cell_ok(si, c);
                            if (ok && sv[c] > mx[si][c]) {
                                mx[si][c] = sv[c];
                                am[si][c] = t;
                            }
                            if (stats && ok) {
                                c1[si] += sv[c];
                                c2[si] = fmaf(sv[c], sv[c], c2[si]);
                            }
                        }
                    }
                }
                if (stats && ++cnt == 16) {
                    cnt = 0;
#pragma unroll
                    for (int si = 1; si < NS; ++si) {
                        dacc[si - 1][0][tid] += (double)c1[si];
                        dacc[si - 1][1][tid] += (double)c2[si];
                        c1[si] = c2[si] = 0.f;
                    }
                }
            }
            if (!good) {
                if (lane == 0) atomicExch(a.err, 1);
            } else {
#pragma unroll
                for (int si = 1; si < NS; ++si) {
#pragma unroll
                    for (int c = 0; c < HC_PT; ++c) {
                        if (cell_ok(si, c) && mx[si][c] >= 0.f) {
                            const int64_t p = p0 + 4 * HC_THREADS * (c >> 2) + (c & 3);
                            const unsigned long long packed =
                                ((unsigned long long)__float_as_uint(mx[si][c]) << 32) |
                                (unsigned long long)(0xFFFFFFFFu - (unsigned)am[si][c]);
                            if (!JERK_CHECK(p < n_cells[si], a.chk, kChkHarmStore)) continue;
                            if (ny == 1)
                                itm->M[si][p] = packed;
                            else
                                atomicMax(itm->M[si] + p, packed);
                        }
                    }
                }
            }
        }
        if (stats) {
            const int warp = tid >> 5;
#pragma unroll
            for (int si = 1; si < NS; ++si) {
                double x1 = dacc[si - 1][0][tid] + (double)c1[si], x2 = dacc[si - 1][1][tid] + (double)c2[si];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    x1 += __shfl_xor_sync(0xffffffffu, x1, o);
                    x2 += __shfl_xor_sync(0xffffffffu, x2, o);
                }
                if (lane == 0) {
                    red[si][0][warp] = x1;
                    red[si][1][warp] = x2;
                }
            }
        }
    }
    __syncthreads();
    if (stats && tid == 0) {
        const int64_t blk = blockIdx.x;
        for (int si = 1; si < NS; ++si) {
            double s1 = 0.0, s2 = 0.0;
            for (int w = 0; w < HC_THREADS / 32; ++w) {
                s1 += red[si][0][w];
                s2 += red[si][1][w];
            }
            a.stat_part[(blk * a.n_stages + si) * 2] = s1;
            a.stat_part[(blk * a.n_stages + si) * 2 + 1] = s2;
        }
    }
}

template <int NS>
static cudaError_t launch_harmonic_ns(const HarmArgs &a, unsigned blocks, bool stats, cudaStream_t st) {
    const int smem = HR * HC_CELLS * (int)sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(harmonic_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    harmonic_kernel<NS><<<blocks, HC_THREADS + 32, smem, st>>>(a, stats);
    return cudaGetLastError();
}

int harmonic_cells_per_block() { return HC_CELLS; }

cudaError_t launch_harmonic(const HarmArgs &a, int64_t blocks, bool stats, cudaStream_t st) {
    if (blocks > INT32_MAX) return cudaErrorInvalidValue;
    switch (a.n_stages) {
        case 2: return launch_harmonic_ns<2>(a, (unsigned)blocks, stats, st);
        case 3: return launch_harmonic_ns<3>(a, (unsigned)blocks, stats, st);
        case 4: return launch_harmonic_ns<4>(a, (unsigned)blocks, stats, st);
        default: return cudaErrorInvalidValue;
    }
}

// ---------------------------------------------------------------------------
// Statistics (Sec. 3: mean and standard deviation) -> thresholds.  Partial
// sums are reduced in a fixed order, so the result is deterministic.  One
// block per (item, stage).
// ---------------------------------------------------------------------------
__global__ void finalise_stats_kernel(const ItemDesc *items, const double *part1, const double *partH,
                                      int n_stages, const double *counts, const float *thresh, int mode,
                                      double *stats_out, float *theta_out) {
    __shared__ double r1[256], r2[256];
    const int si = blockIdx.x, item = blockIdx.y;
    const ItemDesc *itm = items + item;
    double s1 = 0.0, s2 = 0.0;
    if (mode == JERK_THRESH_SIGMA) {
        if (si == 0) {
            const double *p = part1 + 2 * itm->cta0;
            const int64_t n = itm->n_ctas;
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
                s1 += p[2 * i];
                s2 += p[2 * i + 1];
            }
        } else {
            const double *p = partH + 2 * n_stages * itm->harm0;
            const int64_t n = (int64_t)itm->harm_nx * itm->harm_ny;
            for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
                s1 += p[(i * n_stages + si) * 2];
                s2 += p[(i * n_stages + si) * 2 + 1];
            }
        }
    }
    r1[threadIdx.x] = s1;
    r2[threadIdx.x] = s2;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            r1[threadIdx.x] += r1[threadIdx.x + o];
            r2[threadIdx.x] += r2[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double cnt = counts[item * JERK_MAX_STAGES + si];
        double mu = 0.0, sd = 0.0;
        float theta = thresh[si];
        if (mode == JERK_THRESH_SIGMA && cnt > 0.0) {
            mu = r1[0] / cnt;
            const double var = r2[0] / cnt - mu * mu;
            sd = sqrt(var > 0.0 ? var : 0.0);
            theta = (float)(mu + (double)thresh[si] * sd);
        }
        stats_out[2 * (item * JERK_MAX_STAGES + si)] = mu;
        stats_out[2 * (item * JERK_MAX_STAGES + si) + 1] = sd;
        theta_out[item * JERK_MAX_STAGES + si] = theta;
    }
}

cudaError_t launch_finalise_stats(const ItemDesc *items, int n_items, const double *part1, const double *partH,
                                  int n_stages, const double *counts, const float *thresh, int mode,
                                  double *stats_out, float *theta_out, cudaStream_t st) {
    const dim3 grid((unsigned)n_stages, (unsigned)n_items);
    finalise_stats_kernel<<<grid, 256, 0, st>>>(items, part1, partH, n_stages, counts, thresh, mode, stats_out,
                                                theta_out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Peak finding (Sec. 3: "peaks which are above some user specified
// threshold"; the 1-D rule is a reading): p is kept when
// M(p) > theta, M(p) > M(p-1) and M(p) >= M(p+1), a missing neighbour
// counting as -inf.  Kept cells are compacted with one atomic counter.
// ---------------------------------------------------------------------------
__device__ __forceinline__ float mval(unsigned long long x) { return __uint_as_float((unsigned)(x >> 32)); }

__global__ void peaks_kernel(PeakArgs a) {
    const int si = blockIdx.y, item = blockIdx.z;
    const int64_t n = a.items[item].n_cells[si];
    const unsigned long long *M = a.items[item].M[si];
    const float theta = a.theta[item * JERK_MAX_STAGES + si];
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long x = M[p];
        const float v = mval(x);
        if (!(v > theta)) continue;
        const float l = p > 0 ? mval(M[p - 1]) : -FLT_MAX;
        const float r = p + 1 < n ? mval(M[p + 1]) : -FLT_MAX;
        if (v > l && v >= r) {
            const unsigned long long idx = atomicAdd(a.count, 1ull);
            if ((int64_t)idx < a.cap) {
                DevCand c;
                c.p = p;
                c.t = (int32_t)(0xFFFFFFFFu - (unsigned)(x & 0xFFFFFFFFull));
                c.stage_idx = si;
                c.power = v;
                c.item = item;
                a.out[idx] = c;
            }
        }
    }
}

cudaError_t launch_peaks(const PeakArgs &a, int n_items, int n_stages, int64_t most_cells, int sms, cudaStream_t st) {
    int64_t nblk = (most_cells + 255) / 256;
    const int64_t most = std::max<int64_t>(1, (int64_t)sms * 16 / n_items);   // every item and stage has its own blocks
    if (nblk > most) nblk = most;
    if (nblk < 1) nblk = 1;
    const dim3 grid((unsigned)nblk, (unsigned)n_stages, (unsigned)n_items);
    peaks_kernel<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Everything a search starts from 0, in one launch: the max-projections of
// all stages (8-byte words, 16 bytes at a time) and the candidate count.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) clear_kernel(ClearArgs a) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
#pragma unroll
    for (int si = 0; si < JERK_MAX_STAGES; ++si) {
        ulonglong2 *M = reinterpret_cast<ulonglong2 *>(a.M[si]);   // its own allocation: 256-byte aligned
        const int64_t n = a.n[si];
        for (int64_t i = i0; i < n / 2; i += step) M[i] = make_ulonglong2(0ull, 0ull);
        if (i0 == 0 && (n & 1)) a.M[si][n - 1] = 0ull;
    }
    if (i0 == 0) *a.count = 0ull;
}

cudaError_t launch_clear(const ClearArgs &a, int sms, cudaStream_t st) {
    int64_t nblk = (a.n[0] / 2 + 255) / 256;
    nblk = std::max<int64_t>(1, std::min<int64_t>(nblk, (int64_t)sms * 8));
    clear_kernel<<<(unsigned)nblk, 256, 0, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// The results into pinned host memory (one block; only what is there is
// written), so that reading them costs the host one event wait: four blocking
// copies for the candidates and three for each item's statistics took
// 10 us each, more than the kernels of a 2^16-bin search.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) publish_kernel(HostResult *res, double *h_stats, float *h_theta, int n_items,
                                                      const int *err, const unsigned long long *count, int64_t cap,
                                                      const DevCand *cand, const double *stats, const float *theta) {
    for (int i = threadIdx.x; i < n_items * 2 * JERK_MAX_STAGES; i += blockDim.x) h_stats[i] = stats[i];
    for (int i = threadIdx.x; i < n_items * JERK_MAX_STAGES; i += blockDim.x) h_theta[i] = theta[i];
    if (cand) {
        const unsigned long long c = *count;
        int64_t n = c < (unsigned long long)cap ? (int64_t)c : cap;
        if (n > kFirstCands) n = kFirstCands;
        constexpr int W = sizeof(DevCand) / 8;
        const unsigned long long *src = reinterpret_cast<const unsigned long long *>(cand);
        unsigned long long *dst = reinterpret_cast<unsigned long long *>(res->cand);
        for (int64_t i = threadIdx.x; i < n * W; i += blockDim.x) dst[i] = src[i];
        if (threadIdx.x == 0) res->count = c;
    }
    if (threadIdx.x == 0) res->err = *err;
}

cudaError_t launch_publish(HostResult *res, double *h_stats, float *h_theta, int n_items, const int *err,
                           const unsigned long long *count, int64_t cap, const DevCand *cand, const double *stats,
                           const float *theta, cudaStream_t st) {
    static_assert(sizeof(DevCand) % 8 == 0, "copied as 8-byte words");
    publish_kernel<<<1, 256, 0, st>>>(res, h_stats, h_theta, n_items, err, count, cap, cand, stats, theta);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Failure-path check: one thread waits, with the filter kernels' bounded
// wait, on a phase of an mbarrier that nothing completes; when the limit
// expires it sets the device error flag exactly as a filter CTA would, and
// returns.  Nothing else runs in the kernel.
// ---------------------------------------------------------------------------
__global__ void wait_check_kernel(int *err, uint64_t limit_ns) {
    __shared__ __align__(8) uint64_t bar;
    mbar_init(&bar, 1);
    if (!mbar_wait_for(&bar, 0, limit_ns)) atomicExch(err, 1);
}

cudaError_t launch_wait_check(int *err, uint64_t limit_ns, cudaStream_t st) {
    wait_check_kernel<<<1, 1, 0, st>>>(err, limit_ns);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Microbenchmarks for the roofline denominators that are not measured
// elsewhere: FP32 FMA throughput (8 independent FMA chains per thread, every
// SM full) and L2 read bandwidth (a buffer smaller than L2 read repeatedly
// with 16-byte loads).  Their outputs are consumed so nothing is elided.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(512) fma_peak_kernel(float *out, int iters, float a, float b) {
    float x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = (float)(threadIdx.x + i) * 1e-3f;
    for (int k = 0; k < iters; ++k) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = fmaf(x[i], a, b);
        }
    }
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += x[i];
    if (s == 12345.678f) out[blockIdx.x * blockDim.x + threadIdx.x] = s;   // practically never
}

// the same FP32 work as packed FMAs (fma.rn.f32x2, two lanes per instruction):
// 8 independent chains of float2 per thread
__global__ void __launch_bounds__(512) fma2_peak_kernel(float *out, int iters, float a, float b) {
    float2 x[8];
    const float2 a2 = make_float2(a, a), b2 = make_float2(b, b);
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = make_float2((float)(threadIdx.x + i) * 1e-3f, (float)i * 1e-3f);
    for (int k = 0; k < iters; ++k) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = __ffma2_rn(x[i], a2, b2);
        }
    }
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += x[i].x + x[i].y;
    if (s == 12345.678f) out[blockIdx.x * blockDim.x + threadIdx.x] = s;   // practically never
}

__global__ void __launch_bounds__(256) l2_read_kernel(const float4 *__restrict__ buf, int64_t n4, int reps,
                                                      float *out) {
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int r = 0; r < reps; ++r)
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
            const float4 v = __ldcg(buf + i);                 // cached in L2 only
            acc.x += v.x;
            acc.y += v.y;
            acc.z += v.z;
            acc.w += v.w;
        }
    if (acc.x + acc.y + acc.z + acc.w == 12345.678f) out[threadIdx.x] = acc.x;
}

cudaError_t measure_packed_fma(int sms, double *tflops) {
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float *scratch = nullptr;
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaMalloc(&scratch, sizeof(float) * 512 * sms * 4);
    float ms = 0.f;
    const int blocks = sms * 4, iters = 2048;
    for (int rep = 0; rep < 2 && e == cudaSuccess; ++rep) {   // the first run warms up
        cudaEventRecord(e0, st);
        fma2_peak_kernel<<<blocks, 512, 0, st>>>(scratch, iters, 0.999f, 1e-4f);
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    }
    // 4 flops per packed FMA (two lanes, two flops each)
    if (e == cudaSuccess) *tflops = 4.0 * 8 * 16 * (double)iters * blocks * 512 / (ms * 1e-3) / 1e12;
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaFree(scratch);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st) cudaStreamDestroy(st);
    return e;
}

int device_sms(int device) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n < 1) return 1;
    return n;
}

int current_device_sms() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 1;
    return device_sms(dev);
}

cudaError_t measure_peaks(int sms, double *fp32_tflops, double *l2_gbs) {
    cudaStream_t st = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    float *scratch = nullptr;
    float4 *buf = nullptr;
    const int64_t n4 = (64ll << 20) / 16;                    // 64 MB: inside the 129 MB L2
    cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e == cudaSuccess) e = cudaMalloc(&scratch, sizeof(float) * 512 * sms * 4);
    if (e == cudaSuccess) e = cudaMalloc(&buf, sizeof(float4) * n4);
    if (e == cudaSuccess) e = cudaMemsetAsync(buf, 0, sizeof(float4) * n4, st);
    float ms = 0.f;
    const int blocks = sms * 4, iters = 4096;
    for (int rep = 0; rep < 2 && e == cudaSuccess; ++rep) {   // the first run warms up
        cudaEventRecord(e0, st);
        fma_peak_kernel<<<blocks, 512, 0, st>>>(scratch, iters, 0.999f, 1e-4f);
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    }
    if (e == cudaSuccess)
        *fp32_tflops = 2.0 * 8 * 16 * (double)iters * blocks * 512 / (ms * 1e-3) / 1e12;
    const int reps = 20;
    for (int rep = 0; rep < 2 && e == cudaSuccess; ++rep) {
        cudaEventRecord(e0, st);
        l2_read_kernel<<<sms * 8, 256, 0, st>>>(buf, n4, reps, scratch);
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    }
    if (e == cudaSuccess) *l2_gbs = (double)n4 * 16 * reps / (ms * 1e-3) / 1e9;
    if (e == cudaSuccess) e = cudaGetLastError();
    cudaFree(buf);
    cudaFree(scratch);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (st) cudaStreamDestroy(st);
    return e;
}

}  // namespace jerk
