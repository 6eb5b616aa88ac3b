// The fused overlap-and-save filter (conv.cu describes the path) at L = 4096,
// the segment length of every bank whose filters leave it room.
//
// One CTA holds three segments, four warps each, and walks a group of
// templates.  A thread keeps 16 points of the even-cell and 16 of the odd-cell
// half transform (2048 points each) side by side (pair.cuh), so its FP32 work
// is packed: 2048 = 8 x 16 x 16, three passes in registers.  The exchange after
// pass 0 goes over the segment's 128 threads through shared memory, 16 bytes (a
// pair of complex values) per access; the one after pass 1 stays within a warp
// and goes through tensor memory (exchange16).  The exchange buffers are padded
// (element i of sub-problem r at 276 r + i + i / 16), so that every access is free
// of bank conflicts and an immediate away from one base; three of them, the
// two-deep template ring and three staged rows fill 216 KB.  Tensor memory also
// holds what is the same for every template: the twiddles (pass 0: a pair of
// factors per output, the even half's w_2048^{f r} and the odd half's
// w_4096^{f (2r+1)}; pass 1: w_256^{f r}, each part twice, ready for packed
// products) and the segment's spectrum.  Its addresses are broadcast from lane 0
// once, so that the compiler keeps them in uniform registers.
//
// Why three segments of four warps: the passes of one segment wait on barriers
// over its four warps only, one warp on each of the SM's four schedulers, and
// the other two segments fill those waits; 166 registers a thread hold 16
// pairs (64), factors on their way, the running maxima (32) and their 8-bit
// argmaxima (8) without a spill.  What bounds it is latency at these 12 warps:
// FMA 62 %, issue 54 %, shared memory 47 % of their peaks, none of them full
// (with both exchanges in shared memory that pipe was the bound, at 71 %).  Filter alone, ms:
//
//                                         12 261 templates,  3131 templates,  27 391 templates,
//                                         2^21 bins, stages  700 001 bins     six requests,
//                                         1-2-4-8                             stage 1
//   one complex value per register pair,
//   256 threads a segment                 118.6              10.37            10.75
//   pairs, 128 threads a segment          106.4               9.08             9.28
//   second exchange in tensor memory      103.3               8.83             9.19
//   its second store 2 columns at a time,
//   uniform addresses                     101.1               8.65             9.14
//   argmaxima in registers                101.2               8.66             8.96
//   first exchange padded, not swizzled   100.1               8.58             8.84
//   loads and stores of the second
//   exchange under one another             99.2               8.50             8.70
//   statistics' lanes apart, groups cut
//   by parts.h                             98.9               8.20             8.59
//
// Not faster: the factors' loads issued a whole pass earlier (103.5 ms, and 104.2
// with the spectrum's a template earlier), so their latency is hidden already.
// Four segments a CTA, with both exchanges in shared memory: as four of four
// warps (maxima in tensor memory, pass-1 twiddles in shared memory, rows staged in
// the exchange buffer) 27 % slower on short spectra, and as two pairs of eight
// warps that read each template factor once per pair 109.0 against 106.4 ms at
// 2^21 bins and 9.38 against 9.28 ms.  One barrier per template, the buffers handed
// back through mbarriers: 101.6 against 100.1 ms.  The second round's loads under its
// stores as well: 100.8 against 99.2 ms.
#include <type_traits>

#include "device_sync.cuh"
#include "fft.cuh"
#include "jerk_internal.h"
#include "pair.cuh"
#include "rows.cuh"
#include "tmem.cuh"
#include "twosum.cuh"

namespace jerk {
namespace {

constexpr int L = 4096, NT = 128, SEGS = kPairSegs, THREADS = SEGS * NT, NBUF = 2;
constexpr int kFlush = 256;                               // templates per 8-bit argmax
constexpr int PADSUB = 256 + 16 + 4;                      // a sub-problem of 256 pairs, padded: i + i / 16, and 4 apart
constexpr int WORKB = 8 * PADSUB * 16;                    // exchange buffer of a segment (bytes)
constexpr int OFF_WORK = NBUF * L * 8;
constexpr int OFF_STAGE = OFF_WORK + SEGS * WORKB;        // staged power row, float [L] per segment
constexpr int SMEM = OFF_STAGE + SEGS * L * 4;
// tensor-memory columns: twiddles 0 .. 123 (the same words for the three segments'
// warps of a lane range), then 128 per segment: spectrum 32, statistics 4, exchange 64
constexpr uint32_t TMCOLS = 512, TMSEG = 128, TMSTAT = 32, TMX = 64;

// Pass 1's twiddled outputs in the order in which the exchange sends them (and
// their factors lie in tensor memory): 4, 8, 12, then 1, 5, 9, 13, and so on.
__host__ __device__ constexpr int order1(int q) { return (4 * (q + 1)) % 16 + (q + 1) / 4; }

// The forward transform's twiddles: the conjugates of the inverse's even-half
// factors, from this thread's tensor-memory columns.
struct FftTwFwd {
    uint32_t tcol;
    __device__ __forceinline__ static float2 w(const uint32_t (&x)[32], int q) {
        return make_float2(__uint_as_float(x[4 * q]), -__uint_as_float(x[4 * q + 2]));
    }
    template <int R>
    __device__ __forceinline__ void apply0(float2 *b, int i) const {
        static_assert(R == 8, "pass 0 of 2048 points");
        uint32_t x[32];
        tmem_ld32(tcol + 32 * i, x);
        tmem_wait_ld32(x);
#pragma unroll
        for (int r = 1; r < R; ++r) b[r] = cmul(b[r], w(x, r));
    }
    __device__ __forceinline__ void applys(float2 *a, int) const {
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            uint32_t x[32];
            tmem_ld32(tcol + 64 + 32 * c, x);
            tmem_wait_ld32(x);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (8 * c + q < 15) a[order1(8 * c + q)] = cmul(a[order1(8 * c + q)], w(x, q));
        }
    }
};

__device__ __forceinline__ cpair lds_pair(uint32_t addr) {
    cpair v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.re.x), "=f"(v.re.y), "=f"(v.im.x), "=f"(v.im.y)
                 : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_pair(uint32_t addr, cpair v) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.re.x), "f"(v.re.y), "f"(v.im.x),
                 "f"(v.im.y));
}

// times the q-th twiddle pair of 32 tensor-memory columns: (re, re, im, im) each
template <int N>
__device__ __forceinline__ cpair mul_tw(cpair a, const uint32_t (&w)[N], int q) {
    return mul(a, make_float2(__uint_as_float(w[4 * q]), __uint_as_float(w[4 * q + 1])),
               make_float2(__uint_as_float(w[4 * q + 2]), __uint_as_float(w[4 * q + 3])));
}

__device__ __forceinline__ uint32_t word(const cpair &v, int w) {
    return __float_as_uint(w == 0 ? v.re.x : w == 1 ? v.re.y : w == 2 ? v.im.x : v.im.y);
}
// The exchange between passes 1 and 2 through tensor memory.  Thread 2 i + s of
// the warp holds v[r], r = 0 .. 15, of point i of sub-problem s; thread 16 s + r
// leaves with v[i], i = 0 .. 15.  A store of 64 columns by lane and a load of 16
// lanes x 64 columns moves two bits of the register index into the low bits of
// the lane index and the lane index's two high bits into the registers: twice
// that is the whole transpose.
//
// First store, 16 columns of it: outputs r = t, t + 4, t + 8, t + 12
__device__ __forceinline__ void send16(const cpair (&v)[16], uint32_t tx, int t) {
    uint32_t x[16];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int w = 0; w < 4; ++w) x[8 * (w >> 1) + 2 * b + (w & 1)] = word(v[t + 4 * b], w);
    tmem_st16(tx + 16 * t, x);
}
// The rest of it, with t = 0, 1 sent, and the first stage of pass 2.  The first
// round's loads of columns 0 .. 31 run under the stores of the others, the last
// round's of the upper lanes under the butterflies of the lower ones.  The second
// store goes two columns at a time: the loads leave pairs that are two apart, and
// 16-column stores took 64 register moves to gather them.
__device__ __forceinline__ void exchange16(cpair (&v)[16], uint32_t tx) {
    uint32_t y[4][16];                                        // [2 h + u]: lanes 16 h .., columns 32 u ..
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        if (u == 1) {
            send16(v, tx, 2);
            send16(v, tx, 3);
        }
        tmem_wait_st();
        tmem_ld16x32(tx + 32 * u, y[u]);
        tmem_ld16x32(tx + (16u << 16) + 32 * u, y[2 + u]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) tmem_wait_ld16(y[e]);
    // y[2 h + u][4 q + 2 k + p]: point 8 h + 4 k + (lane >> 3), sub-problem (lane >> 2) & 1,
    // r = 4 (lane & 3) + 2 u + (q >> 1), word 2 (q & 1) + p
#pragma unroll
    for (int t = 0; t < 4; ++t)                               // t = 2 h + k
#pragma unroll
        for (int q = 0; q < 8; ++q)
            tmem_st2(tx + 16 * t + 8 * (q & 1) + 2 * (q >> 1), y[(t & 2) + (q >> 2)][4 * (q & 3) + 2 * (t & 1)],
                     y[(t & 2) + (q >> 2)][4 * (q & 3) + 2 * (t & 1) + 1]);
    tmem_wait_st();
    // y[2 H + u][4 Q + 2 K + p]: point 8 u + 4 (Q >> 1) + 2 H + K, word 2 (Q & 1) + p;
    // the first stage of pass 2 on the points of H = 0 while those of H = 1 are on their way
    tmem_ld16x32(tx, y[0]);
    tmem_ld16x32(tx + 32, y[1]);
    tmem_wait_ld16(y[0]);
    tmem_wait_ld16(y[1]);
#pragma unroll
    for (int H = 0; H < 2; ++H) {
        if (H == 0) {
            tmem_ld16x32(tx + (16u << 16), y[2]);
            tmem_ld16x32(tx + (16u << 16) + 32, y[3]);
        } else {
            tmem_wait_ld16(y[2]);
            tmem_wait_ld16(y[3]);
        }
#pragma unroll
        for (int k1 = 2 * H; k1 < 2 * H + 2; ++k1) {
#pragma unroll
            for (int i = k1; i < 16; i += 4) {
                const uint32_t(&z)[16] = y[(i & 2) + (i >> 3)];
                const int o = 4 * (2 * ((i >> 2) & 1)) + 2 * (i & 1);
                v[i].re = make_float2(__uint_as_float(z[o]), __uint_as_float(z[o + 1]));
                v[i].im = make_float2(__uint_as_float(z[o + 4]), __uint_as_float(z[o + 5]));
            }
            dft4(v[k1], v[k1 + 4], v[k1 + 8], v[k1 + 12]);
        }
    }
}

// byte_perm selector: byte b from the second operand's lowest
__host__ __device__ constexpr uint32_t sel_byte(int b) { return 0x3210u ^ ((uint32_t)(b ^ 4) << (4 * b)); }

template <bool ROWS>
__device__ __forceinline__ int bank_row(const ConvArgs &a, int k) {
    if constexpr (ROWS) return __ldg(a.rows + k);
    return k;
}

template <int MODE, bool STATS, bool ROWS>
__global__ void __launch_bounds__(THREADS, 1) conv_pair_kernel(ConvArgs a) {
    extern __shared__ __align__(1024) unsigned char sm[];
    __shared__ __align__(8) uint64_t full[NBUF];              // bulk copy of a template landed
    __shared__ int rel[NBUF];                                 // segments done reading a buffer
    __shared__ int issued[NBUF];                              // bulk copies issued per buffer
    __shared__ double red[2][THREADS / 32];
    __shared__ __align__(16) TplMeta tq[SEGS][4];             // (t, e0, e1) of template k at [k & 3]
    __shared__ __align__(16) RowEntries rent[SEGS][2];        // slot entries of template k at [k & 1]
    __shared__ int sbound[SEGS][JERK_MAX_HARMONIC][2];        // per h: first and last p of the segment
    __shared__ const int64_t *srow[SEGS][2];                  // this spectrum's row offset / length tables
    __shared__ uint32_t tslot;                                // tensor-memory base

    const int tid = threadIdx.x;
    const int seg = tid / NT, j = tid % NT;
    const int warp = tid >> 5;
    float2 *ring = reinterpret_cast<float2 *>(sm);
    float2 *work = reinterpret_cast<float2 *>(sm + OFF_WORK + seg * WORKB);
    float *stage = reinterpret_cast<float *>(sm + OFF_STAGE) + seg * L;
    const SyncNamed bar_seg{1 + seg, NT};

    // (spectrum, template group) entry of this CTA
    const int cta = MODE == 1 ? plane_cta(a) : (int)blockIdx.x;
    const int g = work_entry(a, cta);
    const ItemDesc *itm = a.items + __ldg(&a.grp[g].item);
    const int V = __ldg(&a.grp[g].V), bM = __ldg(&a.grp[g].bM);
    int tb = __ldg(&a.grp[g].tb), te = __ldg(&a.grp[g].te);
    if constexpr (MODE == 1) {
        // plane rows: only the asked-for templates of the group are filtered
        const int g1 = te;
        te = first_at_least(a.order, tb, g1, a.t0 + a.nt);
        tb = first_at_least(a.order, tb, te, a.t0);
        plane_part(a, tb, te);
        if (tb >= te) return;                                 // (uniform over the CTA, nothing set up yet)
    }
    const int s = (cta - __ldg(&a.grp[g].cta0)) * SEGS + seg;
    // first output cell (the last CTA's spare segments may start past every cell: kept below 2^31)
    const int64_t seg0w = (int64_t)s * V;
    const int seg0 = (int)(seg0w < itm->bN ? seg0w : itm->bN);

    if (tid < NBUF) {
        mbar_init(&full[tid], 1);
        rel[tid] = 0;
        issued[tid] = 0;
    }
    if (j == 0) {
        srow[seg][0] = itm->slot_off;
        srow[seg][1] = itm->slot_len;
    }
    if (j < JERK_MAX_HARMONIC) {
        // harmonic slots: cells q = h p in [seg0, seg0 + V), q < bN
        const int64_t bN = itm->bN;
        const int64_t h = j + 1;
        const int64_t pl = ((int64_t)seg0 + V - 1) / h;
        const int64_t pmax = (bN - 1) / h;
        sbound[seg][j][0] = (int)((seg0 + h - 1) / h);
        sbound[seg][j][1] = (int)(pl < pmax ? pl : pmax);
    }
    if (j == 0 && tb < te) {
        // the metadata pipeline's first stages (later ones are prefetched in the loop)
        const int t0 = __ldg(a.order + tb);
        tq[seg][tb & 3] = TplMeta{t0, __ldg(a.slot_beg + t0), __ldg(a.slot_beg + t0 + 1), 0};
        if (tb + 1 < te) tq[seg][(tb + 1) & 3].t = __ldg(a.order + tb + 1);
    }
    if (warp == 0) tmem_alloc_warp(smem_u32(&tslot), TMCOLS);
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    if (tid == 0)
        for (int b = 0; b < NBUF && tb + b < te; ++b) {
            issued[b] = 1;
            bulk_load(ring + b * L, a.bank + (int64_t)bank_row<ROWS>(a, tb + b) * L, (uint32_t)(L * sizeof(float2)),
                      &full[b]);
        }

    // ---- twiddles into tensor memory ---------------------------------------------
    // column 4 c, c = 8 i + r: pass 0, item i (f = j + 128 i), output r: even-half and
    // odd-half factors (re, re, im, im); c = 16 + q: pass 1, output order1(q), each part twice
    const uint32_t tcol = __shfl_sync(0xffffffffu, tslot + ((uint32_t)(32 * (warp & 3)) << 16), 0);
    const uint32_t tseg = __shfl_sync(0xffffffffu, tcol + TMSEG * (uint32_t)(1 + seg), 0);
    // pass 1 works on sub-problem jj >> 4, point jj & 15 (see the exchange below)
    const int jj = (j & 96) + 16 * (j & 1) + ((j & 31) >> 1);
    // (the three segments' warps of a lane range compute a third each)
#pragma unroll 1
    for (int c = seg; c < 16; c += SEGS) {
        float x[8];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int d = 2 * c + u;
            float2 wx, wy;
            if (d < 16) {
                const int f = j + NT * (d >> 3), r = d & 7;
                wx = unit_root<+1>((2 * f * r) & (L - 1), L);
                wy = unit_root<+1>((f * (2 * r + 1)) & (L - 1), L);
            } else {
                wx = wy = unit_root<+1>(((jj & 15) * (d == 31 ? 0 : order1(d - 16))) & 255, 256);
            }
            x[4 * u] = wx.x;
            x[4 * u + 1] = wy.x;
            x[4 * u + 2] = wx.y;
            x[4 * u + 3] = wy.y;
        }
        tmem_st8(tcol + 8 * c, x);
    }
    tmem_wait_st();
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();

    // ---- 1. forward transform of the segment's bins (2048 points) ----------------
    // this thread keeps the spectrum values it multiplies: X[j + 128 m] (the
    // spread segment's spectrum has period L / 2)
    {
        const FftTwFwd twf{tcol};
        const float2 *spec = itm->spec;
        const int64_t N = itm->N;
        const int64_t q0 = (seg0w - bM) / 2;                  // first bin (both even)
        float2 v[16];
#pragma unroll
        for (int m = 0; m < 16; ++m) {
            const int64_t q = q0 + j + NT * m;
            v[m] = q >= 0 && q < N ? spec[q] : make_float2(0.f, 0.f);
        }
        fft_pass0<11, -1>(v, twf);
        fft_store0<11>(v, work, j);
        fft_rest<11, -1>(v, work, jj, twf, bar_seg);
        const int rf = fft_rev<11>(jj);
        bar_seg();                                            // all reads of `work` done
#pragma unroll
        for (int r = 0; r < 16; ++r) work[rf + NT * r] = v[r];
        bar_seg();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float x[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 t = work[j + NT * (4 * c + q)];
                x[2 * q] = t.x;
                x[2 * q + 1] = t.y;
            }
            tmem_st8(tseg + 8 * c, x);
        }
        tmem_wait_st();
    }

    // ---- 2. templates of this group -----------------------------------------
    const uint32_t wb = smem_u32(work);
    const uint32_t w0 = wb + 16u * (uint32_t)(j + (j >> 4));                             // pass-0 stores
    const uint32_t w1 = wb + 16u * (uint32_t)((jj >> 4) * PADSUB + (jj & 15));           // pass-1 loads
    // this thread's outputs: cells c0 + 256 r + (0, 1)
    const int c0 = 2 * (j >> 4) + 16 * (j & 15);
    unsigned vmask = 0;
    // Bit r: the pair of cells r is valid (V, the segment starts and the number
    // of cells are even).  Bit 16: the pairs r < RSAFE of every thread of this
    // segment are, so the statistics mask only the others; uniform per segment.
    constexpr int RSAFE = 13;
    {
        const int64_t bN = itm->bN;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int cell = c0 + 256 * r;
            if (cell < V && seg0w + cell < bN) vmask |= 1u << r;
        }
        if (V >= 256 * RSAFE && seg0w + 256 * RSAFE <= bN) vmask |= 1u << 16;
    }
    uint32_t am[8];                                           // argmax bytes: position within kFlush templates
#pragma unroll
    for (int q = 0; q < 8; ++q) am[q] = 0;
    float2 mx[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) mx[r] = make_float2(-1.0f, -1.0f);
    // FP32 statistics partials, each of 16 cells x 32 templates (even and odd cells
    // apart: one of both was off by 1.4 times as much, RMS)
    float2 fa = make_float2(0.f, 0.f), fq = fa;
    // their FP64 sums sit in the last four of this thread's tensor-memory columns
    auto add_stats = [&] {
        double d0, d1;
        tmem_ld_f64x2(tseg + TMSTAT, d0, d1);
        d0 += (double)take_sum(fa);
        d1 += (double)take_sum(fq);
        tmem_st_f64x2(tseg + TMSTAT, d0, d1);
    };
    if constexpr (STATS) tmem_st_f64x2(tseg + TMSTAT, 0.0, 0.0);
    // Running maxima of the templates tb + base .. into the stage-1
    // max-projection, through the exchange buffer so that a warp's atomics fall on
    // 32 consecutive cells (straight from the registers each lane's was a sector of
    // its own: 27 K cycles per segment triple, nine templates' worth).  The
    // segment's threads call it together; the packed value of cells 2 q, 2 q + 1
    // sits at 16-byte slot q ^ ((q >> 3) & 7).
    auto flush_max = [&](int base) {
        bar_seg();                                            // every thread has read its last points
        ulonglong2 *pk = reinterpret_cast<ulonglong2 *>(work);
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            unsigned long long v[2];
#pragma unroll
            for (int l = 0; l < 2; ++l) {
                // A cell that is not a number under every template has no maximum and no
                // argmax (any valid position is read): 0, which replaces no other group's
                // maximum, where the bits of -1 would replace every one.
                const int t = __ldg(a.order + min(tb + base + (int)((am[(2 * r + l) >> 2] >> (8 * ((2 * r + l) & 3))) & 255u), te - 1));
                const float m = l ? mx[r].y : mx[r].x;
                v[l] = m < 0.f ? 0ull
                               : ((unsigned long long)__float_as_uint(m) << 32) |
                                     (unsigned long long)(0xFFFFFFFFu - (unsigned)t);
            }
            const int q = c0 / 2 + 128 * r;
            pk[q ^ ((q >> 3) & 7)] = make_ulonglong2(v[0], v[1]);
            mx[r] = make_float2(-1.0f, -1.0f);
        }
        bar_seg();
        const unsigned long long *p8 = reinterpret_cast<const unsigned long long *>(work);
        unsigned long long *M1 = itm->M1 + seg0;
        const int64_t left = itm->bN - seg0;
        const int n = left < V ? (int)left : V;
        for (int c = j; c < n; c += NT) {
            const int q = c >> 1;
            if (JERK_CHECK((int64_t)seg0 + c < itm->bN, a.chk, kChkMaxProj))
                atomicMax(M1 + c, p8[2 * (q ^ ((q >> 3) & 7)) + (c & 1)]);
        }
    };
    bool failed = false;
    // The last RD outputs r of every thread (cells at or past 256 (16 - RD)) lie
    // in the overlap of every segment of this group: the epilogue skips them and
    // the compiler drops the butterflies that only they need.
    auto template_loop = [&](auto rd) {
        constexpr int RK = 16 - decltype(rd)::value;          // outputs kept
        for (int k = tb; k < te; ++k) {                       // processing index
            const int it = k - tb;
            const int b = it % NBUF;
            uint32_t x[32];
            tmem_ld32(tseg, x);
            // A thread whose wait expired reads a buffer that may still be landing;
            // its values are discarded: the whole segment leaves at the barrier below.
            const bool ok = mbar_wait_bounded(&full[b], (uint32_t)(it / NBUF) & 1u);
            cpair v[16];
            {
                const float4 *t4 = reinterpret_cast<const float4 *>(ring + b * L) + j;
                tmem_wait_ld32(x);
#pragma unroll
                for (int m = 0; m < 16; ++m) {
                    const float4 t = t4[NT * m];              // even-half and odd-half factor of X[j + 128 m]
                    const float2 q = make_float2(__uint_as_float(x[2 * m]), __uint_as_float(x[2 * m + 1]));
                    v[m].re = make_float2(fmaf(q.x, t.x, -q.y * t.y), fmaf(q.x, t.z, -q.y * t.w));
                    v[m].im = make_float2(fmaf(q.x, t.y, q.y * t.x), fmaf(q.x, t.w, q.y * t.z));
                }
            }
            // pass 0: item i holds points f = j + 128 i + 256 k at v[2 k + i]
            tmem_ld32(tcol, x);
            dft8(v[0], v[2], v[4], v[6], v[8], v[10], v[12], v[14]);
            tmem_wait_ld32(x);
#pragma unroll
            for (int r = 0; r < 8; ++r) v[2 * r] = mul_tw(v[2 * r], x, r);
            tmem_ld32(tcol + 32, x);
            dft8(v[1], v[3], v[5], v[7], v[9], v[11], v[13], v[15]);
            tmem_wait_ld32(x);
#pragma unroll
            for (int r = 0; r < 8; ++r) v[2 * r + 1] = mul_tw(v[2 * r + 1], x, r);
            // One barrier per template over the segment's threads: it reports an
            // expired wait, ends this segment's reads of the buffer, and orders the
            // previous template's reads of `work` and `stage` before their reuse.
            cp_async_wait_all();                              // the copies issued last template
            if (named_any(1 + seg, NT, !ok)) {
                if (j == 0) atomicExch(a.err, 1);
                failed = true;
                break;
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int r = 0; r < 8; ++r) sts_pair(w0 + 16 * (PADSUB * r + (NT + NT / 16) * i), v[2 * r + i]);
            // the segment's last warp releases (and, last of the segments, refills) the buffer
            if (j == NT - 32) __threadfence_block();
            if (j == NT - 32 && atomicAdd(&rel[b], 1) == SEGS - 1) {
                rel[b] = 0;
                if (k + NBUF < te && !inject_at(a, 1, k + NBUF - tb)) {
                    issued[b] += 1;
                    bulk_load(ring + b * L, a.bank + (int64_t)bank_row<ROWS>(a, k + NBUF) * L,
                              (uint32_t)(L * sizeof(float2)), &full[b]);
                }
            }
            // Metadata pipeline (L2-latency loads kept off the critical path, no
            // registers held): order[k + 2], then slot_beg of template k + 1, then the
            // slot entries of template k, each landing before the next template's
            // first barrier.
            {
                if (j == 32) {
                    if (k + 2 < te) cp_async<4>(&tq[seg][(k + 2) & 3].t, a.order + k + 2);
                    if (k + 1 < te) {
                        const int t1 = tq[seg][(k + 1) & 3].t;
                        cp_async<4>(&tq[seg][(k + 1) & 3].e0, a.slot_beg + t1);
                        cp_async<4>(&tq[seg][(k + 1) & 3].e1, a.slot_beg + t1 + 1);
                    }
                }
                if constexpr (MODE == 0) {
                    const int ne = tq[seg][k & 3].e1 - tq[seg][k & 3].e0;   // this template's slot entries
                    const int i = j - 64;
                    if (i >= 0 && i < ne) {
                        const int e = tq[seg][k & 3].e0 + i;
                        RowEntries &en = rent[seg][k & 1];
                        cp_async<4>(&en.h[i], a.slot_h + e);
                        cp_async<8>(&en.off[i], srow[seg][0] + e);
                        cp_async<8>(&en.len[i], srow[seg][1] + e);
                    }
                }
                cp_async_commit();
            }
            if (k > tb) {
                // the previous template's staged row
                const TplMeta mp = tq[seg][(k - 1) & 3];
                if constexpr (MODE == 1)
                    store_plane_row(a, mp.t, stage, seg0, V, itm->bN, j, NT, kChkPlaneStore);
                else if (mp.e0 < mp.e1)
                    store_rows(a, rent[seg][(k - 1) & 1], mp.e1 - mp.e0, stage, sbound[seg], seg0, j, NT, kChkRowStore);
            }
            bar_seg();
            // pass 1: sub-problem jj / 16, points (jj & 15) + 16 k
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
                for (int k2 = 0; k2 < 4; ++k2) {
                    const int m = k1 + 4 * k2;
                    v[m] = lds_pair(w1 + 16 * 17 * m);
                }
            uint32_t xa[16], xb[16];
            tmem_ld16(tcol + 64, xa);
            dft16(v);
            tmem_wait_ld16(xa);
            tmem_ld16(tcol + 80, xb);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[order1(q)] = mul_tw(v[order1(q)], xa, q);
            send16(v, tseg + TMX, 0);
            tmem_wait_ld16(xb);
            tmem_ld16(tcol + 96, xa);
#pragma unroll
            for (int q = 4; q < 8; ++q) v[order1(q)] = mul_tw(v[order1(q)], xb, q - 4);
            send16(v, tseg + TMX, 1);
            tmem_wait_ld16(xa);
            tmem_ld16(tcol + 112, xb);
#pragma unroll
            for (int q = 8; q < 12; ++q) v[order1(q)] = mul_tw(v[order1(q)], xa, q - 8);
            tmem_wait_ld16(xb);
#pragma unroll
            for (int q = 12; q < 15; ++q) v[order1(q)] = mul_tw(v[order1(q)], xb, q - 12);
            exchange16(v, tseg + TMX);
            dft16_rest(v);
            float2 P[16];
#pragma unroll
            for (int r = 0; r < RK; ++r) P[r] = fma2(v[r].re, v[r].re, mul2(v[r].im, v[r].im));

            if constexpr (MODE == 0) {
                if (it > 0 && (it & (kFlush - 1)) == 0) flush_max(it - kFlush);
#pragma unroll
                for (int r = 0; r < RK; ++r) {
                    if (P[r].x > mx[r].x) {
                        mx[r].x = P[r].x;
                        am[(2 * r) >> 2] = __byte_perm(am[(2 * r) >> 2], it, sel_byte((2 * r) & 3));
                    }
                    if (P[r].y > mx[r].y) {
                        mx[r].y = P[r].y;
                        am[(2 * r + 1) >> 2] = __byte_perm(am[(2 * r + 1) >> 2], it, sel_byte((2 * r + 1) & 3));
                    }
                }
                // harmonic rows of this template: stage the power row now, store it
                // during the next template's transform (whose barriers order it)
                if (tq[seg][k & 3].e0 < tq[seg][k & 3].e1) {
#pragma unroll
                    for (int r = 0; r < RK; ++r)              // 256 r only sets bits that swzf neither reads nor changes
                        *reinterpret_cast<float2 *>(stage + swzf(c0) + 256 * r) = P[r];
                }
                if constexpr (STATS) {
                    // invalid cells (overlap, beyond the spectrum) count as 0
                    if (vmask >> 16) {
#pragma unroll
                        for (int r = RSAFE; r < RK; ++r)
                            if (!((vmask >> r) & 1u)) P[r] = make_float2(0.f, 0.f);
                    } else {
#pragma unroll
                        for (int r = 0; r < RK; ++r)
                            if (!((vmask >> r) & 1u)) P[r] = make_float2(0.f, 0.f);
                    }
                    // four packed chains, then their sum
                    float2 a2[4], q2[4];
#pragma unroll
                    for (int r = 0; r < 4; ++r) {
                        a2[r] = P[r];
                        q2[r] = mul2(P[r], P[r]);
                    }
#pragma unroll
                    for (int r = 4; r < RK; ++r) {
                        a2[r & 3] = add2(a2[r & 3], P[r]);
                        q2[r & 3] = fma2(P[r], P[r], q2[r & 3]);
                    }
                    fa = add2(fa, add2(add2(a2[0], a2[1]), add2(a2[2], a2[3])));
                    fq = add2(fq, add2(add2(q2[0], q2[1]), add2(q2[2], q2[3])));
                    if ((it & 31) == 31) add_stats();
                }
            } else {
#pragma unroll
                for (int r = 0; r < RK; ++r) *reinterpret_cast<float2 *>(stage + swzf(c0) + 256 * r) = P[r];
            }
        }
    };
    const int rd = 16 - (V + 255) / 256;
    if (rd >= 2)
        template_loop(std::integral_constant<int, 2>{});
    else if (rd == 1)
        template_loop(std::integral_constant<int, 1>{});
    else
        template_loop(std::integral_constant<int, 0>{});

    cp_async_wait_all();
    bar_seg();
    if (!failed && te > tb) {
        const TplMeta mp = tq[seg][(te - 1) & 3];
        if constexpr (MODE == 1) {
            store_plane_row(a, mp.t, stage, seg0, V, itm->bN, j, NT, kChkPlaneStore);
        } else {
            if (mp.e0 < mp.e1)
                store_rows(a, rent[seg][(te - 1) & 1], mp.e1 - mp.e0, stage, sbound[seg], seg0, j, NT, kChkRowStore);
        }
    }
    double d0 = 0.0, d1 = 0.0;
    if constexpr (STATS) {
        tmem_ld_f64x2(tseg + TMSTAT, d0, d1);
        d0 += (double)fa.x + (double)fa.y;
        d1 += (double)fq.x + (double)fq.y;
    }
    tmem_fence_before();
    __syncthreads();
    if (warp == 0) {
        tmem_fence_after();
        tmem_dealloc_warp(tslot, TMCOLS);
    }
    if (tid == 0) {
        // never leave with a bulk copy still writing into this CTA's shared memory
        for (int b = 0; b < NBUF; ++b)
            if (issued[b] > 0) mbar_wait_bounded(&full[b], (uint32_t)(issued[b] - 1) & 1u);
    }
    if constexpr (MODE == 0) {
        if (tb < te && !failed) flush_max((te - tb - 1) / kFlush * kFlush);
        if constexpr (STATS) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                d0 += __shfl_xor_sync(0xffffffffu, d0, o);
                d1 += __shfl_xor_sync(0xffffffffu, d1, o);
            }
            if ((tid & 31) == 0) {
                red[0][warp] = d0;
                red[1][warp] = d1;
            }
            __syncthreads();
            if (tid == 0) {
                double s1 = 0.0, s2 = 0.0;
                for (int w = 0; w < THREADS / 32; ++w) {
                    s1 += red[0][w];
                    s2 += red[1][w];
                }
                a.stat_part[2 * (int64_t)blockIdx.x] = s1;
                a.stat_part[2 * (int64_t)blockIdx.x + 1] = s2;
            }
        }
    }
}

template <int MODE, bool STATS, bool ROWS>
cudaError_t launch_pair(const ConvArgs &a, int n_ctas, cudaStream_t st) {
    auto k = conv_pair_kernel<MODE, STATS, ROWS>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (e != cudaSuccess) return e;
    k<<<MODE == 1 ? n_ctas * a.plane_parts : n_ctas, THREADS, SMEM, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_conv_pair(int mode, bool stats, const ConvArgs &a, int n_ctas, cudaStream_t st) {
    if (mode == 1) return launch_pair<1, false, false>(a, n_ctas, st);
    if (a.rows) return stats ? launch_pair<0, true, true>(a, n_ctas, st) : launch_pair<0, false, true>(a, n_ctas, st);
    return stats ? launch_pair<0, true, false>(a, n_ctas, st) : launch_pair<0, false, false>(a, n_ctas, st);
}

}  // namespace jerk
