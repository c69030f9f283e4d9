// K5 -- non-maximum suppression (refinement stage of Section 3, run on the
// host in the paper; greedy IoU suppression here, on the device).
//
// One CTA (1024 threads) per frame, or a thread-block cluster of 2-8 CTAs
// that share its collection and suppression passes when the batch leaves SMs
// free. A batch of more frames than clusters that fit on the GPU at once runs
// on persistent clusters that draw frames from a ticket queue, most candidates
// first (a counting kernel and a one-CTA sort set the order), so the heaviest
// frames do not start last. Per frame:
//  1. every CTA of the cluster collects a share of the windows with score >
//     threshold into a list of its own: 64-bit keys (the float score mapped to
//     an order-reversing integer in the high word, level/wy/wx in the low
//     word, so ascending keys = score descending, then level, wy, wx
//     ascending) in its shared memory or, with a candidate cap above 16,384,
//     in its part of the frame's global scratch. The maps of a frame lie back
//     to back, so the scan is flat and all its loads are independent;
//  2. the best keys, at most kSeg of them (all of them, or those below a bound
//     found by a radix select over the cluster's lists), go to the leader,
//     which sorts them (bitonic, in registers and shuffles up to 64 keys per
//     warp) and decodes their boxes (exactly rounded float division);
//  3. the leader walks this segment in batches of the next 64 not yet
//     suppressed: all threads compute the batch's pairwise suppression bits,
//     warp 0 resolves the batch (kept iff no kept earlier member
//     suppresses it) and all threads suppress the rest of the segment against
//     the batch's kept members. This takes the same decisions as the
//     one-at-a-time greedy walk (candidates between batch members are already
//     suppressed);
//  4. if candidates remain, every CTA drops from its list the segment's keys
//     and those that the segment's kept boxes suppress, and the next segment
//     is taken. A later segment's candidates have met every kept box before
//     them, so the decisions stay those of the sequential walk.
// What bounds it: the latency of the one frame with the most candidates: 3,000
// to 10,000 cycles per batch of the walk, 15,000 to collect, 4,000 to 8,000 to sort.
// One 1242x375 frame (1,884 candidates) takes 31 us, 8 frames of 40 levels (up
// to 10,363 candidates) 137, 64 frames of 1242x375 68; with a scan level by level,
// a bitonic sort of all candidates and a cluster-wide pass over all of them after
// every batch it was 80, 317 and 117. A batch's edges lie apart from its boxes: 32
// bytes apart they put 16 lanes on one bank group (3,700 cycles per batch for the
// pairwise bits, 1,200 so).
// The IoU test first evaluates inter - thr * union in float. A coordinate sum or
// difference is off by at most 3 float roundings of values up to m, the frame's
// size or, for maps that reach beyond it, their farthest edge
// (eps = 3 m 2^-24), which moves the intersection by at most (w + h) eps and the
// IoU by at most eps (1 / w + 1 / h) through the intersection and as much again
// through the union (1.7e-5 for 64x128 windows of a 2048-pixel frame). So a float
// IoU further from the threshold than twice that bound for the frame's smallest
// window (plus 1e-6 for the products)
// decides. Otherwise the sign of inter - thr * union is taken from pairs of
// floats, good to 1e-10 of the union, and only nearer pairs go to double
// precision with explicitly rounded operations (no FMA contraction), the exact
// IEEE evaluation of the definition. Decisions are therefore the same as those
// of a plain double-precision implementation. (Double precision runs at two
// lanes per SM here: a call holds up the other warps' calls for over a
// thousand cycles, and one pair in a thousand that overlap is in the band.)
#include <cooperative_groups.h>

#include <algorithm>

#include "pd_internal.h"

namespace pd {
namespace {

constexpr int kThreads = 1024;
constexpr int kMaxCandidates = 16384;     // a CTA's list fits in shared memory
constexpr int kMaxCandidatesBig = 65536;  // lists in global scratch
constexpr int kSeg = 2048;                // candidates sorted and walked at a time
constexpr int kDigit = 11;                // radix select: bits per round
constexpr int kHist = 1 << kDigit;
constexpr int kMaxBoxes = 16384;
constexpr int kBatch = 64;                // greedy walk: candidates resolved per block-wide step
constexpr int kGrid = 32;                 // culling grid: kGrid x kGrid cells over the boxes' extent
constexpr int kCountBlocks = 32;          // blocks per frame counting its candidates
static_assert(nms_sched_ints(1) == 2 + kCountBlocks,
              "scheduling scratch: the ticket, then per frame its order slot and counts");
constexpr int kSoloWindows = 8192;        // frames of at most this many windows: one CTA (two rounds of loads)
constexpr int kOrderMax = 16384;          // frames the order kernel sorts (more: drawn in index order)
static_assert(kThreads == 16 * kBatch, "pairwise matrix: 16 threads per batch member");
static_assert(kThreads == kGrid * kGrid, "one culling cell per thread");
static_assert(kSeg == 2 * kThreads && kSeg / 32 == 64, "two segment entries per thread, two flag words per lane");
static_assert(kHist == 2 * kThreads, "two digits per thread");

__device__ __forceinline__ unsigned long long make_key(float s, int level, int wy, int wx) {
    const uint32_t u = __float_as_uint(s);
    const uint32_t ord = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    return ((unsigned long long)(~ord) << 32) |
           (uint32_t)((level << 24) | (wy << 12) | wx);
}

__device__ __noinline__ void decode_f64(long long nx, long long ny, int W, int H, int2 d, pd_box &b) {
    b.x = (float)__ddiv_rn((double)nx, (double)d.x);
    b.y = (float)__ddiv_rn((double)ny, (double)d.y);
    b.w = (float)__ddiv_rn(64.0 * W, (double)d.x);
    b.h = (float)__ddiv_rn(128.0 * H, (double)d.y);
}

// Score of a key's high word.
__device__ __forceinline__ float key_score(uint32_t hi) {
    const uint32_t ord = ~hi;
    return __uint_as_float((ord & 0x80000000u) ? (ord ^ 0x80000000u) : ~ord);
}

// Box of a key. x = 8*wx*W/Wk etc. are quotients of integers below 2^24, so
// the correctly rounded float quotient (__fdiv_rn) equals the double quotient
// rounded to float (a quotient of two such integers cannot lie within 2^-49
// of a float rounding midpoint without being on it): no double arithmetic.
__device__ __forceinline__ pd_box decode(unsigned long long key, int W, int H, const int2 *wkhk) {
    const uint32_t lo = (uint32_t)key;
    pd_box b;
    b.score = key_score((uint32_t)(key >> 32));
    b.level = (int)(lo >> 24);
    b.wy = (int)((lo >> 12) & 4095);
    b.wx = (int)(lo & 4095);
    const int2 d = wkhk[b.level];
    const long long nx = 8LL * b.wx * W, ny = 8LL * b.wy * H;
    if (nx < (1 << 24) && ny < (1 << 24) && 128LL * H < (1 << 24) && 64LL * W < (1 << 24) &&
        d.x < (1 << 24) && d.y < (1 << 24)) {
        b.x = __fdiv_rn((float)nx, (float)d.x);
        b.y = __fdiv_rn((float)ny, (float)d.y);
        b.w = __fdiv_rn((float)(64 * W), (float)d.x);
        b.h = __fdiv_rn((float)(128 * H), (float)d.y);
    } else {  // operands not exact in float: the double quotient, rounded
        decode_f64(nx, ny, W, H, d, b);
    }
    return b;
}

__device__ __forceinline__ double iou(const pd_box &a, const pd_box &b) {
    const double ax0 = a.x, ay0 = a.y, ax1 = __dadd_rn((double)a.x, (double)a.w),
                 ay1 = __dadd_rn((double)a.y, (double)a.h);
    const double bx0 = b.x, by0 = b.y, bx1 = __dadd_rn((double)b.x, (double)b.w),
                 by1 = __dadd_rn((double)b.y, (double)b.h);
    const double iw = __dsub_rn(fmin(ax1, bx1), fmax(ax0, bx0));
    const double ih = __dsub_rn(fmin(ay1, by1), fmax(ay0, by0));
    if (iw <= 0.0 || ih <= 0.0) return 0.0;
    const double inter = __dmul_rn(iw, ih);
    const double ua = __dsub_rn(__dadd_rn(__dmul_rn((double)a.w, (double)a.h),
                                          __dmul_rn((double)b.w, (double)b.h)),
                                inter);
    return __ddiv_rn(inter, ua);
}

// Out of line on purpose: the double-precision path is rare, and inlined it
// would be if-converted and executed for every pair.
__device__ __noinline__ double iou4(const float4 &a, const float4 &b) {
    pd_box x, y;
    x.x = a.x; x.y = a.y; x.w = a.z; x.h = a.w;
    y.x = b.x; y.y = b.y; y.w = b.z; y.h = b.w;
    return iou(x, y);
}

// IoU > thr by pairs of floats (about 46 bits): 1 yes, 0 no, -1 too near to
// tell. The edges x + w are exact pairs; the sign of inter - thr * union is
// taken as certain when it is more than 1e-10 of the union away from 0 (each
// step errs by at most a few 2^-46 of it).
struct Pair {
    float h, l;
};
__device__ __forceinline__ Pair two_sum(float a, float b) {
    const float s = a + b, t = s - a;
    return {s, (a - (s - t)) + (b - t)};
}
__device__ __forceinline__ Pair renorm(float h, float l) {
    const float s = h + l;
    return {s, l - (s - h)};
}
__device__ __forceinline__ Pair two_prod(float a, float b) {
    const float p = a * b;
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ Pair add(const Pair &a, const Pair &b) {
    const Pair s = two_sum(a.h, b.h), t = two_sum(a.l, b.l);
    const Pair v = renorm(s.h, s.l + t.h);
    return renorm(v.h, v.l + t.l);
}
__device__ __forceinline__ Pair mul(const Pair &a, const Pair &b) {
    const Pair p = two_prod(a.h, b.h);
    return renorm(p.h, p.l + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ Pair extent(float a0, float aw, float b0, float bw) {
    const Pair a = two_sum(a0, aw), b = two_sum(b0, bw);
    const bool less = a.h < b.h || (a.h == b.h && a.l < b.l);
    return add(less ? a : b, {-fmaxf(a0, b0), 0.f});
}
__device__ __noinline__ int iou_above(const float4 &a, const float4 &b, float thr) {
    const Pair iw = extent(a.x, a.z, b.x, b.z), ih = extent(a.y, a.w, b.y, b.w);
    if (iw.h <= 0.f || ih.h <= 0.f) return 0;
    const Pair inter = mul(iw, ih);
    const Pair ua = add(add(two_prod(a.z, a.w), two_prod(b.z, b.w)), {-inter.h, -inter.l});
    const Pair d = add(inter, mul({-thr, 0.f}, ua));
    if (fabsf(d.h) <= 1e-10f * ua.h) return -1;
    return d.h > 0.f ? 1 : 0;
}

// A box as its edges x0, y0, x1, y1 and area, for the float test.
struct Edges {
    float4 e;
    float area;
};
__device__ __forceinline__ Edges edges_of(const float4 &b) {
    return {make_float4(b.x, b.y, b.x + b.z, b.y + b.w), b.z * b.w};
}
__device__ __noinline__ bool suppresses_exact(float4 a, float4 b, float thr) {
    const int p = iou_above(a, b, thr);
    return p >= 0 ? p != 0 : iou4(a, b) > (double)thr;
}
// IoU > thr of boxes a and b (given also as edges), decided in float unless
// the IoU is within `band` of thr.
__device__ __forceinline__ bool suppresses(const Edges &a, const float4 &abox, const Edges &b, const float4 &bbox,
                                           float thr, float band) {
    const float iw = fmaxf(fminf(a.e.z, b.e.z) - fmaxf(a.e.x, b.e.x), 0.f);
    const float inter = iw * fmaxf(fminf(a.e.w, b.e.w) - fmaxf(a.e.y, b.e.y), 0.f);
    const float ua = (a.area + b.area) - inter;
    const float d = fmaf(-thr, ua, inter);
    if (fabsf(d) > band * ua) return d > 0.f;
    return suppresses_exact(abox, bbox, thr);
}

// Ascending bitonic sort of m = R * kThreads keys in shared memory k, with
// each thread holding the R consecutive keys [tid R, tid R + R) in registers:
// compare-exchange steps of stride j < R run in registers, R <= j < 32 R with
// warp shuffles (the partner is lane ^ j / R, same register), and only
// j >= 32 R through shared memory with a block barrier per step. Same network
// (and result) as bitonic_smem, with log2(m / 32R)-many fewer barriers per
// stage.
// The register and shuffle steps of one stage (stride j and below) for the
// R keys a thread holds, whose global indices are g0 .. g0 + R - 1.
template <int R>
__device__ __forceinline__ void bitonic_reg_steps(unsigned long long (&v)[R], int g0, int j, int len, int lane) {
    for (; j >= R; j >>= 1) {
        // partner: lane ^ (j / R), same register
        const int lm = j / R;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const unsigned long long o = __shfl_xor_sync(0xffffffffu, v[i], lm);
            const bool lower = (lane & lm) == 0, asc = ((g0 + i) & len) == 0;
            v[i] = (lower == asc) ? (v[i] < o ? v[i] : o) : (v[i] < o ? o : v[i]);
        }
    }
    // in registers: strides R/2 .. 1 (compile-time, so v stays in registers);
    // a stage of length len has only the strides below len
#pragma unroll
    for (int jj = R / 2; jj > 0; jj >>= 1) {
        if (jj >= len) continue;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int p = i ^ jj;
            if (p > i) {
                const bool asc = ((g0 + i) & len) == 0;
                const unsigned long long a = v[i], b = v[p];
                const bool sw = (a > b) == asc;
                v[i] = sw ? b : a;
                v[p] = sw ? a : b;
            }
        }
    }
}

// Compare-exchange steps of stride j .. jmin (>= jmin) over k[lo, lo + m) in
// shared memory, one block barrier per step (global indices lo + i).
__device__ __forceinline__ void bitonic_smem_steps(unsigned long long *k, int lo, int m, int j, int jmin, int len,
                                                   int tid) {
    for (; j >= jmin; j >>= 1) {
        for (int i = tid; i < m; i += kThreads) {
            const int ixj = i ^ j;
            if (ixj > i) {
                const unsigned long long a = k[lo + i], b = k[lo + ixj];
                if ((a > b) == (((lo + i) & len) == 0)) {
                    k[lo + i] = b;
                    k[lo + ixj] = a;
                }
            }
        }
        __syncthreads();
    }
}

// Ascending bitonic sort of m = R * kThreads keys k[lo, lo + m) in shared
// memory (as part of a larger network when lo > 0: directions follow the
// global index), each thread holding the R consecutive keys [lo + tid R,
// lo + tid R + R) in registers: compare-exchange steps of stride j < R run in
// registers, R <= j < 32 R with warp shuffles (the partner is lane ^ j / R,
// same register), and only j >= 32 R through shared memory with a block
// barrier per step. Same network (and result) as bitonic_smem, with
// log2(32R)-many fewer barriers per stage. Stages len = 2 .. len_max.
template <int R>
__device__ __forceinline__ void bitonic_hybrid(unsigned long long *k, int lo, int len_max, int tid) {
    constexpr int m = R * kThreads;
    unsigned long long v[R];
    const int base = lo + tid * R, lane = tid & 31;
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = k[base + i];
    for (int len = 2; len <= len_max; len <<= 1) {
        int j = len >> 1;
        if (j >= 32 * R) {
            // large strides: through shared memory
#pragma unroll
            for (int i = 0; i < R; ++i) k[base + i] = v[i];
            __syncthreads();
            bitonic_smem_steps(k, lo, m, j, 32 * R, len, tid);
            j = 16 * R;
#pragma unroll
            for (int i = 0; i < R; ++i) v[i] = k[base + i];
            __syncthreads();  // every thread has read its keys before the next stage writes
        }
        bitonic_reg_steps<R>(v, base, j, len, lane);
    }
#pragma unroll
    for (int i = 0; i < R; ++i) k[base + i] = v[i];
    __syncthreads();
}

// 16,384 keys: each 8,192-key half sorted by the hybrid network (the second
// half descending, as the bitonic network has it), then the last stage's
// large strides in shared memory and its small ones per half in registers.
__device__ __forceinline__ void bitonic_hybrid_16k(unsigned long long *k, int tid) {
    constexpr int R = 8, H = R * kThreads, M = 2 * H;
    bitonic_hybrid<R>(k, 0, H, tid);
    bitonic_hybrid<R>(k, H, H, tid);
    bitonic_smem_steps(k, 0, M, M / 2, 32 * R, M, tid);
    const int lane = tid & 31;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        unsigned long long v[R];
        const int base = h * H + tid * R;
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = k[base + i];
        bitonic_reg_steps<R>(v, base, 16 * R, M, lane);
#pragma unroll
        for (int i = 0; i < R; ++i) k[base + i] = v[i];
    }
    __syncthreads();
}

// Ascending sort of m (a power of two) keys in shared memory: the hybrid
// bitonic network for 1024 <= m <= 16384, the plain one otherwise.
__device__ __forceinline__ void bitonic_sort_smem(unsigned long long *k, int m, int tid);

// Ascending bitonic sort of m (a power of two) keys in shared memory.
__device__ __forceinline__ void bitonic_smem(unsigned long long *k, int m, int tid) {
    for (int len = 2; len <= m; len <<= 1) {
        for (int j = len >> 1; j > 0; j >>= 1) {
            for (int i = tid; i < m; i += kThreads) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const unsigned long long a = k[i], b = k[ixj];
                    if ((a > b) == ((i & len) == 0)) {
                        k[i] = b;
                        k[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
}

__device__ __forceinline__ void bitonic_sort_smem(unsigned long long *k, int m, int tid) {
    switch (m) {
        case 1024: bitonic_hybrid<1>(k, 0, m, tid); break;
        case 2048: bitonic_hybrid<2>(k, 0, m, tid); break;
        case 4096: bitonic_hybrid<4>(k, 0, m, tid); break;
        case 8192: bitonic_hybrid<8>(k, 0, m, tid); break;
        case 16384: bitonic_hybrid_16k(k, tid); break;
        default: bitonic_smem(k, m, tid);
    }
}

// A CTA's shared memory beside its key list.
struct NmsSmem {
    unsigned long long key[kSeg];               // the segment (leader)
    float4 box[kSeg];
    unsigned long long cmask[kGrid * kGrid];    // culling grid: kept boxes covering each cell
    int hist[kHist];
    int kept[kSeg];                             // the segment's kept entries, in order
    float4 bbx[kBatch];                         // the batch's boxes; a chunk of kept boxes
    float4 be[kBatch];                          // the same as edges, and areas (apart: 16 threads read
    float ba[kBatch];                           // 16 members in a row without bank conflicts)
    unsigned long long bcol[kBatch];            // member b: bit a set iff a < b and a suppresses b
    unsigned long long lohi[2][32];             // per warp: least and greatest key
    int4 krect[kBatch];                         // kept boxes' cell ranges x0, x1, y0, y1
    int2 wkhk[PD_MAX_LEVELS];                   // level sizes of this frame
    int first[PD_MAX_LEVELS];                   // its levels' first windows
    int cols[PD_MAX_LEVELS];
    int batch[kBatch];
    unsigned short rest[kSeg];                  // alive entries after the batch, in order
    uint32_t alive[kSeg / 32];
    int wsum[32];
    unsigned long long lo, hi;                  // least and greatest key of this CTA's list
    uint32_t keep[2];                           // the batch's kept members
    int n_list, n_seg, n_kept_seg, done, frame, digit, below;
    __device__ __forceinline__ Edges edges(int i) const { return {be[i], ba[i]}; }
    __device__ __forceinline__ void set_box(int i, const float4 &b) {
        const Edges e = edges_of(b);
        bbx[i] = b;
        be[i] = e.e;
        ba[i] = e.area;
    }
};

__device__ __forceinline__ unsigned long long umin64(unsigned long long a, unsigned long long b) { return a < b ? a : b; }
__device__ __forceinline__ unsigned long long umax64(unsigned long long a, unsigned long long b) { return a < b ? b : a; }

// Sorts the segment's m <= kSeg distinct keys ascending. Up to 256 keys by
// counting the smaller ones, four threads per key. More by the score's place
// among kHist equal parts of the segment's range of scores (monotone in the
// key: each float step rounds monotonically): a histogram gives every part its
// place, and a key's place among the few of its part is again the number of
// smaller ones. Where a part holds more than kCrowd keys (scores that hardly
// differ, infinities), by the bitonic network, whose 66 steps for 2,048 keys
// take 26,000 cycles.
constexpr int kCrowd = 64;
__device__ __forceinline__ void sort_segment(NmsSmem &S, int m, int tid) {
    unsigned long long *k = S.key;
    const int lane = tid & 31, warp = tid >> 5;
    if (m <= 256) {
        const int i = tid >> 2, q = tid & 3;
        const unsigned long long key = i < m ? k[i] : ~0ull;
        int c = 0;
        for (int j = q; j < m; j += 4) c += k[j] < key;
        c += __shfl_xor_sync(0xffffffffu, c, 1);
        c += __shfl_xor_sync(0xffffffffu, c, 2);
        __syncthreads();
        if (i < m && q == 0) k[c] = key;
        __syncthreads();
        return;
    }
    const bool has0 = tid < m, has1 = tid + kThreads < m;
    const unsigned long long k0 = has0 ? k[tid] : 0ull, k1 = has1 ? k[tid + kThreads] : 0ull;
    // least and greatest high words: the greatest and least score
    const uint32_t h0 = (uint32_t)(k0 >> 32), h1 = (uint32_t)(k1 >> 32);
    uint32_t mn = __reduce_min_sync(0xffffffffu, min(has0 ? h0 : ~0u, has1 ? h1 : ~0u));
    uint32_t mx = __reduce_max_sync(0xffffffffu, max(h0, h1));
    if (lane == 0) S.lohi[0][warp] = ((unsigned long long)mn << 32) | mx;
    S.hist[2 * tid] = S.hist[2 * tid + 1] = 0;
    __syncthreads();
    mn = __reduce_min_sync(0xffffffffu, (uint32_t)(S.lohi[0][lane] >> 32));
    mx = __reduce_max_sync(0xffffffffu, (uint32_t)S.lohi[0][lane]);
    const float best = key_score(mn), range = best - key_score(mx);
    const float scale = range > 0.f && range <= 3e38f ? (float)(kHist - 1) / range : 0.f;
    auto digit = [&](uint32_t h) { return min((int)((best - key_score(h)) * scale), kHist - 1); };
    // (scale 0: every key in part 0, also where the product is not a number, and the network sorts)
    const int d0 = scale > 0.f && has0 ? digit(h0) : 0, d1 = scale > 0.f && has1 ? digit(h1) : 0;
    const int r0 = has0 ? atomicAdd(&S.hist[d0], 1) : 0, r1 = has1 ? atomicAdd(&S.hist[d1], 1) : 0;
    __syncthreads();
    const int c0 = S.hist[2 * tid], c1 = S.hist[2 * tid + 1];
    if (__syncthreads_or(c0 > kCrowd || c1 > kCrowd)) {
        const int np = m <= kThreads ? kThreads : 2 * kThreads;
        for (int i = m + tid; i < np; i += kThreads) k[i] = ~0ull;
        __syncthreads();
        if (np == kThreads) bitonic_hybrid<1>(k, 0, np, tid);
        else bitonic_hybrid<2>(k, 0, np, tid);
        return;
    }
    int incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += a;
    }
    if (lane == 31) S.wsum[warp] = incl;
    __syncthreads();
    int w = lane < warp ? S.wsum[lane] : 0;
    w = __reduce_add_sync(0xffffffffu, w);
    const int start = w + incl - c0 - c1;
    S.hist[2 * tid] = start;  // a digit's first place; the next one's ends it
    S.hist[2 * tid + 1] = start + c0;
    __syncthreads();
    unsigned long long *t = reinterpret_cast<unsigned long long *>(S.box);  // the boxes come later
    if (has0) t[S.hist[d0] + r0] = k0;
    if (has1) t[S.hist[d1] + r1] = k1;
    __syncthreads();
    auto place = [&](unsigned long long key, int d) {
        const int a = S.hist[d], e = d + 1 < kHist ? S.hist[d + 1] : m;
        int c = a;
        for (int j = a; j < e; ++j) c += t[j] < key;
        k[c] = key;
    };
    if (has0) place(k0, d0);
    if (has1) place(k1, d1);
    __syncthreads();
}

__global__ void __launch_bounds__(kThreads) k_nms(const FrameDesc *__restrict__ frames,
                                                  const LevelDesc *__restrict__ levels,
                                                  const float *__restrict__ scores, float threshold,
                                                  float iou_thr, int cap, float4 *__restrict__ scratch,
                                                  pd_box *__restrict__ boxes, int max_boxes,
                                                  int32_t *__restrict__ counts, int n_frames,
                                                  const int *__restrict__ order, int *__restrict__ queue,
                                                  const unsigned *__restrict__ err, unsigned *__restrict__ err_out) {
    extern __shared__ __align__(16) unsigned char nms_raw[];
    NmsSmem &S = *reinterpret_cast<NmsSmem *>(nms_raw);
    // A frame is one cluster of C CTAs (C = 1 without a cluster launch); rank 0
    // leads. All ranks pass the same cluster barriers: what comes next follows
    // from values that all of them read after one.
    // Without a queue, cluster i takes frame i. With one (more frames than
    // clusters that fit on the GPU), the clusters are persistent: the leader
    // draws the next ticket, takes that frame of `order` (heaviest first)
    // and writes it into every rank's S.frame before the barrier that starts
    // the frame, so all ranks work on the same frame and stop together.
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const bool leader = rank == 0;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool big = cap > kMaxCandidates;
    NmsSmem &Lead = *cluster.map_shared_rank(&S, 0);
    auto csync = [&] {
        if (C > 1) cluster.sync();
        else __syncthreads();
    };
    const bool cull = iou_thr >= 0.5f;
    if (err_out && blockIdx.x == 0 && tid == 0) *err_out = *err;
    if (queue) csync();  // every CTA of the cluster runs before the leader writes into it
    for (;;) {
        if (queue) {
            if (leader && tid == 0) {
                const int t = atomicAdd(queue, 1);
                const int fr = t < n_frames ? (order ? order[t] : t) : -1;
                for (int r = 0; r < C; ++r) cluster.map_shared_rank(&S, r)->frame = fr;
            }
        } else if (tid == 0) {
            S.frame = (int)(blockIdx.x / C);
        }
        if (tid == 0) S.n_list = S.n_seg = 0;
        if (queue) csync();  // every rank knows the frame
        else __syncthreads();
        const int f = S.frame;
        if (f < 0) return;  // the same value in every rank: all leave together
        const FrameDesc &fd = frames[f];
        const int W = fd.W, H = fd.H, nl = fd.n_levels;
        const LevelDesc *lv = levels + fd.first_level;
        int n_win = 0;
        int64_t base = 0;
        if (nl > 0) {
            base = lv[0].score_off;
            n_win = (int)(lv[nl - 1].score_off + (int64_t)lv[nl - 1].rows * lv[nl - 1].cols - base);
        }
        for (int k = tid; k < nl; k += kThreads) {
            const LevelDesc &L = lv[k];
            S.wkhk[k] = make_int2(L.Wk, L.Hk);
            S.first[k] = (int)(L.score_off - base);
            S.cols[k] = L.cols;
        }
        __syncthreads();
        // the float test's band (see above): from the boxes' extent and the smallest window
        int wk = 1, hk = 1;
        for (int k = lane; k < nl; k += 32) {
            wk = max(wk, S.wkhk[k].x);
            hk = max(hk, S.wkhk[k].y);
        }
        wk = __reduce_max_sync(0xffffffffu, wk);
        hk = __reduce_max_sync(0xffffffffu, hk);
        const float band = 4.f * (3.f * 5.9604645e-8f * fmaxf(fd.ex, fd.ey)) *
                               ((float)wk / (64.f * (float)W) + (float)hk / (128.f * (float)H)) + 1e-6f;
        unsigned long long *list = big ? reinterpret_cast<unsigned long long *>(scratch + (size_t)f * nms_scratch_float4s(cap))
                                       : reinterpret_cast<unsigned long long *>(nms_raw + sizeof(NmsSmem));
        // ---- 1. candidates: this rank's share of the windows (every C-th run of
        // kThreads * kU), kU independent loads in flight; warp-aggregated appends.
        // With lists in global memory a first scan counts, which gives every rank its part.
        const float *sc = scores + base;
        auto scan = [&](bool count_only) {
            constexpr int kU = 4;
            for (int i0 = rank * kThreads * kU; i0 < n_win; i0 += C * kThreads * kU) {
                float v[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int i = i0 + u * kThreads + tid;
                    v[u] = i < n_win ? __ldg(sc + i) : -INFINITY;
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int i = i0 + u * kThreads + tid;
                    const bool hit = i < n_win && v[u] > threshold;
                    const unsigned m = __ballot_sync(0xffffffffu, hit);
                    if (!m) continue;
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&S.n_list, __popc(m));
                    if (count_only) continue;
                    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                    if (hit && (big || at < cap)) {
                        int lo = 0, hi = nl - 1;  // the window's level: the last one that starts at or before it
                        while (lo < hi) {
                            const int mid = (lo + hi + 1) >> 1;
                            if (S.first[mid] <= i) lo = mid;
                            else hi = mid - 1;
                        }
                        const int w = i - S.first[lo], wy = w / S.cols[lo];
                        list[at] = make_key(v[u], lo, wy, w - wy * S.cols[lo]);
                    }
                }
            }
        };
        scan(big);
        csync();  // every rank's count is in
        int n = 0, before = 0;
        for (int r = 0; r < C; ++r) {
            const int c = cluster.map_shared_rank(&S, r)->n_list;
            n += c;
            before += r < rank ? c : 0;
        }
        if (n == 0 || n > cap) {
            if (leader && tid == 0) {
                counts[2 * f] = 0;
                counts[2 * f + 1] = n > cap ? -n : 0;
            }
            csync();  // nobody clears its count or leaves while another rank reads it
            if (!queue) return;
            continue;
        }
        int n_list = S.n_list;  // this rank's list
        if (big) {
            csync();  // the counts have been read
            list += before;
            if (tid == 0) S.n_list = 0;
            __syncthreads();
            scan(false);
            __syncthreads();
        }
        int alive = n, kept_total = 0;  // candidates left in the cluster; kept boxes (leader)
        pd_box *out = boxes + (size_t)f * max_boxes;
        for (;;) {
            // ---- 2. the segment: all keys, or those below the bound of a radix select
            unsigned long long bound = ~0ull;
            if (alive > kSeg) {
                unsigned long long mn = ~0ull, mx = 0ull;
                for (int i = tid; i < n_list; i += kThreads) {
                    const unsigned long long k = list[i];
                    mn = umin64(mn, k);
                    mx = umax64(mx, k);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    mn = umin64(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                    mx = umax64(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                }
                if (lane == 0) {
                    S.lohi[0][warp] = mn;
                    S.lohi[1][warp] = mx;
                }
                __syncthreads();
                if (warp == 0) {
                    mn = S.lohi[0][lane];
                    mx = S.lohi[1][lane];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        mn = umin64(mn, __shfl_xor_sync(0xffffffffu, mn, o));
                        mx = umax64(mx, __shfl_xor_sync(0xffffffffu, mx, o));
                    }
                    if (lane == 0) {
                        S.lo = mn;
                        S.hi = mx;
                    }
                }
                csync();
                mn = ~0ull;
                mx = 0ull;
                for (int r = 0; r < C; ++r) {
                    mn = umin64(mn, cluster.map_shared_rank(&S, r)->lo);
                    mx = umax64(mx, cluster.map_shared_rank(&S, r)->hi);
                }
                // digits of kDigit bits from the highest bit in which the keys differ; the keys
                // of the digits below the one that overfills the segment are taken, and that
                // one is split further while they are less than half a segment
                int top = 64 - __clzll((long long)(mn ^ mx));  // bits [0, top) differ (at least 12: the keys are distinct)
                unsigned long long prefix = top < 64 ? mn >> top << top : 0ull;
                int taken = 0;
                for (;;) {
                    const int shift = top > kDigit ? top - kDigit : 0;
                    for (int i = tid; i < kHist; i += kThreads) S.hist[i] = 0;
                    __syncthreads();
                    for (int i = tid; i < n_list; i += kThreads) {
                        const unsigned long long k = list[i];
                        if (top == 64 || (k >> top) == (prefix >> top)) atomicAdd(&S.hist[(int)(k >> shift) & (kHist - 1)], 1);
                    }
                    csync();
                    // every rank adds up all histograms (two digits per thread) and finds the digit
                    int c0 = 0, c1 = 0;
                    for (int r = 0; r < C; ++r) {
                        const int2 c = *reinterpret_cast<const int2 *>(&cluster.map_shared_rank(&S, r)->hist[2 * tid]);
                        c0 += c.x;
                        c1 += c.y;
                    }
                    int incl = c0 + c1;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int a = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += a;
                    }
                    if (lane == 31) S.wsum[warp] = incl;
                    __syncthreads();
                    int excl = taken + incl - c0 - c1;
                    for (int w = 0; w < warp; ++w) excl += S.wsum[w];
                    // one thread holds the first digit whose keys no longer fit
                    if (excl <= kSeg && excl + c0 > kSeg) {
                        S.digit = 2 * tid;
                        S.below = excl;
                    } else if (excl + c0 <= kSeg && excl + c0 + c1 > kSeg) {
                        S.digit = 2 * tid + 1;
                        S.below = excl + c0;
                    }
                    csync();  // found; nobody clears its histogram while another rank reads it
                    taken = S.below;
                    prefix |= (unsigned long long)S.digit << shift;
                    top = shift;
                    if (taken >= kSeg / 2 || shift == 0) break;
                }
                bound = prefix - 1ull;  // the keys below the digit
            }
            for (int i0 = 0; i0 < n_list; i0 += kThreads) {
                const int i = i0 + tid;
                const unsigned long long k = i < n_list ? list[i] : 0ull;
                const bool take = i < n_list && k <= bound;
                const unsigned m = __ballot_sync(0xffffffffu, take);
                if (!m) continue;
                int at = 0;
                if (lane == 0) at = atomicAdd(&Lead.n_seg, __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (take && at < kSeg) Lead.key[at] = k;  // (the select keeps it below)
            }
            csync();  // the segment is with the leader
            // ---- 3. the leader sorts and walks it
            if (leader) {
                const int m = min(S.n_seg, kSeg);
                sort_segment(S, m, tid);
                for (int i = tid; i < m; i += kThreads) {
                    const pd_box b = decode(S.key[i], W, H, S.wkhk);
                    S.box[i] = make_float4(b.x, b.y, b.w, b.h);
                }
                if (tid < kSeg / 32) {
                    const int left = m - 32 * tid;
                    S.alive[tid] = left >= 32 ? 0xffffffffu : left > 0 ? (1u << left) - 1u : 0u;
                }
                __syncthreads();
                const float4 own0 = S.box[tid], own1 = S.box[tid + kThreads];  // (unused past m)
                int kept_seg = 0;
                for (;;) {
                    // the next (up to) 64 alive entries, in order: every warp ranks the entries of its
                    // two flag words by the words' prefix counts
                    const uint32_t wa = S.alive[2 * lane], wb = S.alive[2 * lane + 1];
                    int incl = __popc(wa) + __popc(wb);
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int a = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += a;
                    }
                    const int total = __shfl_sync(0xffffffffu, incl, 31);
                    if (total == 0 || kept_total >= max_boxes) break;
                    const int nb = min(total, kBatch);
                    uint32_t mine[2];
                    bool member[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int word = warp + 32 * h, src = word >> 1;
                        const uint32_t a = __shfl_sync(0xffffffffu, wa, src), b = __shfl_sync(0xffffffffu, wb, src);
                        const int pre = __shfl_sync(0xffffffffu, incl, src) - __popc(b) - (word & 1 ? 0 : __popc(a));
                        mine[h] = word & 1 ? b : a;
                        const int slot = pre + __popc(mine[h] & ((1u << lane) - 1u));
                        const bool on = (mine[h] >> lane) & 1u;
                        member[h] = on && slot < kBatch;
                        if (on && !member[h]) S.rest[slot - kBatch] = (unsigned short)(tid + h * kThreads);
                        if (member[h]) {
                            const float4 b = h ? own1 : own0;
                            S.batch[slot] = tid + h * kThreads;
                            S.set_box(slot, b);
                        }
                    }
                    __syncthreads();
                    {
                        // member b = tid / 16 is tested against members a = tid % 16, + 16, ..
                        // (a < b); the 16 threads of a member OR their bits together
                        const int b = tid >> 4, a0 = tid & 15;
                        unsigned long long bits = 0;
                        if (b < nb && a0 < b) {
                            const Edges bb = S.edges(b);
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int a = a0 + 16 * q;
                                if (a < b && suppresses(S.edges(a), S.bbx[a], bb, S.bbx[b], iou_thr, band)) bits |= 1ull << a;
                            }
                        }
#pragma unroll
                        for (int o = 8; o > 0; o >>= 1) bits |= __shfl_xor_sync(0xffffffffu, bits, o);
                        if ((tid & 15) == 0) S.bcol[b] = bits;
                    }
                    __syncthreads();
                    // Resolve in rounds (warp 0): a member is dropped once a kept member suppresses
                    // it, and kept once every member that could suppress it is decided and none of
                    // them is kept. This reaches the in-order result (induction on the member
                    // index) in as many rounds as the longest chain of suppressions. Lane l decides
                    // members l and l + 32; only members before it can suppress a member.
                    if (warp == 0) {
                        const uint32_t c0 = (uint32_t)S.bcol[lane];
                        const uint32_t c1 = (uint32_t)S.bcol[lane + 32], c2 = (uint32_t)(S.bcol[lane + 32] >> 32);
                        uint32_t kl = 0, kh = 0;                       // kept, low and high members
                        uint32_t ul = nb >= 32 ? ~0u : (1u << nb) - 1u;  // undecided
                        uint32_t uh = nb <= 32 ? 0u : nb == 64 ? ~0u : (1u << (nb - 32)) - 1u;
                        while (ul | uh) {
                            const bool u0 = (ul >> lane) & 1u, u1 = (uh >> lane) & 1u;
                            const bool s0 = c0 & kl, s1 = (c1 & kl) | (c2 & kh);   // suppressed
                            const bool k0 = u0 && !s0 && !(c0 & ul), k1 = u1 && !s1 && !((c1 & ul) | (c2 & uh));
                            kl |= __ballot_sync(0xffffffffu, k0);
                            kh |= __ballot_sync(0xffffffffu, k1);
                            ul &= ~__ballot_sync(0xffffffffu, u0 && (k0 || s0));
                            uh &= ~__ballot_sync(0xffffffffu, u1 && (k1 || s1));
                        }
                        // the cap on kept boxes: only the first (max_boxes - kept so far) in order
                        while (__popc(kl) + __popc(kh) > max_boxes - kept_total) {
                            if (kh) kh &= ~(0x80000000u >> __clz((int)kh));
                            else kl &= ~(0x80000000u >> __clz((int)kl));
                        }
                        if (lane < 2) S.keep[lane] = lane ? kh : kl;
                    }
                    // the members leave the flags meanwhile
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const uint32_t off = __ballot_sync(0xffffffffu, member[h]);
                        if (lane == 0) S.alive[warp + 32 * h] = mine[h] & ~off;
                    }
                    __syncthreads();
                    const uint32_t keep[2] = {S.keep[0], S.keep[1]};
                    const int n_keep = __popc(keep[0]) + __popc(keep[1]);
                    const uint32_t kw = warp ? keep[1] : keep[0];
                    if (tid < kBatch && ((kw >> lane) & 1u)) {  // warps 0 and 1
                        const int r = (warp ? __popc(keep[0]) : 0) + __popc(kw & ((1u << lane) - 1u));
                        const int e = S.batch[tid];
                        const unsigned long long key = S.key[e];
                        const uint32_t lo = (uint32_t)key;
                        const float4 bc = S.bbx[tid];
                        pd_box b;
                        b.x = bc.x;
                        b.y = bc.y;
                        b.w = bc.z;
                        b.h = bc.w;
                        b.score = key_score((uint32_t)(key >> 32));
                        b.level = (int)(lo >> 24);
                        b.wy = (int)((lo >> 12) & 4095);
                        b.wx = (int)(lo & 4095);
                        out[kept_total + r] = b;
                        S.kept[kept_seg + r] = e;
                    }
                    // the segment's later entries against the batch's kept members: 1 to 32 threads
                    // per entry, as many as the block has for the entries that are left
                    const int n_rest = total - nb;
                    int per = 1;
                    while (per < 32 && 2 * per * n_rest <= kThreads) per *= 2;
                    const int sub = tid & (per - 1);
                    // the members this thread tests: every per-th, from sub
                    const uint32_t part = (per == 1    ? ~0u
                                           : per == 2  ? 0x55555555u
                                           : per == 4  ? 0x11111111u
                                           : per == 8  ? 0x01010101u
                                           : per == 16 ? 0x00010001u
                                                       : 1u) << sub;
                    for (int i0 = 0; i0 < n_rest; i0 += kThreads / per) {
                        const int i = i0 + tid / per;
                        bool gone = false;
                        int e = 0;
                        if (i < n_rest) {
                            e = S.rest[i];
                            const float4 bj = S.box[e];
                            const Edges ej = edges_of(bj);
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                for (uint32_t k = keep[h] & part; k && !gone; k &= k - 1u) {
                                    const int j = 32 * h + __ffs((int)k) - 1;
                                    gone = suppresses(S.edges(j), S.bbx[j], ej, bj, iou_thr, band);
                                }
                        }
                        for (int o = per / 2; o > 0; o >>= 1) gone |= __shfl_xor_sync(0xffffffffu, (int)gone, o) != 0;
                        if (gone && sub == 0) atomicAnd(&S.alive[e >> 5], ~(1u << (e & 31)));
                    }
                    kept_total += n_keep;
                    kept_seg += n_keep;
                    __syncthreads();
                }
                if (tid == 0) {
                    S.n_kept_seg = kept_seg;
                    S.done = kept_total >= max_boxes;
                    S.n_seg = 0;
                }
            }
            if (bound == ~0ull) break;  // nothing is left behind the segment
            csync();  // the segment is walked
            if (Lead.done) break;
            // ---- 4. drop the segment's keys and what its kept boxes suppress, 64 of them at a time
            const int nk = Lead.n_kept_seg;
            const float gsx = (float)kGrid / fd.ex, gsy = (float)kGrid / fd.ey;
            // one run of keys per thread: test each against all kept boxes of the chunk; more:
            // only against those that cover its centre's cell
            const bool grid = cull && n_list > kThreads;
            for (int k0 = 0; k0 < nk || k0 == 0; k0 += kBatch) {
                const int kc = min(kBatch, nk - k0);
                if (tid < kc) {
                    const float4 b = Lead.box[Lead.kept[k0 + tid]];
                    S.set_box(tid, b);
                    S.krect[tid] = make_int4(max((int)floorf(b.x * gsx) - 1, 0),
                                             min((int)floorf((b.x + b.z) * gsx) + 1, kGrid - 1),
                                             max((int)floorf(b.y * gsy) - 1, 0),
                                             min((int)floorf((b.y + b.w) * gsy) + 1, kGrid - 1));
                }
                __syncthreads();
                if (grid) {
                    // Culling (IoU threshold >= 0.5): if IoU(A, B) > 0.5 then A's centre lies
                    // in B (were it outside B on one axis, A and B would overlap on at most
                    // half of A's extent there, so inter <= |A| / 2, and inter > (|A| + |B|)
                    // / 3 would need |B| < |A| / 2 while inter <= |B| needs |B| > |A| / 2).
                    // For every cell of a 32 x 32 grid over the boxes' extent: which of the kept boxes
                    // cover it (one cell of margin for rounding).
                    const int cx = tid & (kGrid - 1), cy = tid / kGrid;
                    unsigned long long m = 0ull;
                    for (int k = 0; k < kc; ++k) {
                        const int4 r = S.krect[k];
                        if (cx >= r.x && cx <= r.y && cy >= r.z && cy <= r.w) m |= 1ull << k;
                    }
                    S.cmask[tid] = m;
                    __syncthreads();
                }
                int left = 0;  // keys kept so far (the list is compacted in place, a run at a time)
                for (int i0 = 0; i0 < n_list; i0 += kThreads) {
                    const int i = i0 + tid;
                    const unsigned long long key = i < n_list ? list[i] : 0ull;
                    bool stay = i < n_list && key > bound;
                    if (stay && kc > 0) {
                        const pd_box b = decode(key, W, H, S.wkhk);
                        const float4 bj = make_float4(b.x, b.y, b.w, b.h);
                        const Edges ej = edges_of(bj);
                        if (grid) {
                            const int cx = min(max((int)floorf((b.x + 0.5f * b.w) * gsx), 0), kGrid - 1);
                            const int cy = min(max((int)floorf((b.y + 0.5f * b.h) * gsy), 0), kGrid - 1);
                            const unsigned long long m = S.cmask[cy * kGrid + cx];
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                for (uint32_t k = (uint32_t)(m >> (32 * h)); k && stay; k &= k - 1u) {
                                    const int j = 32 * h + __ffs((int)k) - 1;
                                    stay = !suppresses(S.edges(j), S.bbx[j], ej, bj, iou_thr, band);
                                }
                        } else {
                            for (int j = 0; j < kc && stay; ++j)
                                stay = !suppresses(S.edges(j), S.bbx[j], ej, bj, iou_thr, band);
                        }
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, stay);
                    if (lane == 0) S.wsum[warp] = __popc(m);
                    __syncthreads();  // also: the run has been read
                    const int c = S.wsum[lane];
                    const int total = __reduce_add_sync(0xffffffffu, c);
                    const int at = left + __reduce_add_sync(0xffffffffu, lane < warp ? c : 0);
                    if (stay) list[at + __popc(m & ((1u << lane) - 1u))] = key;
                    left += total;
                    __syncthreads();
                }
                n_list = left;
            }
            if (tid == 0) S.n_list = n_list;
            csync();  // the lists are compacted, the leader's segment is free
            alive = 0;
            for (int r = 0; r < C; ++r) alive += cluster.map_shared_rank(&S, r)->n_list;
            if (alive == 0) {
                csync();  // nobody clears its count while another rank reads it
                break;
            }
        }
        if (leader && tid == 0) {
            counts[2 * f] = kept_total;
            counts[2 * f + 1] = n;
        }
        if (!queue) {
            // one frame per cluster: after the last segment nobody reads another rank's
            // memory unless there were several (their bookkeeping is the leader's)
            if (n > kSeg) csync();
            return;
        }
    }
}

// Candidates per frame for the order of the persistent clusters. A frame's
// score maps lie back to back (its levels in order); block x of frame y
// counts the scores above the threshold in every kCountBlocks-th run of
// 4 x 256 of them, four loads in flight per thread.
__global__ void __launch_bounds__(256) k_nms_count(const FrameDesc *__restrict__ frames,
                                                   const LevelDesc *__restrict__ levels,
                                                   const float *__restrict__ scores, float threshold,
                                                   int *__restrict__ partial) {
    const int f = blockIdx.y;
    const FrameDesc fd = frames[f];
    int c = 0;
    if (fd.n_levels > 0) {
        const LevelDesc &a = levels[fd.first_level], &z = levels[fd.first_level + fd.n_levels - 1];
        const float *sc = scores + a.score_off;
        const int n = (int)(z.score_off + (int64_t)z.rows * z.cols - a.score_off);
        constexpr int kU = 4;
        for (int i0 = blockIdx.x * 256 * kU + threadIdx.x; i0 < n; i0 += kCountBlocks * 256 * kU) {
            float v[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) v[u] = i0 + u * 256 < n ? __ldg(sc + i0 + u * 256) : -INFINITY;
#pragma unroll
            for (int u = 0; u < kU; ++u) c += v[u] > threshold;
        }
    }
    c = __reduce_add_sync(0xffffffffu, c);
    __shared__ int ws[8];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < 8; ++w) t += ws[w];
        partial[f * kCountBlocks + blockIdx.x] = t;
    }
}

// The frames by candidates, most first (ties: lower frame first), and the
// ticket counter reset. One CTA, a bitonic sort of n_frames keys.
__global__ void __launch_bounds__(kThreads) k_nms_order(const int *__restrict__ partial, int n_frames,
                                                        int *__restrict__ order, int *__restrict__ queue) {
    extern __shared__ unsigned long long okeys[];
    const int tid = threadIdx.x;
    int np = 1;
    while (np < n_frames) np <<= 1;
    for (int i = tid; i < np; i += kThreads) {
        unsigned long long key = ~0ull;
        if (i < n_frames) {
            int c = 0;
            for (int b = 0; b < kCountBlocks; ++b) c += partial[i * kCountBlocks + b];
            key = ((unsigned long long)(uint32_t)(0x7fffffff - c) << 32) | (uint32_t)i;
        }
        okeys[i] = key;
    }
    __syncthreads();
    bitonic_sort_smem(okeys, np, tid);
    __syncthreads();
    for (int t = tid; t < n_frames; t += kThreads) order[t] = (int)(uint32_t)okeys[t];
    if (tid == 0) *queue = 0;
}

size_t nms_smem(int cap) {
    int p = 1;
    while (p < cap) p <<= 1;
    return sizeof(NmsSmem) + (cap > kMaxCandidates ? 0 : (size_t)p * sizeof(unsigned long long));
}

}  // namespace

namespace {
int g_nms_max_cluster = 1;  // largest cluster of k_nms CTAs the device can hold (1, 2, 4 or 8)
int g_nms_active[4] = {1, 0, 0, 0};  // clusters of 1, 2, 4, 8 CTAs that fit on the device at once

int log2_cluster(int c) { return c == 8 ? 3 : c == 4 ? 2 : c == 2 ? 1 : 0; }
}  // namespace

cudaError_t init_nms(bool occupancy) {
    const int smem = (int)nms_smem(kMaxCandidates);
    cudaError_t e = cudaFuncSetAttribute(k_nms, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_nms_order, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kOrderMax * (int)sizeof(unsigned long long));
    if (e != cudaSuccess || !occupancy) return e;
    int dev = 0, sms = 0, per_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
        (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_nms, kThreads, (size_t)smem)) != cudaSuccess)
        return e;
    g_nms_active[0] = std::max(sms * per_sm, 1);
    g_nms_max_cluster = 1;
    for (int c = 8; c >= 2; c >>= 1) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = (size_t)smem;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = c;
        attr.val.clusterDim.y = 1;
        attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_nms, &cfg) == cudaSuccess && n > 0) {
            g_nms_active[log2_cluster(c)] = n;
            g_nms_max_cluster = std::max(g_nms_max_cluster, c);
        } else {
            g_nms_active[log2_cluster(c)] = 0;
            (void)cudaGetLastError();  // a refused size is not an error
        }
    }
    return cudaSuccess;
}

int nms_cluster_for(int n_frames, int sm_count, int max_cand, int64_t windows) {
    // few windows: a second round of a CTA's loads costs less than the cluster's
    // barriers (320x240 frame, 139 candidates: 18.4 us with 8 CTAs, 16.4 with one)
    if (windows <= kSoloWindows) return 1;
    // the CTAs of a frame share its collection and passes; only while every CTA
    // still gets an SM of its own (one 1024-thread CTA per SM), or, for large
    // candidate lists, while two rounds of clusters cover the frames (the
    // clusters then draw the frames heaviest first)
    const int64_t budget = (max_cand > kMaxCandidates ? 2 : 1) * (int64_t)sm_count;
    int c = 1;
    while (2 * c <= g_nms_max_cluster && g_nms_active[log2_cluster(2 * c)] > 0 && (int64_t)n_frames * 2 * c <= budget)
        c *= 2;
    return c;
}

bool nms_persistent(int n_frames, int cluster) { return n_frames > g_nms_active[log2_cluster(cluster)]; }

int nms_launches(int n_frames, int cluster) {
    if (n_frames <= 0) return 0;
    return nms_persistent(n_frames, cluster) && n_frames <= kOrderMax ? 3 : 1;
}

cudaError_t launch_nms(cudaStream_t s, const FrameDesc *d_frames, const LevelDesc *d_levels,
                       int n_frames, const float *scores, float threshold, float iou,
                       float4 *scratch, int max_cand, pd_box *boxes, int max_boxes,
                       int32_t *counts, int cluster, int *sched, const unsigned *err, unsigned *err_out) {
    if (n_frames <= 0) return cudaSuccess;
    if (max_cand < 1 || max_cand > kMaxCandidatesBig || max_boxes < 1 || max_boxes > kMaxBoxes ||
        cluster < 1 || cluster > 8 || (cluster & (cluster - 1)))
        return cudaErrorInvalidValue;
    const size_t smem = nms_smem(max_cand);
    // more frames than clusters that fit at once: persistent clusters over a
    // ticket queue, frames ordered by their candidate counts (most first)
    int *queue = nullptr, *order = nullptr;
    int n_clusters = n_frames;
    if (sched && nms_persistent(n_frames, cluster)) {
        queue = sched;
        n_clusters = g_nms_active[log2_cluster(cluster)];
        if (n_frames <= kOrderMax) {
            order = sched + 1;
            int *partial = order + n_frames;
            k_nms_count<<<dim3(kCountBlocks, n_frames), 256, 0, s>>>(d_frames, d_levels, scores, threshold,
                                                                       partial);
            int np = 1;
            while (np < n_frames) np <<= 1;
            k_nms_order<<<1, kThreads, (size_t)np * sizeof(unsigned long long), s>>>(partial, n_frames, order,
                                                                                     queue);
        } else {
            const cudaError_t e = cudaMemsetAsync(queue, 0, sizeof(int), s);
            if (e != cudaSuccess) return e;
        }
    }
    if (cluster == 1) {
        k_nms<<<n_clusters, kThreads, smem, s>>>(d_frames, d_levels, scores, threshold, iou, max_cand, scratch,
                                                 boxes, max_boxes, counts, n_frames, order, queue, err, err_out);
        return cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_clusters * cluster);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = cluster;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_nms, d_frames, d_levels, scores, threshold, iou, max_cand, scratch, boxes,
                              max_boxes, counts, n_frames, (const int *)order, queue, err, err_out);
}

// ---------------------------------------------------------------------------
// Allocation-free NMS (pd_nms_noalloc). The kernel above needs device memory
// beyond its inputs and outputs: the frame / level descriptors it reads. For
// callers that cannot allocate device memory, that scratch lives in one file-scope array that every GPU loading
// this library holds until the process exits. A small set-up kernel copies
// the level geometry (passed by value) into it before the unchanged NMS
// kernel runs.
namespace {

constexpr int kNoAllocMaxCandidates = 16384;
constexpr int kNoAllocMaxLevels = PD_MAX_LEVELS;

struct NoAllocScratch {
    FrameDesc frame;
    LevelDesc levels[kNoAllocMaxLevels];
};

struct NoAllocGeometry {
    int32_t W, H, n_levels, pad;
    float ex, ey;
    int32_t Wk[kNoAllocMaxLevels], Hk[kNoAllocMaxLevels];
    int32_t rows[kNoAllocMaxLevels], cols[kNoAllocMaxLevels];
    int64_t score_off[kNoAllocMaxLevels];
};

}  // namespace

static __device__ __align__(256) unsigned char g_nms_scratch[sizeof(NoAllocScratch)];

namespace {

__global__ void k_nms_noalloc_setup(const __grid_constant__ NoAllocGeometry g, NoAllocScratch *s) {
    if (threadIdx.x == 0) {
        FrameDesc f{};
        f.W = g.W;
        f.H = g.H;
        f.first_level = 0;
        f.n_levels = g.n_levels;
        f.ex = g.ex;
        f.ey = g.ey;
        s->frame = f;
    }
    for (int k = threadIdx.x; k < g.n_levels; k += blockDim.x) {
        LevelDesc L{};
        L.W = g.W;
        L.H = g.H;
        L.Wk = g.Wk[k];
        L.Hk = g.Hk[k];
        L.rows = g.rows[k];
        L.cols = g.cols[k];
        L.score_off = g.score_off[k];
        s->levels[k] = L;
    }
}

}  // namespace

}  // namespace pd

extern "C" int pd_nms_noalloc(void *stream, const float *d_scores, int n_levels, const int32_t *rows,
                              const int32_t *cols, const int32_t *Wk, const int32_t *Hk, int W, int H,
                              float threshold, float nms_iou, int max_candidates, pd_box *d_boxes,
                              int max_boxes, int32_t *d_counts) {
    using namespace pd;
    if (!d_scores || !rows || !cols || !Wk || !Hk || !d_boxes || !d_counts || n_levels < 0 ||
        n_levels > kNoAllocMaxLevels || max_candidates < 1 || max_candidates > kNoAllocMaxCandidates ||
        max_boxes < 1 || max_boxes > kMaxBoxes || W < 1 || H < 1 || !(nms_iou >= 0.f))
        return PD_EINVAL;
    NoAllocGeometry g{};
    g.W = W;
    g.H = H;
    g.n_levels = n_levels;
    g.ex = (float)W;
    g.ey = (float)H;
    int64_t off = 0;
    for (int k = 0; k < n_levels; ++k) {
        if (rows[k] < 0 || cols[k] < 0 || rows[k] > 4096 || cols[k] > 4096 || Wk[k] < 1 || Hk[k] < 1)
            return PD_EINVAL;
        g.Wk[k] = Wk[k];
        g.Hk[k] = Hk[k];
        g.rows[k] = rows[k];
        g.cols[k] = cols[k];
        g.score_off[k] = off;
        off += (int64_t)rows[k] * cols[k];
        add_extent(g.ex, g.ey, W, H, Wk[k], Hk[k], rows[k], cols[k]);
    }
    // Every call: the current device's address of the scratch array (the
    // host-side symbol is only a stand-in) and the kernel's shared-memory
    // opt-in. Both are cheap host calls; doing them each time keeps the
    // address right after a device reset or on a new primary context.
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_nms_scratch) != cudaSuccess || !p) return PD_ECUDA;
    if (init_nms(false) != cudaSuccess) return PD_ECUDA;  // one cluster-less CTA: no occupancy table
    NoAllocScratch *scratch = reinterpret_cast<NoAllocScratch *>(p);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    k_nms_noalloc_setup<<<1, 128, 0, s>>>(g, scratch);
    if (cudaGetLastError() != cudaSuccess) return PD_ECUDA;
    if (launch_nms(s, &scratch->frame, scratch->levels, 1, d_scores, threshold, nms_iou, nullptr,
                   max_candidates, d_boxes, max_boxes, d_counts) != cudaSuccess)
        return PD_ECUDA;
    return PD_OK;
}
