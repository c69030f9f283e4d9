// K4 on the tensor cores -- block normalisation fused with the sliding-window
// linear SVM (Section 4.4, Algorithm 6; block features of Sections 4.2-4.3).
//
// score[wy][wx] = b + sum_{i<15} sum_{j<7} < f[wy+i][wx+j], w[i][j] >
// with f[by][bx] the 95-value block feature (36 L2-Hys HOG values of the 2x2
// cells, then the 59 L1-sqrt LBP values of their summed counts).
//
// Per block row r this is one GEMM: P[bx][(i, j)] = < f[r][bx], w[i][j] > for
// all 105 template positions (M = blocks, N = 105 padded to 112, K = 95 padded
// to 96). Window (wy, wx) then collects P_{wy+i}[wx+j][(i, j)] over its 15 x 7
// positions: the j terms come from the 7 neighbouring blocks of one block row,
// the i terms from 15 consecutive block rows. The GEMM runs on tcgen05 (bf16
// operands, fp32 accumulators in tensor memory); fp32 accuracy is kept by
// splitting both operands into bf16 high and low parts, x = xh + xl and
// w = wh + wl, and summing xh.wh + xl.wh + xh.wl (K = 3 x 96; the dropped
// xl.wl and the rounding of the low parts are below 2^-16 of |x w| per term).
//
// One persistent CTA per SM. Its 128 MMA rows are four groups of 32 (a TMEM
// lane quarter each), and every group walks its own items: up to 26 window
// columns (32 blocks, 33 cells) and up to 64 window rows of one level, one
// cell row per step. The groups share a step's MMAs and nothing else, so a
// level's width is padded to 26 columns and not to 104 (23 levels of a
// 1242x375 frame: 89 groups of work instead of 4 x 30), and items of any
// level or frame run side by side. The roles (mbarriers between them, bounded
// waits):
//  * warp 13, lane g: the items of group g (the first by its place in the
//    grid, the next ones from a queue), its TMA (cp.async.bulk.tensor.3d) of
//    one cell row per step into a ring of slots (9 HOG planes, f32, of 36
//    cells from a 4-cell boundary; 33 cells x 64 LBP count bytes, 64-byte
//    swizzle), and the step's description for the other roles;
//  * warps 0-3 (group = warp): 36 L2-Hys HOG values per block, warps 4-7 its
//    59 LBP values, written as bf16 high and low parts straight into the A
//    operand in tensor memory (tcgen05.st: row m = lane m, two bf16 per
//    column). A block needs two cell rows; the upper one stays in registers
//    from the step before, so every cell is read from shared memory once. LBP
//    counts are cell-major: a lane reads its cell's bins 16 at a time and adds
//    four at once, and a 512-entry table gives the bf16 split of the L1-sqrt;
//  * warp 12, one thread: the 18 MMAs of every step (A in tensor memory, the
//    template's B operand K-major no-swizzle canonical in shared memory, D in
//    one of two 128-column TMEM buffers), committed to the A-free and D-full
//    barriers;
//  * warps 8-11 (group = warp - 8): lane l adds P[l + j][(i, j)] (a shuffle by
//    j) to the running score of window row r - i, for all 105 positions, in
//    the fixed order (i, j) = (0,0), (0,1), ..., so every score is b plus its
//    terms in one order whatever the item cut; window row r - 14 is complete
//    and stored.
// A has three stages and D two buffers: the producers build steps s + 1 and
// s + 2 and the epilogue reads step s - 1 while step s's MMAs run.
// What bounds it: a step takes about 1,850 cycles, and the LBP warps, the HOG
// warps and the MMA warp are all busy for most of it: an LBP warp needs about
// 1,500 for its 320 instructions (3.5 warps per scheduler, fixed latencies and the
// shared-memory pipe, half busy), a HOG warp 1,400, the 18 MMAs 1,000 to issue
// and 1,280 to finish, and each wait on a barrier that is already complete costs
// about 100. The LBP warps were alone the slowest (1,780) while they held the
// spread sums of both cell rows and all of a step's results in registers, so
// that only a few table reads were in flight, and added the table's address
// to each. Handing on the finished stores later, or a packed bf16 split, changed
// nothing.
// 64 x 1242x375 frames: 0.293 ms (0.332 with those LBP warps and the MMAs
// issued by lane 0 alone); 0.661 ms with one strip of 104 columns per
// CTA, LBP planes read a byte per bin and summed in place, and a single warp
// issuing the MMAs between its epilogue rows (3,400 cycles per row, 901 rows
// per frame; now 693 steps). One 1242x375 frame: 84 -> 27 us, with items cut
// until every SM has work (see the planner). 14 warps leave 128 registers per
// thread (4 warps on a scheduler), which the epilogue's loads are staged for.
// Per-block HOG (Algorithm 5 read per block): each staged cell row holds 36
// HOG planes, the cell's 4 block-restricted histograms (plane 9 q + bin, q =
// its place in the block); a block takes q = 0, 1 from its upper row and
// q = 2, 3 from its lower one, and nothing else changes.
// Sparse path: a window is scored when every cell tile under it was computed;
// cell rows that no such window of the item needs are skipped. The caller has
// filled the score maps with -inf; a walked row's other windows get it again. A wait that gives up (1 s) sets the error word and a CTA flag that
// ends every role's waits; the CTA then drains its copies and MMAs, frees its
// tensor memory and leaves.
#include "pd_internal.h"

#include <cuda_bf16.h>

#include <cstring>
#include <vector>

#include "f32x2.cuh"

namespace pd {
namespace {

constexpr int kWarps = 14;            // 4 HOG, 4 LBP, 4 epilogue, MMA issue, items and TMA
constexpr int kThreads = 32 * kWarps;
constexpr int kGroups = 4;            // lane quarters of the A operand
constexpr int kM = 128;               // A rows = TMEM lanes
constexpr int kN = 112;               // 105 template positions, padded
constexpr int kChunks = 24;           // 16-byte K chunks per operand row: 12 high + 12 low
constexpr int kSBO = kChunks * 128;   // bytes per 8-row group
constexpr int kHogX = 36;             // HOG cells per staged row of a group (from a 4-cell boundary)
constexpr int kLbpX = 33;             // LBP cells per staged row of a group
constexpr int kTileRows = (kTcSparseRows - 1 + kWinBH) / kCellTH + 2;  // cell-tile rows under an item at most
static_assert(kTileRows <= 32 && kWinBW < kCellTW && kWinBH < 2 * kCellTH && kTcSparseRows + kWinBH <= 64 &&
                  kTcSparseRows > 32, "sparse masks");
constexpr int kMeta = 16;             // step descriptions in flight (more than any role can lag behind)
// Tensor memory: accumulators in columns 0..111 and 128..239, three A stages of
// 96 columns (bf16 pairs: 48 of high parts, 48 of low parts). The third stage's
// last low parts take the 16 columns that each accumulator leaves of its 128.
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kStages = 3;
__device__ __forceinline__ uint32_t a_hi(uint32_t stage) { return 256 + 96 * stage; }
// columns of the low parts [16 part, 16 part + 16)
__device__ __forceinline__ uint32_t a_lo(uint32_t stage, int part) {
    return stage < 2 ? 304 + 96 * stage + 16 * part : part == 0 ? 496 : part == 1 ? 112 : 240;
}
constexpr uint64_t kWaitNs = 1000000000ull;
constexpr int kBBytes = 14 * kSBO;    // B operand: template high | low parts
constexpr int kTabBytes = 512 * 4;    // sum of 4 cell counts -> bf16 high | low << 16 of sqrt(S / 256)
static_assert(kTcStrip + kWinBW - 1 <= 32, "a window's blocks inside a group");
static_assert(kBBytes + kTabBytes == kTcConstBytes, "constant block");

template <int HP>  // HOG planes per cell row: 9, or 36 for per-block HOG
struct SlotT {
    static constexpr int kHogBytes = (HP * kHogX * 4 + 127) / 128 * 128;
    uint8_t lbp[kGroups][2560];            // 33 cells x 64 bytes, swizzled; a 512-byte multiple per group
    uint8_t hog[kGroups][kHogBytes];       // [HP][36] floats
};
static_assert(sizeof(SlotT<9>) % 512 == 0 && sizeof(SlotT<36>) % 512 == 0, "TMA destinations");

// What a step is for one group. kind: 0 idle, 1 an item's (or run's) first
// cell row (no block row yet), 2 a block row, 3 no more steps.
struct StepMeta {
    uint32_t flags;  // kind | store << 2 | HOG x offset << 4 | window columns << 8
    uint32_t keep;   // windows of the stored row that are scored (others: -inf)
    int64_t out;     // score index of the stored row's first window
};

template <int HP>
struct TcSmemT {
    static constexpr int kSlots = HP == 9 ? 6 : 4;
    uint8_t b[kBBytes];
    uint32_t tab[512];
    SlotT<HP> slot[kSlots];               // staged cell rows
    StepMeta meta[kMeta][kGroups];
    uint32_t keep[kGroups][kTcSparseRows];  // sparse: scored windows of an item's rows
    unsigned long long bfull;             // constants arrived
    unsigned long long cfull[kSlots];     // cell row arrived (TMA transaction count)
    unsigned long long cempty[kSlots];    // cell row no longer read (8 producer warps)
    unsigned long long mready[kMeta];     // step description written
    unsigned long long afull[kStages];    // A operand written (8 producer warps)
    unsigned long long aempty[kStages];   // A operand read by the MMAs (commit)
    unsigned long long dfull[2];          // accumulators written (commit)
    unsigned long long dempty[2];         // accumulators read (4 epilogue warps)
    uint32_t tmem;
    volatile int failed;
};
static_assert(offsetof(TcSmemT<9>, slot) % 512 == 0 && offsetof(TcSmemT<36>, slot) % 512 == 0, "alignment");

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool try_wait(unsigned long long *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, 1000;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)  // suspended for up to 1000 ns: a spinning role takes issue slots
        : "memory");
    return ok != 0;
}
// Bounded wait for phase `parity`; gives up after 1 s (and marks the CTA
// failed) or as soon as another role has marked it failed.
template <class SM>
__device__ __forceinline__ bool bar_wait(SM &S, unsigned long long *bar, uint32_t parity, unsigned *err) {
    if (try_wait(bar, parity)) return true;
    const uint64_t t0 = global_ns();
    while (!S.failed) {
        if (try_wait(bar, parity)) return true;
        if (global_ns() - t0 > kWaitNs) {
            S.failed = 1;
            atomicOr(err, kErrTimeout);
            break;
        }
    }
    return false;
}
// Drain wait (after a failure): bounded, ignores the failed flag.
__device__ __forceinline__ void drain_wait(unsigned long long *bar, uint32_t parity) {
    const uint64_t t0 = global_ns();
    while (!try_wait(bar, parity) && global_ns() - t0 < kWaitNs) {
    }
}
__device__ __forceinline__ void arrive(unsigned long long *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void arrive_tx(unsigned long long *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_3d(void *dst, const CUtensorMap *map, unsigned long long *bar, int x, int y,
                                       int z) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
        : "memory");
}

// ---- tcgen05
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr) {  // K chunk stride 128 B, row group stride kSBO
    return (uint64_t)((saddr >> 4) & 0x3fff) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(kSBO >> 4) << 32) |
           (1ull << 46);
}
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kN >> 3) << 17) |
                            ((uint32_t)(kM >> 4) << 24);  // f32 D, bf16 A and B, K-major, N, M
// A from tensor memory (lane m = row m, K packed two bf16 per column)
__device__ __forceinline__ void umma_ts(uint32_t d, uint32_t a_tmem, uint64_t b, int acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
        "r"(a_tmem), "l"(b), "r"(kIdesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void umma_commit(unsigned long long *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

#define PD_LD_X16(taddr, v)                                                                                \
    asm volatile(                                                                                          \
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, "  \
        "[%16];"                                                                                           \
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),   \
          "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]),          \
          "=f"(v[15])                                                                                      \
        : "r"(taddr))
// waits for the loads so far; names the registers so that nothing reads them earlier
#define PD_WAIT_X16(v)                                                                                     \
    asm volatile("tcgen05.wait::ld.sync.aligned;"                                                          \
                 : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]),      \
                   "+f"(v[7]), "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), \
                   "+f"(v[14]), "+f"(v[15])::"memory")

// true in one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(p));
    return p != 0;
}
// bf16 high and low parts of a pair of floats, packed (first float in the low half)
__device__ __forceinline__ void split2(f32x2 x, uint32_t &hi, uint32_t &lo) {
    float a, b;
    unpack2(x, a, b);
    uint32_t h, l;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(b), "f"(a));
    const float ah = __uint_as_float(h << 16), bh = __uint_as_float(h & 0xffff0000u);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(b - bh), "f"(a - ah));
    hi = h;
    lo = l;
}
// this thread's TMEM lane: 2, 4, 8 or 16 consecutive 32-bit columns from taddr
__device__ __forceinline__ void tst2(uint32_t t, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(t), "r"(v[0]), "r"(v[1]) : "memory");
}
__device__ __forceinline__ void tst4(uint32_t t, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(t), "r"(v[0]), "r"(v[1]),
                 "r"(v[2]), "r"(v[3])
                 : "memory");
}
__device__ __forceinline__ void tst8(uint32_t t, const uint32_t *v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(t), "r"(v[0]),
                 "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tst16(uint32_t t, const uint32_t *v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(t),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}

// The 36 HOG values of A row m into its TMEM lane (feature f in column f / 2 of
// the stage's high and low parts): cells (r, c), (r, c+1),
// (r+1, c), (r+1, c+1) in the template's order (TL, TR, BL, BR, 9 bins each),
// L2-Hys, bf16 split.
__device__ __forceinline__ void build_hog(const float (&x)[36], float clip, uint32_t lanes, uint32_t stage) {
    // sums of squares in four interleaved partial sums (independent chains)
    f32x2 v[18], q01 = 0ull, q23 = 0ull;
#pragma unroll
    for (int t = 0; t < 18; ++t) {
        v[t] = pack2(x[2 * t], x[2 * t + 1]);
        f32x2 &q = t & 1 ? q23 : q01;
        q = fma2(v[t], v[t], q);
    }
    const float i1 = rsqrtf((lo2(q01) + hi2(q01)) + (lo2(q23) + hi2(q23)) + 1.0f);
    const f32x2 i11 = dup2(i1);
    q01 = q23 = 0ull;
#pragma unroll
    for (int t = 0; t < 18; ++t) {
        float p, r;
        unpack2(mul2(v[t], i11), p, r);
        v[t] = pack2(fminf(p, clip), fminf(r, clip));
        f32x2 &q = t & 1 ? q23 : q01;
        q = fma2(v[t], v[t], q);
    }
    const float i2 = rsqrtf((lo2(q01) + hi2(q01)) + (lo2(q23) + hi2(q23)) + 1e-6f);
    const f32x2 i22 = dup2(i2);
    uint32_t hi[18], lo[18];
#pragma unroll
    for (int t = 0; t < 18; ++t) split2(mul2(v[t], i22), hi[t], lo[t]);
    tst16(lanes + a_hi(stage), hi);
    tst2(lanes + a_hi(stage) + 16, hi + 16);
    tst16(lanes + a_lo(stage, 0), lo);
    tst2(lanes + a_lo(stage, 1), lo + 16);
}

// Horizontal sums of the LBP counts of a cell and its right neighbour, four
// bins per word. Cells are 64 bytes, 16-byte chunks swizzled by the cell's bits
// 1, 2. Counts are at most 64, so byte sums do not carry (larger ones would only
// give another entry of the 512-entry table).
__device__ __forceinline__ void lbp_row(const uint8_t *base, int cell, uint32_t (&h)[15]) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint4 x = *reinterpret_cast<const uint4 *>(base + cell * 64 + ((k ^ ((cell >> 1) & 3)) << 4));
        const uint4 y =
            *reinterpret_cast<const uint4 *>(base + (cell + 1) * 64 + ((k ^ (((cell + 1) >> 1) & 3)) << 4));
        const uint32_t v[4] = {x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (4 * k + u < 15) h[4 * k + u] = v[u];
    }
}

__device__ __forceinline__ uint32_t table_word(uint32_t at) {  // read-only once the constants are there
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(at));
    return v;
}
// bf16 split pairs of four bins from the table (columns 2 w, 2 w + 1 of the LBP
// part): u, l the bins' sums of the upper and the lower cell row; base: the table's
// shared-memory address, in both halves (it is below 2^16, so two addresses fit a word).
__device__ __forceinline__ void lbp_word(uint32_t base, uint32_t u, uint32_t l, uint32_t *hi, uint32_t *lo) {
    const uint32_t e = 4u * (__byte_perm(u, 0u, 0x4240) + __byte_perm(l, 0u, 0x4240)) + base;  // bins 4 w, 4 w + 2
    const uint32_t o = 4u * (__byte_perm(u, 0u, 0x4341) + __byte_perm(l, 0u, 0x4341)) + base;  // bins 4 w + 1, 4 w + 3
    const uint32_t v0 = table_word(e & 0xffffu), v1 = table_word(o & 0xffffu);
    const uint32_t v2 = table_word(e >> 16), v3 = table_word(o >> 16);
    hi[0] = __byte_perm(v0, v1, 0x5410);
    lo[0] = __byte_perm(v0, v1, 0x7632);
    hi[1] = __byte_perm(v2, v3, 0x5410);
    lo[1] = __byte_perm(v2, v3, 0x7632);
}

template <int HP>
__global__ void __launch_bounds__(kThreads, 1)
    k_svm_tc(const __grid_constant__ CUtensorMap hog_map, const __grid_constant__ CUtensorMap lbp_map,
             const LevelDesc *__restrict__ levels, const TcItem *__restrict__ items, int n_items,
             int *__restrict__ queue, const unsigned char *__restrict__ consts, float bias, float clip,
             float *__restrict__ scores, const uint32_t *__restrict__ c_flag, unsigned *__restrict__ err,
             const CUtensorMap *__restrict__ level_maps) {
    using Slot = SlotT<HP>;
    using TcSmem = TcSmemT<HP>;
    constexpr int kSlots = TcSmem::kSlots;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    TcSmem &S = *reinterpret_cast<TcSmem *>(smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // operand and TMA alignment, table addresses of 16 bits: never expected to fail
    if ((smem_u32(smem_raw) & 1023u) || smem_u32(S.tab) + kTabBytes > 65536u) {
        if (tid == 0) atomicOr(err, kErrTimeout);
        return;
    }
    if (tid == 0) {
        auto init = [](unsigned long long *bar, uint32_t count) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
        };
        init(&S.bfull, 1);
        for (int s = 0; s < kSlots; ++s) {
            init(&S.cfull[s], 1);
            init(&S.cempty[s], 2 * kGroups);
        }
        for (int s = 0; s < kMeta; ++s) init(&S.mready[s], 1);
        for (int s = 0; s < (int)kStages; ++s) {
            init(&S.afull[s], 2 * kGroups);
            init(&S.aempty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            init(&S.dfull[s], 1);
            init(&S.dempty[s], kGroups);
        }
        S.failed = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // the template's B operand and the LBP table, laid out by the host
        arrive_tx(&S.bfull, kTcConstBytes);
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                smem_u32(S.b)),
            "l"(reinterpret_cast<uint64_t>(consts)), "r"(kTcConstBytes), "r"(smem_u32(&S.bfull))
            : "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&S.tmem)),
                     "r"(kTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem;
    // bounded wait by every lane of a warp, decided for the whole warp
    auto warp_wait = [&](unsigned long long *bar, uint32_t parity) {
        return __all_sync(0xffffffffu, bar_wait(S, bar, parity, err)) != 0;
    };
    uint32_t loads = 0, committed = 0;  // cell-row steps sent (warp 13), MMA steps committed (warp 12)

    if (warp < 8) {
        // ---- producers: warps 0-3 the HOG part of group `warp`, warps 4-7 the
        // LBP part of group warp - 4; lane m = block m of the group
        const int g = warp & 3;
        const bool is_lbp = warp >= 4;
        const uint32_t lanes = tmem + ((uint32_t)(32 * g) << 16);
        bool ok = !is_lbp || warp_wait(&S.bfull, 0);
        auto stage_free = [&](uint32_t s) {
            return s < kStages || warp_wait(&S.aempty[s % kStages], (s / kStages - 1) & 1u);
        };
        auto publish = [&](uint32_t s) {
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive(&S.afull[s % kStages]);
        };
        if (!is_lbp) {
            constexpr int pq = HP == 36 ? kHogBins : 0;  // per-block: plane set of the cell's place
            float up[18];                                // the upper cell row: cells c, c + 1
#pragma unroll
            for (int t = 0; t < 18; ++t) up[t] = 0.f;
            for (uint32_t s = 0; ok; ++s) {
                if (!(ok = warp_wait(&S.cfull[s % kSlots], (s / kSlots) & 1u))) break;
                const uint32_t fl = S.meta[s % kMeta][g].flags, kind = fl & 3u;
                if (kind == 3u) break;
                const float *hs = reinterpret_cast<const float *>(S.slot[s % kSlots].hog[g]) + lane + ((fl >> 4) & 3u);
                float x[36], nxt[18];
#pragma unroll
                for (int t = 0; t < 18; ++t) x[t] = up[t];
#pragma unroll
                for (int t = 0; t < kHogBins; ++t) {
                    x[18 + t] = hs[(2 * pq + t) * kHogX];
                    x[27 + t] = hs[(3 * pq + t) * kHogX + 1];
                    nxt[t] = pq ? hs[t * kHogX] : x[18 + t];
                    nxt[9 + t] = pq ? hs[(pq + t) * kHogX + 1] : x[27 + t];
                }
#pragma unroll
                for (int t = 0; t < 18; ++t) up[t] = nxt[t];
                __syncwarp();
                if (lane == 0) arrive(&S.cempty[s % kSlots]);
                if (!(ok = stage_free(s))) break;
                if (kind == 2u) {
                    tc_fence_after();
                    build_hog(x, clip, lanes, s % kStages);
                }
                publish(s);
            }
        } else {
            const uint32_t base = smem_u32(S.tab) * 0x10001u;
            uint32_t up[15];  // the upper cell row's sums
#pragma unroll
            for (int t = 0; t < 15; ++t) up[t] = 0u;
            for (uint32_t s = 0; ok; ++s) {
                if (!(ok = warp_wait(&S.cfull[s % kSlots], (s / kSlots) & 1u))) break;
                const uint32_t kind = S.meta[s % kMeta][g].flags & 3u;
                if (kind == 3u) break;
                uint32_t h[15];
                lbp_row(S.slot[s % kSlots].lbp[g], lane, h);
                __syncwarp();
                if (lane == 0) arrive(&S.cempty[s % kSlots]);
                if (!(ok = stage_free(s))) break;
                if (kind == 2u) {
                    // words 0, 1-2, 3-6, 7-10, 11-14: stored as they are ready, so that few
                    // registers are live and many table reads in flight
                    tc_fence_after();
                    const uint32_t a = lanes + a_hi(s % kStages), b = lanes + a_lo(s % kStages, 1),
                                   c = lanes + a_lo(s % kStages, 2);
                    uint32_t hi[8], lo[8];
#pragma unroll
                    for (int w = 0; w < 3; ++w) lbp_word(base, up[w], h[w], hi + 2 * w, lo + 2 * w);
                    tst2(a + 18, hi);
                    tst4(a + 20, hi + 2);
                    tst2(b + 2, lo);
                    tst4(b + 4, lo + 2);
#pragma unroll
                    for (int w = 0; w < 4; ++w) lbp_word(base, up[3 + w], h[3 + w], hi + 2 * w, lo + 2 * w);
                    tst8(a + 24, hi);
                    tst8(b + 8, lo);
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
#pragma unroll
                        for (int w = 0; w < 4; ++w)
                            lbp_word(base, up[7 + 4 * q + w], h[7 + 4 * q + w], hi + 2 * w, lo + 2 * w);
                        tst8(a + 32 + 8 * q, hi);
                        tst8(c + 8 * q, lo);
                    }
                }
#pragma unroll
                for (int w = 0; w < 15; ++w) up[w] = h[w];
                publish(s);
            }
        }
    } else if (warp < 12) {
        // ---- epilogue of group g
        const int g = warp - 8;
        float acc[kWinBH];  // running scores of window rows r - i (an item's first rows start afresh)
#pragma unroll
        for (int i = 0; i < kWinBH; ++i) acc[i] = 0.f;
        for (uint32_t s = 0;; ++s) {
            if (!warp_wait(&S.mready[s % kMeta], (s / kMeta) & 1u)) break;
            const StepMeta m = S.meta[s % kMeta][g];
            const uint32_t kind = m.flags & 3u;
            if (kind == 3u) break;
            if (!warp_wait(&S.dfull[s & 1], (s >> 1) & 1u)) break;
            if (kind != 2u) {
                if (lane == 0) arrive(&S.dempty[s & 1]);
                continue;
            }
            tc_fence_after();
            const uint32_t t0 = tmem + ((uint32_t)(32 * g) << 16) + (s & 1) * 128;
            // Columns from the last template row up, so that acc[i] = acc[i - 1] + the terms
            // of row i moves the running scores on by one row without copies. The 7 terms of
            // a row are added in order of j; rows i, i + 1 (i odd) are packed.
            // The next 16 columns load while the current ones are added (three in flight fit
            // the 128 registers that 14 warps leave a thread).
            float v[7][16];
            auto term = [&](int i, int j) {
                const int n = i * kWinBW + j;
                return j ? __shfl_down_sync(0xffffffffu, v[n >> 4][n & 15], j) : v[n >> 4][n & 15];
            };
            auto rows = [&](int i) {  // rows i, i - 1
                f32x2 t = pack2(acc[i - 2] + term(i - 1, 0), acc[i - 1] + term(i, 0));
#pragma unroll
                for (int j = 1; j < kWinBW; ++j) t = add2(t, pack2(term(i - 1, j), term(i, j)));
                unpack2(t, acc[i - 1], acc[i]);
            };
            PD_LD_X16(t0 + 96, v[6]);
            PD_LD_X16(t0 + 80, v[5]);
            PD_WAIT_X16(v[6]);
            PD_WAIT_X16(v[5]);
            PD_LD_X16(t0 + 64, v[4]);
            rows(14);
            PD_WAIT_X16(v[4]);
            PD_LD_X16(t0 + 48, v[3]);
            rows(12);
            PD_WAIT_X16(v[3]);
            PD_LD_X16(t0 + 32, v[2]);
            rows(10);
            rows(8);
            PD_WAIT_X16(v[2]);
            PD_LD_X16(t0 + 16, v[1]);
            rows(6);
            PD_WAIT_X16(v[1]);
            PD_LD_X16(t0, v[0]);
            rows(4);
            PD_WAIT_X16(v[0]);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive(&S.dempty[s & 1]);  // the accumulators may be overwritten
            rows(2);
            acc[0] = bias;
#pragma unroll
            for (int j = 0; j < kWinBW; ++j) acc[0] += term(0, j);
            if ((m.flags & 4u) && lane < (int)(m.flags >> 8))
                scores[m.out + lane] = (m.keep >> lane) & 1u ? acc[kWinBH - 1] : -INFINITY;
        }
    } else if (warp == 12) {
        // ---- MMA issue. The whole warp walks the loop and one elected lane issues: the
        // loop's values are uniform, so each MMA finds its operands where it reads them
        // (a loop of lane 0 alone took 8 us longer for 64 x 1242x375 frames).
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const uint32_t b_base = smem_u32(S.b);
        bool ok = warp_wait(&S.bfull, 0);
        for (uint32_t s = 0; ok; ++s) {
            const uint32_t st = s % kStages;
            if (!warp_wait(&S.mready[s % kMeta], (s / kMeta) & 1u)) break;
            if (__any_sync(0xffffffffu, (S.meta[s % kMeta][0].flags & 3u) == 3u)) break;
            if (!warp_wait(&S.afull[st], (s / kStages) & 1u)) break;
            if (s >= 2 && !warp_wait(&S.dempty[s & 1], ((s >> 1) - 1) & 1u)) break;
            tc_fence_after();
            const uint32_t d = tm + (s & 1) * 128;
            const uint32_t ah = tm + a_hi(st);  // 8 columns per K step
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < 6; ++k) umma_ts(d, ah + 8 * k, umma_desc(b_base + 256 * k), k > 0);
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    umma_ts(d, tm + a_lo(st, k / 2) + 8 * (k & 1), umma_desc(b_base + 256 * k), 1);
#pragma unroll
                for (int k = 0; k < 6; ++k) umma_ts(d, ah + 8 * k, umma_desc(b_base + 12 * 128 + 256 * k), 1);
                umma_commit(&S.aempty[st]);
                umma_commit(&S.dfull[s & 1]);
            }
            __syncwarp();
            committed = s + 1;
        }
    } else {
        // ---- items and cell rows; lane g < 4 serves group g. A group draws its next item when
        // it needs it: the ring of slots covers the chain of loads, and a ticket drawn ahead
        // holds an item back from groups that are free (8 x 1920x1080 sparse: 191 us with the
        // ticket drawn when the item before it starts, 172 so).
        const bool sparse = c_flag != nullptr;
        const bool mine = lane < kGroups;
        bool more = mine, drawn = true;
        int ticket = (int)blockIdx.x + lane * (int)gridDim.x;  // the first items by place, the next from the queue
        // the item being walked
        bool active = false;
        const CUtensorMap *hm = &hog_map, *lm = &lbp_map;
        int wx0 = 0, ncols = 0, wy0 = 0, n_rows = 0, cols = 0, cell_row = 0, citem0 = 0, ctx = 0;
        int r = 0, r0 = 0, r_end = -1;  // next cell row, first and last one of the run
        bool first = false;
        int64_t score_off = 0;
        unsigned long long walk = 0;  // sparse: cell rows of the later runs
        auto next_run = [&]() {
            if (!walk) return false;
            const int a = __ffsll((long long)walk) - 1;
            const unsigned long long after = ~(walk >> a);  // its lowest bit ends the run
            const int len = after ? __ffsll((long long)after) - 1 : 64 - a;
            walk = a + len < 64 ? walk >> (a + len) << (a + len) : 0ull;
            r = r0 = wy0 + a;
            r_end = r + len - 1;
            first = true;
            return true;
        };
        // Sparse, whole warp: the scored windows of group g's item, and the cell rows they
        // need (a window row needs 16 of them).
        auto prepare = [&](int g) {
            const int y0 = __shfl_sync(0xffffffffu, wy0, g), x0 = __shfl_sync(0xffffffffu, wx0, g);
            const int n = __shfl_sync(0xffffffffu, n_rows, g), nc = __shfl_sync(0xffffffffu, ncols, g);
            const int nx = __shfl_sync(0xffffffffu, ctx, g);
            // lane = window column: a window lies in one or two cell tiles across; the
            // ballot of tile row t stays with lane t
            const int ty0 = y0 / kCellTH, nt = (y0 + n - 1 + kWinBH) / kCellTH - ty0 + 1;
            const int wx = x0 + lane;
            const int cl = lane < nc ? wx / kCellTW : 0, cr = lane < nc ? (wx + kWinBW) / kCellTW : 0;
            const uint32_t *flags = c_flag + __shfl_sync(0xffffffffu, citem0, g) + ty0 * nx;
            uint32_t f[kTileRows][2];
#pragma unroll
            for (int t = 0; t < kTileRows; ++t) {
                const uint32_t *row = flags + min(t, nt - 1) * nx;
                f[t][0] = __ldg(row + cl);
                f[t][1] = __ldg(row + cr);
            }
            uint32_t bits = 0;
#pragma unroll
            for (int t = 0; t < kTileRows; ++t) {
                const uint32_t b = __ballot_sync(0xffffffffu, lane < nc && f[t][0] && f[t][1]);
                if (lane == t) bits = b;
            }
            // lane = window row: its 16 cell rows lie in two or three tile rows
            unsigned long long kept = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int row = 32 * h + lane, y = y0 + min(row, n - 1);
                const int a0 = y / kCellTH - ty0, a1 = (y + kWinBH) / kCellTH - ty0;
                const uint32_t k = __shfl_sync(0xffffffffu, bits, a0) & __shfl_sync(0xffffffffu, bits, a0 + 1) &
                                   __shfl_sync(0xffffffffu, bits, a1);
                if (row < n) S.keep[g][row] = k;
                kept |= (unsigned long long)__ballot_sync(0xffffffffu, row < n && k) << (32 * h);
            }
            __syncwarp();
            if (lane == g) {
                kept |= kept << 1;  // 16 wide: kTcSparseRows + 15 bits
                kept |= kept << 2;
                kept |= kept << 4;
                kept |= kept << 8;
                walk = kept;
                active = next_run();
            }
        };
        for (uint32_t s = 0;; ++s) {
            // groups whose item (or run) is done take the next
            if (active && r > r_end) active = sparse && next_run();
            for (;;) {
                const bool want = !active && more;
                if (!__any_sync(0xffffffffu, want)) break;
                if (want) {
                    if (!drawn) ticket = kGroups * (int)gridDim.x + atomicAdd(queue, 1);
                    drawn = false;
                    more = ticket < n_items;
                }
                if (want && more) {
                    const TcItem it = items[ticket];
                    const LevelDesc &L = levels[it.level];
                    wx0 = it.wx0;
                    wy0 = it.wy0;
                    n_rows = it.wy1 - it.wy0;
                    cols = L.cols;
                    ncols = min(kTcStrip, cols - wx0);
                    cell_row = L.cell_row;
                    citem0 = L.citem0;
                    ctx = L.ctx;
                    score_off = L.score_off;
                    if (level_maps) {
                        hm = level_maps + 2 * L.tc_map;
                        lm = hm + 1;
                    }
                    r = r0 = wy0;
                    r_end = it.wy1 - 1 + kWinBH;
                    first = active = true;
                }
                if (!sparse) break;
                for (unsigned left = __ballot_sync(0xffffffffu, want && more); left; left &= left - 1u)
                    prepare(__ffs((int)left) - 1);
            }
            const uint32_t slot = s % kSlots;
            if (s >= kSlots && !warp_wait(&S.cempty[slot], (s / kSlots - 1) & 1u)) break;
            const unsigned act = __ballot_sync(0xffffffffu, active);
            if (mine) {
                StepMeta m{};
                if (!act) m.flags = 3u;
                if (active) {
                    const int wy = r - kWinBH;  // the window row that this cell row completes
                    const bool store = wy >= r0;
                    m.flags = (first ? 1u : 2u) | (store ? 4u : 0u) | ((uint32_t)(wx0 & 3) << 4) | ((uint32_t)ncols << 8);
                    m.keep = sparse && store ? S.keep[lane][wy - wy0] : 0xffffffffu;
                    m.out = score_off + (int64_t)wy * cols + wx0;
                }
                S.meta[s % kMeta][lane] = m;
            }
            __syncwarp();
            if (lane == 0) {
                arrive_tx(&S.cfull[slot], __popc(act) * (uint32_t)(HP * kHogX * 4 + kLbpX * 64));
                arrive(&S.mready[s % kMeta]);
            }
            __syncwarp();
            if (!act) break;
            if (active) {
                Slot &sl = S.slot[slot];
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                tma_3d(sl.hog[lane], hm, &S.cfull[slot], wx0 & ~3, cell_row + r, 0);
                tma_3d(sl.lbp[lane], lm, &S.cfull[slot], 0, wx0, cell_row + r);
                first = false;
                ++r;
            }
            loads = s + 1;
        }
    }

    __syncthreads();
    if (S.failed) {
        // drain this CTA's copies and MMAs (bounded) before the tensor memory is
        // freed: the constants, the last load of every slot, the last commit
        if (warp == 13 && lane == 0) {
            drain_wait(&S.bfull, 0);
            for (uint32_t i = loads > kSlots ? loads - kSlots : 0u; i < loads; ++i)
                drain_wait(&S.cfull[i % kSlots], (i / kSlots) & 1u);
        }
        if (warp == 12 && lane == 0 && committed > 0)
            drain_wait(&S.dfull[(committed - 1) & 1], ((committed - 1) >> 1) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

#undef PD_LD_X16
#undef PD_WAIT_X16

// LBP count planes [59][rows][pitch] -> 64 bytes per cell, [rows][width][64]
// (bins 59..63 zero): one thread per 16 bins of a cell, a block per row (or
// every kRowBlocks-th: a grid has no more). For callers' planes;
// the detector's own cells are written that way.
constexpr int kRowBlocks = 65535;
__global__ void __launch_bounds__(128) k_lbp_cells(const uint8_t *__restrict__ planes, int64_t plane, int pitch,
                                                   int width, int rows, uint8_t *__restrict__ out) {
    const int x = blockIdx.x * 32 + (threadIdx.x & 31), k = threadIdx.x >> 5;
    if (x >= width) return;
    for (int y = blockIdx.y; y < rows; y += gridDim.y) {
        const uint8_t *src = planes + (int64_t)y * pitch + x;
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            w[u] = 0u;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int t = 16 * k + 4 * u + b;
                if (t < kLbpBins) w[u] |= (uint32_t)__ldg(src + t * plane) << (8 * b);
            }
        }
        reinterpret_cast<uint4 *>(out)[((int64_t)y * width + x) * 4 + k] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

}  // namespace

cudaError_t init_svm_tc() {
    cudaError_t e = cudaFuncSetAttribute(k_svm_tc<kHogBins>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(TcSmemT<kHogBins>));
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(k_svm_tc<4 * kHogBins>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)sizeof(TcSmemT<4 * kHogBins>));
}

void build_tc_consts(const float *wt, unsigned char *out) {
    std::memset(out, 0, kTcConstBytes);
    // B operand: template position n = 7 i + j (rows), feature t (K); high
    // parts in chunks 0..11, low parts in chunks 12..23
    for (int n = 0; n < kWinBH * kWinBW; ++n)
        for (int t = 0; t < kFeat; ++t) {
            const float w = wt[((size_t)t * kWinBH + n / kWinBW) * kWPad + n % kWinBW];
            const __nv_bfloat16 h = __float2bfloat16_rn(w);
            const __nv_bfloat16 l = __float2bfloat16_rn(w - __bfloat162float(h));
            const size_t off = (size_t)(n >> 3) * kSBO + (t >> 3) * 128 + (n & 7) * 16 + (t & 7) * 2;
            std::memcpy(out + off, &h, 2);
            std::memcpy(out + off + 12 * 128, &l, 2);
        }
    for (int s = 0; s <= 256; ++s) {
        const float f = sqrtf((float)s * (1.0f / 256.0f));
        const __nv_bfloat16 h = __float2bfloat16_rn(f);
        const __nv_bfloat16 l = __float2bfloat16_rn(f - __bfloat162float(h));
        std::memcpy(out + kBBytes + 4 * s, &h, 2);
        std::memcpy(out + kBBytes + 4 * s + 2, &l, 2);
    }
}

int encode_tc_maps(CUtensorMap *hog_map, CUtensorMap *lbp_map, const float *hog, int64_t hog_pitch, int64_t hog_plane,
                   int hog_planes, const uint8_t *lbp, int64_t lbp_pitch, int64_t rows, int64_t width) {
    // 36 cells of one row of every HOG plane; 33 cells x 64 bytes of one row
    if (encode_plane_map(hog_map, const_cast<float *>(hog), CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, hog_pitch, rows,
                         hog_planes, hog_plane, kHogX, 1, hog_planes, width) != PD_OK)
        return PD_ECUDA;
    return encode_cell_map(lbp_map, const_cast<uint8_t *>(lbp), lbp_pitch, rows, width, kLbpX);
}

cudaError_t launch_lbp_cells(cudaStream_t s, const uint8_t *planes, int64_t plane, int pitch, int width, int rows,
                             uint8_t *out) {
    if (width <= 0 || rows <= 0) return cudaSuccess;
    k_lbp_cells<<<dim3((width + 31) / 32, rows < kRowBlocks ? rows : kRowBlocks), 128, 0, s>>>(planes, plane, pitch,
                                                                                              width, rows, out);
    return cudaGetLastError();
}

cudaError_t launch_svm_tc(cudaStream_t s, const CUtensorMap &hog_map, const CUtensorMap &lbp_map,
                          const LevelDesc *d_levels, const TcItem *d_items, int n_items, int *d_queue, int grid,
                          const unsigned char *d_consts, float bias, float clip, float *scores,
                          const uint32_t *c_flag, unsigned *d_err, int hog_planes, const CUtensorMap *level_maps) {
    if (n_items <= 0) return cudaSuccess;
    if ((reinterpret_cast<uintptr_t>(level_maps) & 63) || (reinterpret_cast<uintptr_t>(d_consts) & 15))
        return cudaErrorInvalidValue;
    grid = grid < n_items ? grid : n_items;
    if (hog_planes == 4 * kHogBins)
        k_svm_tc<4 * kHogBins><<<grid, kThreads, sizeof(TcSmemT<4 * kHogBins>), s>>>(
            hog_map, lbp_map, d_levels, d_items, n_items, d_queue, d_consts, bias, clip, scores, c_flag, d_err,
            level_maps);
    else
        k_svm_tc<kHogBins><<<grid, kThreads, sizeof(TcSmemT<kHogBins>), s>>>(
            hog_map, lbp_map, d_levels, d_items, n_items, d_queue, d_consts, bias, clip, scores, c_flag, d_err,
            level_maps);
    return cudaGetLastError();
}

}  // namespace pd
