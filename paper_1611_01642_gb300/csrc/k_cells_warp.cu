// K2 + K3 -- HOG and uniform-LBP cell histograms of the pyramid levels
// (Section 4.2, Algorithms 1-2; Section 4.3, Algorithms 4-5), one warp per
// strip of cells, four pixel columns per lane.
//
// Persistent warps (4 per CTA, independent of each other) take strips from a
// queue, tallest first. A strip is 15 cells wide and up to kStripTiles cell
// tiles (8 cell rows each) tall; the planner takes shorter strips, down to 2
// cell rows, when a batch is small. Its warp walks the 128 pixel columns
// [8 cx0 - 4, 8 cx0 + 124) (the strip and the 4 columns on each side whose
// HOG votes still reach it): lane t owns columns 8 cx0 - 4 + 4t .. + 3, which
// lie in one cell (strip cell (t - 1) / 2; lanes 0 and 31 lie in the
// neighbouring strips). The warp walks the pixel rows from the top in bands
// of 8: band k covers the rows [8 (cy0 + k) - 4, 8 (cy0 + k) + 4), which vote
// only into cell rows cy0 + k - 1 and cy0 + k, so after band k cell row
// cy0 + k - 1 is final and the warp writes it out. A tall strip walks the
// 4-row vertical halo of a band once per strip.
//
// Per row a lane loads three aligned 32-bit words of the level row (its own
// 4 bytes and its neighbours'; byte loads clamped to the level at its left
// and right edges), one row pair ahead, and keeps the rows above and below
// in registers. For its 4 pixels:
//  * LBP (Algorithm 1) on packed bytes. For bytes n, c: n >= c exactly when
//    the subtraction n - c does not borrow out of bit 7, which is the
//    majority of (n7, not c7, bit 7 of (n | 0x80) - (c & 0x7f)); one
//    subtraction and one 3-input logic operation compare 4 pixels with one
//    neighbour. The 8 comparisons of a lane's 32 pixels of a cell (4 columns x
//    8 rows) are 8 bit planes, shifted in row by row, and a uniform code is
//    one run of ones around the circle: the pixels of a code are three planes
//    ANDed and their number a population count (Algorithm 2 without a histogram
//    in memory).
//    Counting in shared memory instead (a code -> counter table and an atomic
//    per pixel) took a third of the kernel's shared-memory wavefronts and kept
//    that pipe 79% busy (now 57%): 0.961 -> 0.887 ms per 64 x 1242x375 frames.
//  * HOG (Algorithm 4). One byte permute and two dp2a (weights +1, -1) give
//    the central differences of two pixels; the accumulator 0x4B400000 makes
//    the 32-bit result the float 1.5 * 2^23 + g, so one multiply-add turns it
//    into g / 2 (exact). Magnitude sqrt(gx^2 + gy^2); unsigned orientation in
//    bin units (degrees / 20): the angle phi of (|gx|, |gy|) is 45 degrees +
//    atan(t) with t = (|gy| - |gx|) / (|gy| + |gx|) in [-1, 1], where an odd
//    polynomial t P(t^2) of degree 13 fitted to atan on [0, 1] (weighted
//    least squares on Chebyshev nodes, scaled to bin units; error < 1e-6
//    bin) holds; theta is phi or 180 degrees - phi as the signs of gx and gy
//    agree or not (one sign flip, no branch). The vote is linear between the
//    two nearest of the 9 bins and between the two cell rows of the band
//    (weights (7.5 - k) / 8 and (k + 0.5) / 8 for band row k), and bilinear
//    on x through the columns' weights in the epilogue.
//    floor(theta / 20deg - 0.5) comes from rounding 2 (theta - 1) to an even
//    integer by adding 3 * 2^23, where floats are spaced by 2 (a tie gives
//    the other neighbour with weight 1, the same votes); the residual e in
//    [-1, 1] gives the lower and upper bins' weights (1 - e) / 2 and
//    (1 + e) / 2 with one multiply-add each, and the float's bits are the
//    bin number plus a constant, so they index the column's vote slots
//    directly. There are 11 slots per column, slot s holding bin
//    (s - 1) mod 9 (bin -1 and bin 9 wrap), which the epilogue folds back:
//    the loop needs no wrap logic. Two pixels share an instruction wherever
//    both take the same step (fma.rn.f32x2 rounds each half as the scalar
//    does): 11 fewer instructions per pixel, 0.887 -> 0.828 ms; shared-memory
//    addresses of the slots as integers, 0.828 -> 0.810.
//    The slots of lane t's 4 columns sit at 4t + (j ^ ((t >> 3) & 3)), so
//    that a warp's data-dependent scatter hits 32 distinct banks and the
//    epilogue reads them with one 16-byte load.
// Rows outside the cell grid are whole halves of the level's first and last
// bands and are not walked (0.810 -> 0.785 ms). Each lane of a cell counts its
// own 32 pixels of all bins and swaps half of them with the other (both lanes'
// pixels for half of the bins took 80 instructions more per cell row: 0.785 ->
// 0.766 ms). What bounds the kernel:
// issue (72% of cycles, 75 thread instructions per pixel) with 16 warps per SM
// at 125 registers; 20 warps at 96 registers measured slower (0.875 against
// 0.828 ms), all of a row's slot loads before its stores no faster.
// HOG epilogue of cell row r: each lane forms, per bin, the weighted sums of
// its 4 columns for its own cell and for the neighbouring cell they reach;
// three shuffles add the 4 lanes that reach a cell (fixed order:
// deterministic). The LBP counts of a cell go out as 64 bytes, two 16-byte
// stores from each of its two lanes, or, for callers that ask for planes,
// bin-plane by bin-plane. At the top and bottom of a
// level the votes of the clamped cell row (Algorithm 5's interpolation
// clamped into the grid) are added into the first and last row before they
// are written. The result does not depend on the strip height: every cell
// row sums its votes in the same order.
//
// Per-block HOG (kFeatHogBlock, Algorithm 5 read per 16x16 block): a block's
// 4 cell histograms take only the block's own pixels, with the votes of the
// shared grid left unclamped (a vote towards a cell outside the block is
// dropped). Cell (cy, cx) sits at one of 4 places q = 2a + b of the blocks
// that contain it (a = 0: it is the block's top cell, so the block spans
// pixel rows [8cy, 8cy + 16); a = 1: rows [8cy - 8, 8cy + 8); b likewise on
// x), and the kernel writes its 4 restricted histograms Q_q to planes
// 9q + bin. Block (by, bx) is then [Q_0(by, bx), Q_1(by, bx+1),
// Q_2(by+1, bx), Q_3(by+1, bx+1)]. The walk and its votes are the shared
// grid's: of the rows that vote into cell row t, A = [8t - 4, 8t),
// B = [8t, 8t + 8) and C = [8t + 8, 8t + 12), a = 1 takes A and B, a = 0 takes
// B and C, and the ends of A, B and C are ends of half bands. So the slots are
// summed over the columns three times per cell row: after A (set aside, slots
// cleared), after B (with A: a = 1) and after C (a = 0); of a cell's 16 columns
// b drops the first or the last 4, one b per lane of the cell. Against a CTA
// of 128 threads per 15 x 8-cell tile, one column per thread, which voted
// three times per pixel and counted LBP by shared-memory atomics: 583 -> 266 us
// per 16 x 1242x375 frames (the shared grid: about 200). What bounds it: the
// shared-memory pipe, where the column sums and the second clear add about
// 170 wavefronts per cell row to the walk's 370.
//
// Sparse path: c_flag marks the 15 x 8-cell tiles to compute; a band is
// walked when one of its two cell rows lies in a marked tile, and a cell
// row is written when its tile is marked.
#include <algorithm>
#include <type_traits>
#include <utility>

#include "f32x2.cuh"
#include "pd_internal.h"

namespace pd {
namespace {

constexpr int kWarps = 4;                        // strips per CTA
constexpr int kSCols = 8 * kCellTW + 8;          // 128 pixel columns walked per strip
static_assert(kSCols == 4 * 32, "four pixel columns per lane");
constexpr int kSlots = kHogBins + 2;             // vote slots per column (bins -1 .. 9)
constexpr int kRingStride = kSlots * kSCols;     // floats per open cell row
constexpr uint32_t kHi = 0x80808080u;
constexpr float kMagic = 12582912.0f;            // 1.5 * 2^23: dp2a accumulator
constexpr uint32_t kMagicBits = 0x4B400000u;
constexpr float kMagic2 = 25165824.0f;           // 3 * 2^23 (spacing 2): rounds to even integers
constexpr uint32_t kMagic2Bits = 0x4BC00000u;

template <bool PB>
struct WarpSmem {
    float R[2 * kRingStride];       // HOG vote slots of the 2 open cell rows
};
template <>
struct WarpSmem<true> {
    float R[2 * kRingStride];
    float top[kHogBins][32];        // per-block HOG: per lane, the votes of the 4 pixel rows above the open cell row
};
template <bool PB>
struct StripSmem {
    WarpSmem<PB> w[kWarps];
};

struct Row {
    uint32_t l, c, r;  // bytes x - 1 .. x + 2, x .. x + 3, x + 1 .. x + 4 of a lane's columns
};

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return min(max(v, lo), hi); }

// c + b.byte0 - b.byte1 (lo) / c + b.byte2 - b.byte3 (hi), bytes unsigned
__device__ __forceinline__ int dp2a_diff_lo(uint32_t b, int c) {
    int d;
    asm("dp2a.lo.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(0xFFFF0001u), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ int dp2a_diff_hi(uint32_t b, int c) {
    int d;
    asm("dp2a.hi.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(0xFFFF0001u), "r"(b), "r"(c));
    return d;
}

// Operands here are 0 or >= 1e-30 (never subnormal), so the flush-to-zero
// forms are exact.
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// -2 atan(z) * 9/pi / z as a polynomial in s = z^2 (|z| <= 1), two values at
// a time: the fitted coefficients scaled to 20-degree bins, doubled and negated
// (exact: every step of the evaluation scales by -2). PREC: one degree more (15,
// fitted to the least largest error), 3.3e-7 bin instead of 8.9e-7 in float32;
// the histograms' error is 1.1e-7 of their norm with it and 2.9e-7 without. The
// scores' error, most of it from K4's split operands (5.2e-7 on exact histograms),
// is 6.8e-7 of theirs (16 x 1242x375 frames); with the kernel before, whose
// histograms were off by 2.8e-7 the other way, it was 6.1e-7.
template <bool PREC>
__device__ __forceinline__ f32x2 atan_bins2_poly(f32x2 s) {
    if constexpr (PREC) {
        f32x2 p = dup2(-2.0f * -0.01161547377705574f);
        p = fma2(p, s, dup2(-2.0f * 0.06263275444507599f));
        p = fma2(p, s, dup2(-2.0f * -0.16017703711986542f));
        p = fma2(p, s, dup2(-2.0f * 0.2762286365032196f));
        p = fma2(p, s, dup2(-2.0f * -0.39845290780067444f));
        p = fma2(p, s, dup2(-2.0f * 0.571427047252655f));
        p = fma2(p, s, dup2(-2.0f * -0.9548301696777344f));
        return fma2(p, s, dup2(-2.0f * 2.8647871017456055f));
    }
    f32x2 p = dup2(-2.0f * 0.019514326006174088f);
    p = fma2(p, s, dup2(-2.0f * -0.09626893699169159f));
    p = fma2(p, s, dup2(-2.0f * 0.22810496389865875f));
    p = fma2(p, s, dup2(-2.0f * -0.3791072964668274f));
    p = fma2(p, s, dup2(-2.0f * 0.5674521327018738f));
    p = fma2(p, s, dup2(-2.0f * -0.9544723033905029f));
    return fma2(p, s, dup2(-2.0f * 2.8647778034210205f));
}

// A vote slot at a shared-memory address (the compiler's own indexing spends a
// shift per access). Volatile and clobbering: the epilogue reads the slots
// through ordinary pointers.
constexpr int kSlotBytes = 4 * kSCols;
template <int OFF>
__device__ __forceinline__ float lds(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1 + %2];" : "=f"(v) : "r"(a), "n"(OFF) : "memory");
    return v;
}
template <int OFF>
__device__ __forceinline__ void sts(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0 + %1], %2;" ::"r"(a), "n"(OFF), "f"(v) : "memory");
}

template <class F, int... I>
__device__ __forceinline__ void static_for(F &&f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}

// 4 pixels' n >= c comparisons, as bit 7 of each byte (the other bits are not
// meaningful); cn = ~c.
__device__ __forceinline__ uint32_t ge4(uint32_t n, uint32_t c_lo, uint32_t cn) {
    const uint32_t t = (n | kHi) - c_lo;
    return (n & cn) | (t & (n | cn));  // majority of n, not c, t
}

// Uniform codes in ascending order (at most two changes around the circle): code of
// bin b, 0 .. 57. All but 0 and 255 are one run of ones, from run_start over
// run_length positions around the circle.
__host__ __device__ constexpr int uniform_code(int b) {
    int i = -1;
    for (int c = 0; c < 256; ++c) {
        int changes = 0;
        for (int k = 0; k < 8; ++k) changes += ((c >> k) & 1) != ((c >> ((k + 1) & 7)) & 1);
        if (changes <= 2 && ++i == b) return c;
    }
    return -1;
}
__host__ __device__ constexpr int run_start(int c) {
    for (int k = 0; k < 8; ++k)
        if (((c >> k) & 1) && !((c >> ((k + 7) & 7)) & 1)) return k;
    return -1;
}
__host__ __device__ constexpr int run_length(int c) {
    int n = 0;
    for (int k = 0; k < 8; ++k) n += (c >> k) & 1;
    return n;
}
static_assert(uniform_code(0) == 0 && uniform_code(57) == 255 && uniform_code(58) == -1, "58 uniform codes");

// The comparison planes of 32 pixels (bit k of their codes in x[k]) -> pixels
// whose code is one run starting at s (run[s]) or has two or more runs (many: not
// uniform). Codes 0 and 255 have none.
__device__ __forceinline__ void lbp_runs(const uint32_t (&x)[8], uint32_t (&run)[8], uint32_t &many) {
    uint32_t r[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) r[k] = x[k] & ~x[(k + 7) & 7];  // a run starts at k
    const uint32_t s1 = r[0] ^ r[1] ^ r[2], c1 = (r[0] & r[1]) | (r[2] & (r[0] | r[1]));
    const uint32_t s2 = r[3] ^ r[4] ^ r[5], c2 = (r[3] & r[4]) | (r[5] & (r[3] | r[4]));
    const uint32_t s3 = r[6] ^ r[7], c3 = r[6] & r[7];
    const uint32_t c4 = (s1 & s2) | (s3 & (s1 | s2));
    many = (c1 | c2 | c3) | c4;
#pragma unroll
    for (int k = 0; k < 8; ++k) run[k] = r[k] & ~many;
}

template <int FEAT, bool CELLS>  // CELLS: cell-major LBP counts
__global__ void __launch_bounds__(kWarps * 32, 4)
    k_cells_warp(const LevelDesc *__restrict__ levels, const uint8_t *__restrict__ pyr, CellAtlas atlas,
                 const StripItem *__restrict__ items, int n_items, int *__restrict__ queue,
                 const uint32_t *__restrict__ c_flag) {
    constexpr bool kHog = (FEAT & kFeatHog) != 0, kLbp = (FEAT & kFeatLbp) != 0;
    constexpr bool kPb = (FEAT & kFeatHogBlock) != 0;  // per-block HOG
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StripSmem<kPb> &S = *reinterpret_cast<StripSmem<kPb> *>(smem_raw);
    const int lane = threadIdx.x & 31;
    WarpSmem<kPb> &Wm = S.w[threadIdx.x >> 5];
    // persistent warps: each takes the next strip (tallest first) until none is left
    for (;;) {
        int item = lane == 0 ? atomicAdd(queue, 1) : 0;
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= n_items) return;
        const StripItem it = items[item];
        const LevelDesc L = levels[it.level];
        const uint8_t *img = pyr + L.img_off;
        const int pitch = L.img_pitch, Wk = L.Wk, Hk = L.Hk, Wc = L.Wc, Hc = L.Hc;
        const int cx0 = it.cx0, cy0 = it.cy0, nb = it.cy1 - it.cy0;
        const int tx = cx0 / kCellTW;
        const int x = 8 * cx0 - 4 + 4 * lane;  // first pixel column of this lane
        const bool fast = (((reinterpret_cast<uintptr_t>(img) | (uintptr_t)pitch) & 3u) == 0) && x >= 4 &&
                          x + 8 <= Wk;

        if (kHog)
            for (int i = lane; i < 2 * kRingStride / 4; i += 32)
                reinterpret_cast<float4 *>(Wm.R)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (kPb) {
#pragma unroll
            for (int h = 0; h < kHogBins; ++h) Wm.top[h][lane] = 0.f;  // a level's first cell row has no rows above it
        }
        uint32_t plane[8];  // LBP comparisons of the last 8 rows: plane k, byte = column, bit = row
#pragma unroll
        for (int k = 0; k < 8; ++k) plane[k] = 0u;

        // ---- lane constants
        const int sw = (lane >> 3) & 3;
        // shared-memory address of slot 0 of pixel j's column, less the bias of the rounded angle's bits
        uint32_t vb[4];
        const uint32_t slots = (uint32_t)__cvta_generic_to_shared(Wm.R);
#pragma unroll
        for (int j = 0; j < 4; ++j) vb[j] = slots + 4u * (uint32_t)(4 * lane + (j ^ sw)) + 512u - kMagic2Bits * 512u;
        // epilogue x-weights by slot position p (column j = p ^ sw): own cell, neighbour cell
        float wo[4], wn[4];
        {
            const int own = cx0 + ((lane - 1) >> 1);
            const int nbr = own + ((lane & 1) ? -1 : 1);
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const int xc = x + (p ^ sw);
                float a = 0.f, b = 0.f;
                if (xc >= 0 && xc < 8 * Wc) {
                    const float ux = ((float)xc - 3.5f) * 0.125f;
                    const float fx = floorf(ux);
                    const float w1 = ux - fx, w0 = 1.f - w1;
                    const int c0 = kPb ? (int)fx : clampi((int)fx, 0, Wc - 1);
                    const int c1 = kPb ? (int)fx + 1 : clampi((int)fx + 1, 0, Wc - 1);
                    a = (c0 == own ? w0 : 0.f) + (c1 == own ? w1 : 0.f);
                    b = (c0 == nbr ? w0 : 0.f) + (c1 == nbr ? w1 : 0.f);
                }
                wo[p] = a;
                wn[p] = b;
            }
        }
        __syncwarp();

        // ---- rows
        auto fetch = [&](int y, uint32_t (&w)[3]) {
            const uint8_t *row = img + (size_t)clampi(y, 0, Hk - 1) * pitch;
            if (fast) {
                const uint32_t *p = reinterpret_cast<const uint32_t *>(row + x);
                w[0] = __ldg(p - 1);
                w[1] = __ldg(p);
                w[2] = __ldg(p + 1);
            } else {
                uint32_t v[6];
#pragma unroll
                for (int i = 0; i < 6; ++i) v[i] = __ldg(row + clampi(x - 1 + i, 0, Wk - 1));
                w[0] = v[0] << 24;
                w[1] = v[1] | (v[2] << 8) | (v[3] << 16) | (v[4] << 24);
                w[2] = v[5];
            }
        };
        auto mkrow = [](const uint32_t (&w)[3]) {
            Row r;
            r.l = __funnelshift_r(w[0], w[1], 24);
            r.c = w[1];
            r.r = __funnelshift_r(w[1], w[2], 8);
            return r;
        };
        auto need = [&](int r) -> bool {  // strip cell row r is computed
            if (r < 0 || r >= nb) return false;
            return !c_flag || c_flag[L.citem0 + ((cy0 + r) / kCellTH) * L.ctx + tx] != 0u;
        };

        // ---- one pixel row (rows a / b / c = y - 1, y, y + 1): HOG votes with
        // weights fa, fb into the vote slots at byte addresses va[j] (cell row
        // band - 1; the rounded angle's bits are added) and va[j] + dB (cell row
        // band); the LBP comparisons are shifted into the lane's bit planes
        auto pixel_row = [&](const Row &ra, const Row &rb, const Row &rc, float fa, float fb, const uint32_t (&va)[4],
                             uint32_t dB) {
            if (kHog) {
                const f32x2 wa = dup2(fa), wb = dup2(fb);
                const uint32_t P01 = __byte_perm(rb.r, rb.l, 0x5140), P23 = __byte_perm(rb.r, rb.l, 0x7362);
                const uint32_t Q01 = __byte_perm(rc.c, ra.c, 0x5140), Q23 = __byte_perm(rc.c, ra.c, 0x7362);
                const int gxb[4] = {dp2a_diff_lo(P01, (int)kMagicBits), dp2a_diff_hi(P01, (int)kMagicBits),
                                    dp2a_diff_lo(P23, (int)kMagicBits), dp2a_diff_hi(P23, (int)kMagicBits)};
                const int gyb[4] = {dp2a_diff_lo(Q01, (int)kMagicBits), dp2a_diff_hi(Q01, (int)kMagicBits),
                                    dp2a_diff_lo(Q23, (int)kMagicBits), dp2a_diff_hi(Q23, (int)kMagicBits)};
#pragma unroll
                for (int j = 0; j < 4; j += 2) {  // pixels j, j + 1: packed where both take the same step
                    // half gradients, exact: (1.5 * 2^23 + g) / 2 - 0.75 * 2^23
                    const f32x2 half = dup2(0.5f), bias = dup2(-0.5f * kMagic), neg = dup2(-1.0f);
                    const f32x2 hx = fma2(pack2(__int_as_float(gxb[j]), __int_as_float(gxb[j + 1])), half, bias);
                    const f32x2 hy = fma2(pack2(__int_as_float(gyb[j]), __int_as_float(gyb[j + 1])), half, bias);
                    float x0, x1, y0, y1, q0, q1;
                    unpack2(hx, x0, x1);
                    unpack2(hy, y0, y1);
                    unpack2(fma2(hx, hx, mul2(hy, hy)), q0, q1);
                    const f32x2 hm = pack2(sqrt_approx(q0), sqrt_approx(q1));  // magnitude / 2
                    // phi = atan(ay / ax) = 45deg + atan(t), t = (ay - ax) / (ay + ax) in [-1, 1];
                    // ax + ay is 0 or >= 0.5: the 1e-30 only turns 0 / 0 into 0
                    float d0, d1;
                    unpack2(add2(pack2(fabsf(x0) + fabsf(y0), fabsf(x1) + fabsf(y1)), dup2(1e-30f)), d0, d1);
                    const f32x2 t = mul2(pack2(fabsf(y0) - fabsf(x0), fabsf(y1) - fabsf(x1)),
                                         pack2(rcp_approx(d0), rcp_approx(d1)));
                    // u = 2 (4.5 - phi) in bins, in [0, 9]
                    float u0, u1;
                    unpack2(fma2(t, atan_bins2_poly<kPb>(mul2(t, t)), dup2(4.5f)), u0, u1);
                    // theta = phi (same signs) or 9 - phi (opposite signs); the vote position is
                    // theta - 0.5, rounded below through theta - 1: p2 = 2 (theta - 1) = 7 -/+ u
                    const uint32_t f0 = ~(__float_as_uint(x0) ^ __float_as_uint(y0)) & 0x80000000u;
                    const uint32_t f1 = ~(__float_as_uint(x1) ^ __float_as_uint(y1)) & 0x80000000u;
                    const f32x2 p2 = add2(pack2(__uint_as_float(__float_as_uint(u0) ^ f0),
                                                __uint_as_float(__float_as_uint(u1) ^ f1)), dup2(7.0f));
                    const f32x2 r2 = add2(p2, dup2(kMagic2));       // 2 round(theta - 1) + 3 * 2^23
                    const f32x2 rr = add2(r2, dup2(-kMagic2));
                    const f32x2 e2 = fma2(rr, neg, p2);             // 2 (theta - 1 - round(...)), in [-1, 1]
                    const f32x2 n2 = fma2(p2, neg, rr);             // -e2
                    // slot addresses of the two pixels, in the cell rows above and below
                    const uint32_t v = (uint32_t)__float_as_int(lo2(r2)) * 512u + va[j], w = v + dB;
                    const uint32_t z = (uint32_t)__float_as_int(hi2(r2)) * 512u + va[j + 1], o = z + dB;
                    // upper / lower bin: magnitude times (1 +/- e2) / 2
                    const f32x2 mo1 = fma2(hm, e2, hm), mo0 = fma2(hm, n2, hm);
                    const f32x2 a0 = fma2(mo0, wa, pack2(lds<0>(v), lds<0>(z)));
                    const f32x2 a1 = fma2(mo1, wa, pack2(lds<kSlotBytes>(v), lds<kSlotBytes>(z)));
                    const f32x2 b0 = fma2(mo0, wb, pack2(lds<0>(w), lds<0>(o)));
                    const f32x2 b1 = fma2(mo1, wb, pack2(lds<kSlotBytes>(w), lds<kSlotBytes>(o)));
                    sts<0>(v, lo2(a0));
                    sts<0>(z, hi2(a0));
                    sts<kSlotBytes>(v, lo2(a1));
                    sts<kSlotBytes>(z, hi2(a1));
                    sts<0>(w, lo2(b0));
                    sts<0>(o, hi2(b0));
                    sts<kSlotBytes>(w, lo2(b1));
                    sts<kSlotBytes>(o, hi2(b1));
                }
            }
            if (kLbp) {
                const uint32_t clo = rb.c & ~kHi, cn = ~rb.c;
                const uint32_t nb8[8] = {ra.l, ra.c, ra.r, rb.r, rc.r, rc.c, rc.l, rb.l};
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    plane[k] = ((plane[k] >> 1) & ~kHi) | (ge4(nb8[k], clo, cn) & kHi);
            }
        };

        // ---- LBP of cell row r = band - 1 is final after the band's first 4 rows: the planes
        // hold its 8 rows (older bits are shifted out). A cell is the two lanes 2c + 1 and
        // 2c + 2, 32 pixels each: each counts its own (59 bins, a byte each), they swap
        // halves of the bins and the first writes bins 0 .. 31, the second the others.
        auto emit_lbp = [&](int band) {
            const int r = band - 1;
            if (!need(r)) return;
            const uint32_t half = (lane & 1) ^ 1u;
            uint32_t run[8], many;
            lbp_runs(plane, run, many);
            uint32_t q[16];  // counts, 4 bins per word
            static_for([&](auto B) {
                constexpr int bin = decltype(B)::value;
                uint32_t n = 0u;
                if constexpr (bin == 0) {
                    n = __popc(~((plane[0] | plane[1] | plane[2]) | (plane[3] | plane[4] | plane[5]) | (plane[6] | plane[7])));
                } else if constexpr (bin == 57) {
                    n = __popc((plane[0] & plane[1] & plane[2]) & (plane[3] & plane[4] & plane[5]) & (plane[6] & plane[7]));
                } else if constexpr (bin == 58) {
                    n = __popc(many);
                } else if constexpr (bin < 58) {
                    constexpr int s = run_start(uniform_code(bin)), e = s + run_length(uniform_code(bin));
                    n = __popc(run[s] & plane[(e - 1) & 7] & ~plane[e & 7]);
                }
                if constexpr (bin % 4 == 0) q[bin / 4] = n;
                else if constexpr (bin <= 58) q[bin / 4] += n << (8 * (bin % 4));
            }, std::make_integer_sequence<int, 64>{});
            uint32_t v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint32_t give = half ? q[i] : q[8 + i], keep = half ? q[8 + i] : q[i];
                v[i] = keep + __shfl_sync(0xffffffffu, give, ((lane - 1) ^ 1) + 1);
            }
            const int c = (lane - 1) >> 1;
            if (lane < 1 || lane > 2 * kCellTW || cx0 + c >= Wc) return;
            if (CELLS) {
                uint4 *dst = reinterpret_cast<uint4 *>(
                    atlas.lbp + ((int64_t)(L.cell_row + cy0 + r) * atlas.pitch + cx0 + c) * kLbpCellBytes + 32 * half);
                dst[0] = make_uint4(v[0], v[1], v[2], v[3]);
                dst[1] = make_uint4(v[4], v[5], v[6], v[7]);
            } else {
                const int64_t pl = atlas.lbp_plane;
                uint8_t *dst = atlas.lbp + (int64_t)(L.cell_row + cy0 + r) * atlas.pitch + cx0 + c + 32 * half * pl;
#pragma unroll
                for (int i = 0; i < 32; ++i, dst += pl)
                    if (i < 27 || !half) *dst = (uint8_t)(v[i >> 2] >> (8 * (i & 3)));
            }
        };

        // ---- HOG bin h of a cell row: the lane's columns of the slots at Rl (bin h is slot
        // h + 1; bin 0 also slot 10, bin 8 also slot 0), weighted for its own cell and for
        // the neighbouring cell they reach
        auto columns = [&](const float *Rl, int h, float &own, float &nbv) {
            float4 v = *reinterpret_cast<const float4 *>(Rl + (h + 1) * kSCols);
            if (h == 0 || h == kHogBins - 1) {
                const float4 u = *reinterpret_cast<const float4 *>(Rl + (h == 0 ? kSlots - 1 : 0) * kSCols);
                v.x += u.x;
                v.y += u.y;
                v.z += u.z;
                v.w += u.w;
            }
            own = wo[0] * v.x;
            own = fmaf(wo[1], v.y, own);
            own = fmaf(wo[2], v.z, own);
            own = fmaf(wo[3], v.w, own);
            nbv = wn[0] * v.x;
            nbv = fmaf(wn[1], v.y, nbv);
            nbv = fmaf(wn[2], v.z, nbv);
            nbv = fmaf(wn[3], v.w, nbv);
        };
        auto clear = [&](float *Rl) {  // only this lane wrote its columns
#pragma unroll
            for (int s = 0; s < kSlots; ++s)
                *reinterpret_cast<float4 *>(Rl + s * kSCols) = make_float4(0.f, 0.f, 0.f, 0.f);
        };

        // ---- per-block HOG: bin h of the cell's blocks on one side of it. Lane 2c + 1 sums the
        // columns of the block that starts at cell c (b = 0), lane 2c + 2 those of the block
        // that ends with it (b = 1).
        auto block_sum = [&](const float *Rl, int h) {
            float own, nbv;
            columns(Rl, h, own, nbv);
            const float o = __shfl_sync(0xffffffffu, own, ((lane - 1) ^ 1) + 1);
            const float n = __shfl_sync(0xffffffffu, nbv, (lane & 1) ? lane + 2 : lane - 2);
            return (own + o) + n;
        };
        auto block_dst = [&](int r, int a) {  // plane 9 (2a + b) of the cell
            return atlas.hog + (int64_t)((2 * a + ((lane & 1) ^ 1)) * kHogBins) * atlas.hog_plane +
                   (int64_t)(L.cell_row + cy0 + r) * atlas.pitch + cx0 + ((lane - 1) >> 1);
        };
        const bool block_st = lane >= 1 && lane <= 2 * kCellTW && cx0 + ((lane - 1) >> 1) < Wc;
        // After a band's first 4 rows, cell row band - 1 has the votes of its own 8 rows: with
        // those of the 4 rows above it they are the blocks that end with the row (a = 1). Cell
        // row band has the votes of the 4 rows above it: set aside, its slots start again.
        auto emit_half = [&](int band) {
            if constexpr (kPb) {
                const int ringA = (band + 1) & 1, ringB = band & 1;
                if (need(band - 1)) {
                    const float *Ra = Wm.R + ringA * kRingStride + 4 * lane;
                    float *dst = block_dst(band - 1, 1);
#pragma unroll
                    for (int h = 0; h < kHogBins; ++h) {
                        const float v = Wm.top[h][lane] + block_sum(Ra, h);
                        if (block_st) dst[(int64_t)h * atlas.hog_plane] = v;
                    }
                }
                if (need(band)) {
                    float *Rb = Wm.R + ringB * kRingStride + 4 * lane;
#pragma unroll
                    for (int h = 0; h < kHogBins; ++h) Wm.top[h][lane] = block_sum(Rb, h);
                    clear(Rb);
                }
            }
        };

        // ---- HOG of cell row r = band - 1 is final: write it, recycle its slots
        auto emit = [&](int band, bool walked) {
            const int ringA = (band + 1) & 1, ringB = band & 1;
            const int r = band - 1;
            const bool out = walked && need(r);
            const int64_t rowoff = (int64_t)(L.cell_row + cy0 + r) * atlas.pitch;
            if (kHog) {
                float *Ra = Wm.R + ringA * kRingStride + 4 * lane;
                if (kPb) {
                    // the 4 rows below the cell row added: the blocks that start with it (a = 0)
                    if (out) {
                        float *dst = block_dst(r, 0);
#pragma unroll
                        for (int h = 0; h < kHogBins; ++h) {
                            const float v = block_sum(Ra, h);
                            if (block_st) dst[(int64_t)h * atlas.hog_plane] = v;
                        }
                    }
                    clear(Ra);
                    return;
                }
                if (walked && band == 0 && cy0 == 0) {
                    // top of the level: the rows above cell row 0 vote into row 0
                    float *Rb = Wm.R + ringB * kRingStride + 4 * lane;
#pragma unroll
                    for (int s = 0; s < kSlots; ++s) {
                        float4 a = *reinterpret_cast<float4 *>(Ra + s * kSCols);
                        float4 &b = *reinterpret_cast<float4 *>(Rb + s * kSCols);
                        b.x += a.x;
                        b.y += a.y;
                        b.z += a.z;
                        b.w += a.w;
                    }
                }
                if (out) {
                    if (band == nb && cy0 + nb == Hc) {
                        // bottom of the level: the rows below the last cell row vote into it
                        const float *Rb = Wm.R + ringB * kRingStride + 4 * lane;
#pragma unroll
                        for (int s = 0; s < kSlots; ++s) {
                            float4 &a = *reinterpret_cast<float4 *>(Ra + s * kSCols);
                            const float4 b = *reinterpret_cast<const float4 *>(Rb + s * kSCols);
                            a.x += b.x;
                            a.y += b.y;
                            a.z += b.z;
                            a.w += b.w;
                        }
                    }
                    const bool st = (lane & 1) && lane <= 2 * kCellTW - 1 && cx0 + ((lane - 1) >> 1) < Wc;
                    float *dst = atlas.hog + rowoff + cx0 + ((lane - 1) >> 1);
#pragma unroll
                    for (int h = 0; h < kHogBins; ++h) {
                        float own, nbv;
                        columns(Ra, h, own, nbv);
                        // cell (t - 1) / 2 at odd lane t: own(t) + own(t + 1) + nb(t - 1) + nb(t + 2)
                        const float o_next = __shfl_down_sync(0xffffffffu, own, 1);
                        const float n_prev = __shfl_up_sync(0xffffffffu, nbv, 1);
                        const float n_next2 = __shfl_down_sync(0xffffffffu, nbv, 2);
                        const float tot = ((own + o_next) + n_prev) + n_next2;
                        if (st) dst[(int64_t)h * atlas.hog_plane] = tot;
                    }
                }
                clear(Ra);  // for row r + 2
            }
        };

        // ---- the walk: bands 0..nb. Rows arrive in pairs, the next pair loaded
        // while the current one is processed (across band boundaries too).
        uint32_t p0[3], p1[3];
        Row ra, rb;
        bool have = false;   // p0, p1 and ra, rb hold this band's first rows
        bool walked_prev = false;
#pragma unroll 1
        for (int band = 0; band <= nb; ++band) {
            const int yb = 8 * (cy0 + band) - 4;
            if (!(need(band - 1) || need(band))) {
                if (walked_prev) {  // recycle row band - 1's slots
                    emit(band, false);
                }
                have = false;
                walked_prev = false;
                continue;
            }
            // rows outside the cell grid: the first half of the level's first band and the
            // second half of its last one are not walked
            const int i0 = cy0 + band == 0 ? 2 : 0, i1 = cy0 + band == Hc ? 2 : 4;
            if (!have) {
                uint32_t w[3];
                fetch(yb + 2 * i0 - 1, w);
                ra = mkrow(w);
                fetch(yb + 2 * i0, w);
                rb = mkrow(w);
                fetch(yb + 2 * i0 + 1, p0);
                fetch(yb + 2 * i0 + 2, p1);
            }
            const bool pf = band + 1 <= nb && (need(band) || need(band + 1));
            const int ringA = (band + 1) & 1;
            const uint32_t dB = (ringA ? -4 : 4) * kRingStride;  // bytes from row band - 1's slots to row band's
            uint32_t va[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) va[j] = vb[j] + 4u * (uint32_t)(ringA * kRingStride);
            float wa = (7.5f - 2 * i0) * 0.125f;  // weight of cell row band - 1 in band row k: (7.5 - k) / 8
#pragma unroll 1
            for (int i = i0; i < i1; ++i) {
                const Row c0 = mkrow(p0), c1 = mkrow(p1);
                if (i < 3 || pf) {
                    fetch(yb + 3 + 2 * i, p0);
                    fetch(yb + 4 + 2 * i, p1);
                }
                // band rows 2i, 2i + 1; LBP cell row band - 1 for rows < 4, band for the others
                pixel_row(ra, rb, c0, wa, 1.f - wa, va, dB);
                pixel_row(rb, c0, c1, wa - 0.125f, 1.125f - wa, va, dB);
                ra = c0;
                rb = c1;
                wa -= 0.25f;
                if (kPb && i == 1) emit_half(band);
                if (kLbp && i == 1) emit_lbp(band);
            }
            emit(band, true);
            have = pf;
            walked_prev = true;
        }
        __syncwarp();  // the next strip reuses the warp's shared memory
    }
}

using StripFn = void (*)(const LevelDesc *, const uint8_t *, CellAtlas, const StripItem *, int, int *,
                         const uint32_t *);
constexpr int kBlk = kFeatHogBlock;
// [feature set][cell-major LBP counts]; without LBP the layout does not matter
const StripFn kStripFns[5][2] = {{k_cells_warp<kFeatHog | kFeatLbp, false>, k_cells_warp<kFeatHog | kFeatLbp, true>},
                                 {k_cells_warp<kFeatHog, false>, k_cells_warp<kFeatHog, false>},
                                 {k_cells_warp<kFeatLbp, false>, k_cells_warp<kFeatLbp, true>},
                                 {k_cells_warp<kFeatHog | kFeatLbp | kBlk, false>,
                                  k_cells_warp<kFeatHog | kFeatLbp | kBlk, true>},
                                 {k_cells_warp<kFeatHog | kBlk, false>, k_cells_warp<kFeatHog | kBlk, false>}};

int strip_fn_index(int feat) {
    const int blk = (feat & kBlk) ? 3 : 0;
    if ((feat & ~kBlk) == kFeatHog) return blk + 1;
    if (feat == kFeatLbp) return 2;
    return blk;
}

int strip_smem(int index) { return (int)(index >= 3 ? sizeof(StripSmem<true>) : sizeof(StripSmem<false>)); }

}  // namespace

cudaError_t init_cells_warp() {
    for (int i = 0; i < 10; ++i) {
        const cudaError_t e = cudaFuncSetAttribute(kStripFns[i / 2][i % 2], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   strip_smem(i / 2));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_cells_warp(cudaStream_t s, const LevelDesc *d_levels, const uint8_t *pyr, CellAtlas atlas,
                              const StripItem *d_items, int n_items, int *d_queue, int sm_count,
                              const uint32_t *c_flag, int feat) {
    if (n_items <= 0) return cudaSuccess;
    // resident CTAs: 4 per SM (shared memory); the warps share the strip queue. A
    // small plan gets one CTA per strip, so that its warps spread over the SMs.
    static_assert(kWarps * 4 == kStripWarpsPerSm, "resident warps per SM");
    const int grid = std::min(n_items, 4 * sm_count);
    const int k = strip_fn_index(feat);
    kStripFns[k][atlas.lbp_cells != 0]<<<grid, kWarps * 32, strip_smem(k), s>>>(
        d_levels, pyr, atlas, d_items, n_items, d_queue, c_flag);
    return cudaGetLastError();
}

}  // namespace pd
