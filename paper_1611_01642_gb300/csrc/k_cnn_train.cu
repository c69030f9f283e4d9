// Learned window proposal: training kernels (forward with stored
// activations, BCE-with-logits loss, backward, Adam), all on CUDA cores with
// fp32 accumulation. Activations a1, a2 are stored in bf16 exactly as the
// inference kernel stores them; a3 and h stay fp32. Every reduction runs in
// a fixed order (no floating-point atomics, a fixed number of blocks), so a
// training step is deterministic and resuming from a checkpoint reproduces
// the same run.
//
// Layout: for each pyramid level of the batch, planar activation maps
// a1[16][H1][P1], a2[32][H2][P2] (bf16), a3[32][H3][P3] (fp32) and
// dz2[32][H2][P2] (fp32) at offsets of a TrainLevel table, rows padded to a
// multiple of 8 elements so that four of them move per access; h, dh on the
// cell atlas (row cell_row + cy, pitch P); logits, labels and dz at the
// score-map offsets of the level.
//
// What bounds them: the convolutions are 3 x 468 multiply-adds per pyramid
// pixel, all on the FP32 pipe, two multiply-adds per instruction
// (fma.rn.f32x2 over pairs of channels or positions). In the gradients one
// operand, dz, is fp32; the forward convolutions of layers 2 and 3 have bf16
// operands and could run on the tensor cores as in inference. Every kernel
// walks a contiguous share of the batch's tiles with persistent blocks; the
// operands of a tile sit in shared memory, the next tile's arrive there
// (cp.async) while this one is worked on, and a thread holds 4 to 16 positions
// times 4 to 16 channels (or 8 channels times 9 taps), so that one broadcast
// load feeds 4 to 8 instructions. Weight gradients stay in registers over a
// block's whole share and leave as one partial per block, summed in block
// order by the last kernel.
// 4 x 1280x720 frames (38 M pyramid pixels, 36 levels each), one step:
// 74.4 -> 6.67 ms against one thread per position with all levels of a weight's
// gradient in one block, and 6.67 -> 3.25 ms by fetching ahead (half of every
// warp's waiting was for the tile's loads, with 8 to 16 warps per SM to hide
// them): weight gradient of layer 1 with the data gradient of layer 2 2.05 ->
// 0.675, weight gradients of layers 2 and 3 1.31 -> 0.67 and 0.75 -> 0.38, data
// gradient of layer 3 0.55 -> 0.31, forward convolutions 0.20 -> 0.15, 0.84 ->
// 0.49 and 0.61 -> 0.35 ms. The FP32 pipe is now 50 to 76% busy in them;
// what is left is its throttle and dispatch stalls more than waiting.
#include "pd_internal.h"

#include <cuda_bf16.h>

#include "f32x2.cuh"

namespace pd {
namespace {

__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// A block's contiguous share [t, end) of a tile grid over all levels
// (TrainLevel::g[GRID] is a level's first tile; the grids are listed there).
template <int GRID>
struct Walk {
    const TrainLevel *tl;
    int n, t, end, k, next;
    __device__ Walk(const TrainLevel *levels, int n_levels, int total) : tl(levels), n(n_levels) {
        t = (int)((int64_t)total * blockIdx.x / gridDim.x);
        end = (int)((int64_t)total * (blockIdx.x + 1) / gridDim.x);
        int lo = 0, hi = n - 1;  // the last level whose first tile is <= t
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tl[mid].g[GRID] <= t) lo = mid;
            else hi = mid - 1;
        }
        k = lo;
        next = k + 1 < n ? tl[k + 1].g[GRID] : total;
    }
    __device__ bool valid() const { return t < end; }
    __device__ int local() const { return t - tl[k].g[GRID]; }
    __device__ void step(int total) {
        ++t;
        while (t >= next && k + 1 < n) {
            ++k;
            next = k + 1 < n ? tl[k + 1].g[GRID] : total;
        }
    }
};

// ---- staging: before a block works on a tile it starts the copies of the next
// one into its other buffer (cp.async, 16 bytes per copy, zeros outside the
// plane); a thread waits for its own copies and the block's barrier hands them over.
__device__ __forceinline__ uint32_t smem_at(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
// 16 bytes to shared memory, of which the first n come from src and the rest are 0 (n <= 0: all)
__device__ __forceinline__ void copy16(void *dst, const void *src, int n) {
    n = min(max(n, 0), 16);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_at(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One chunk of row y, elements [x, x + 16 / sizeof(T)), of a plane of H rows and
// W valid columns (row pitch P); zeros outside.
template <class T>
__device__ __forceinline__ void copy_row16(void *dst, const T *plane, int y, int x, int H, int W, int P) {
    const bool in = y >= 0 && y < H && x >= 0 && x < W;
    copy16(dst, in ? plane + (int64_t)y * P + x : plane, in ? (int)sizeof(T) * (W - x) : 0);
}

constexpr int kXE = 64, kXO = 68;  // input tile row pitches: even columns, odd columns (from -1)

// Input of the 64 x 16 layer-1 positions from (i0, j0): rows 2 i0 - 1 .., 144
// bytes from column 2 j0 - 16. copy_pixels: thread e's copy (e < 33 * 9).
constexpr int kRawP = 144;
__device__ __forceinline__ void copy_pixels(uint8_t *raw, const uint8_t *img, const LevelDesc &L, int i0, int j0, int e) {
    const int r = e / 9, q = e - 9 * r;
    copy_row16(raw + 16 * e, img, 2 * i0 + r - 1, 2 * j0 - 16 + 16 * q, L.Hk, L.Wk, L.img_pitch);
}
// E[r][j] = x at column 2 (j0 + j), O[r][j] = x at column 2 (j0 + j) - 1, row
// 2 i0 + r - 1; zero outside the level.
template <int THREADS>
__device__ __forceinline__ void spread_pixels(const uint8_t *raw, const LevelDesc &L, const float *lut, int i0, int j0,
                                              float *E, float *O) {
    const int Wk = L.Wk, Hk = L.Hk;
    for (int e = threadIdx.x; e < 33 * 33; e += THREADS) {
        const int r = e / 33, w4 = e - 33 * r, y = 2 * i0 + r - 1, x = 2 * j0 - 4 + 4 * w4, m = 2 * w4 - 2;
        const uint32_t v = *reinterpret_cast<const uint32_t *>(raw + r * kRawP + 12 + 4 * w4);
        const bool in = y >= 0 && y < Hk && x >= 0;
        if (m >= 0) {
            E[r * kXE + m] = in && x < Wk ? lut[v & 255u] : 0.f;
            O[r * kXO + m + 1] = in && x + 1 < Wk ? lut[(v >> 8) & 255u] : 0.f;
            E[r * kXE + m + 1] = in && x + 2 < Wk ? lut[(v >> 16) & 255u] : 0.f;
        }
        O[r * kXO + m + 2] = in && x + 3 < Wk ? lut[v >> 24] : 0.f;
    }
}

// ---- layer 1: 64 x 16 positions per tile, 4 positions x 16 channels per
// thread. The sum of a channel runs over (dy, dx) in order, as everywhere.
// Bound by issue and its stores (a1 is 32 bytes per position): 154 us, 197
// before the pixels of the next tile were fetched ahead.
__global__ void __launch_bounds__(256) t_conv1(const TrainLevel *__restrict__ tl, int n_tl, int n_tiles,
                                               const LevelDesc *__restrict__ levels, const uint8_t *__restrict__ pyr,
                                               const float *__restrict__ in_tab, const float *__restrict__ w,
                                               const float *__restrict__ b, __nv_bfloat16 *__restrict__ act) {
    __shared__ __align__(16) float E[33 * kXE], O[33 * kXO], ws[9 * 16], bs[16], lut[256];
    __shared__ __align__(16) uint8_t raw[2][33 * kRawP];
    const int tid = threadIdx.x;
    lut[tid] = in_tab[tid];
    if (tid < 144) ws[(tid % 9) * 16 + tid / 9] = w[tid];
    if (tid < 16) bs[tid] = b[tid];
    const int g = tid & 15, ir = tid >> 4;
    Walk<0> wk(tl, n_tl, n_tiles);
    auto fetch = [&](uint8_t *dst) {
        const TrainLevel &T = tl[wk.k];
        const LevelDesc &L = levels[T.level];
        const int ntx = (T.W2 + 31) / 32, lt = wk.local();
        for (int e = tid; e < 33 * 9; e += 256)
            copy_pixels(dst, pyr + L.img_off, L, 16 * (lt / ntx), 64 * (lt % ntx), e);
    };
    if (wk.valid()) fetch(raw[0]);
    for (int buf = 0; wk.valid(); buf ^= 1) {
        const TrainLevel &T = tl[wk.k];
        const LevelDesc &L = levels[T.level];
        const int ntx = (T.W2 + 31) / 32, lt = wk.local();
        const int i0 = 16 * (lt / ntx), j0 = 64 * (lt % ntx);
        copies_done();
        __syncthreads();
        spread_pixels<256>(raw[buf], L, lut, i0, j0, E, O);
        wk.step(n_tiles);
        if (wk.valid()) fetch(raw[buf ^ 1]);
        __syncthreads();
        f32x2 acc[4][8];
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const f32x2 bb = pack2(bs[2 * o], bs[2 * o + 1]);
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[p][o] = bb;
        }
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
            const int r = 2 * ir + dy;
            const float4 e = *reinterpret_cast<const float4 *>(E + r * kXE + 4 * g);
            const float4 o4 = *reinterpret_cast<const float4 *>(O + r * kXO + 4 * g);
            const float ol = O[r * kXO + 4 * g + 4];
            const f32x2 v0[4] = {dup2(o4.x), dup2(o4.y), dup2(o4.z), dup2(o4.w)};
            const f32x2 v1[4] = {dup2(e.x), dup2(e.y), dup2(e.z), dup2(e.w)};
            const f32x2 v2[4] = {v0[1], v0[2], v0[3], dup2(ol)};
#pragma unroll
            for (int dx = 0; dx < 3; ++dx) {
                const f32x2 *v = dx == 0 ? v0 : dx == 1 ? v1 : v2;
#pragma unroll
                for (int o = 0; o < 8; o += 2) {
                    const ulonglong2 ww = *reinterpret_cast<const ulonglong2 *>(ws + (dy * 3 + dx) * 16 + 2 * o);
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        acc[p][o] = fma2(ww.x, v[p], acc[p][o]);
                        acc[p][o + 1] = fma2(ww.y, v[p], acc[p][o + 1]);
                    }
                }
            }
        }
        const int i = i0 + ir, j = j0 + 4 * g;
        if (i < T.H1 && j < T.P1) {
            __nv_bfloat16 *dst = act + T.a1 + (int64_t)i * T.P1 + j;
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                float v[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) v[p] = fmaxf(o & 1 ? hi2(acc[p][o >> 1]) : lo2(acc[p][o >> 1]), 0.f);
                const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), c = __floats2bfloat162_rn(v[2], v[3]);
                uint2 u;
                u.x = *reinterpret_cast<const uint32_t *>(&a);
                u.y = *reinterpret_cast<const uint32_t *>(&c);
                *reinterpret_cast<uint2 *>(dst + (int64_t)o * T.H1 * T.P1) = u;
            }
        }
    }
}

// ---- layers 2 and 3: 32 x 8 positions per tile, 4 positions x 16 output
// channels per thread; kCS input channels are worked on while the next kCS
// (or the next tile's first) arrive. Activations stay two bf16 columns to a
// word: per input channel and window row 2 activation loads and 12 broadcast
// weight loads for 96 packed multiply-adds. Layer 3 forms the head on its way
// out: h = bh + wh . a3 on the cells, channel by channel (a kernel of its own
// read a3 back for it, 68 us; layer 3 takes 5 us longer).
constexpr int kAP = 36;  // words per staged activation row: columns 2 j0 - 8 ..
template <int CIN>
struct ConvSmem {
    static constexpr int kCS = 128 / CIN;  // 8 or 4: three blocks per SM
    float ws[CIN * 9 * 32];                // [c][tap][o]
    uint32_t as[2][kCS * 17 * kAP];
    float4 head[64];                       // layer 3: bh + wh . a3 over the first 16 channels
    float wh[32];
};
template <int CIN, bool LAST>
__global__ void __launch_bounds__(128) t_conv23(const TrainLevel *__restrict__ tl, int n_tl, int n_tiles,
                                                const __nv_bfloat16 *__restrict__ act, const float *__restrict__ w,
                                                const float *__restrict__ b, __nv_bfloat16 *__restrict__ out16,
                                                float *__restrict__ out32, const LevelDesc *__restrict__ levels,
                                                const float *__restrict__ wh, const float *__restrict__ bh,
                                                float *__restrict__ hmap, int32_t hp) {
    constexpr int kCS = ConvSmem<CIN>::kCS;
    extern __shared__ __align__(16) unsigned char smem_b[];
    ConvSmem<CIN> &S = *reinterpret_cast<ConvSmem<CIN> *>(smem_b);
    const int tid = threadIdx.x;
    for (int i = tid; i < CIN * 9 * 32; i += 128) {
        const int o = i & 31, ct = i >> 5;
        S.ws[i] = w[o * CIN * 9 + ct];
    }
    if (LAST && tid < 32) S.wh[tid] = wh[tid];
    const int o0 = 16 * (tid >> 6), g = tid & 7, ir = (tid >> 3) & 7;
    constexpr int GRID = LAST ? 2 : 0;
    Walk<GRID> wk(tl, n_tl, n_tiles);
    auto fetch = [&](uint32_t *as, int cb) {  // this thread's share of channels cb .. of the tile of wk
        const TrainLevel &T = tl[wk.k];
        const int Hi = LAST ? T.H2 : T.H1, Wi = LAST ? T.W2 : T.W1, Pi = LAST ? T.P2 : T.P1;
        const int ntx = ((LAST ? T.W3 : T.W2) + 31) / 32, lt = wk.local();
        const int i0 = 8 * (lt / ntx), j0 = 32 * (lt % ntx);
        const __nv_bfloat16 *a = act + (LAST ? T.a2 : T.a1) + (int64_t)cb * Hi * Pi;
        for (int e = tid; e < kCS * 17 * 9; e += 128) {
            const int cr = e / 9, q = e - 9 * cr, cc = cr / 17, r = cr - 17 * cc;
            copy_row16(as + 4 * e, a + (int64_t)cc * Hi * Pi, 2 * i0 + r - 1, 2 * j0 - 8 + 8 * q, Hi, Wi, Pi);
        }
    };
    f32x2 bias[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) bias[o] = pack2(b[o0 + 2 * o], b[o0 + 2 * o + 1]);
    int buf = 0;
    if (wk.valid()) fetch(S.as[0], 0);
    while (wk.valid()) {
        const TrainLevel &T = tl[wk.k];
        const int Ho = LAST ? T.H3 : T.H2, Wo = LAST ? T.W3 : T.W2, Po = LAST ? T.P3 : T.P2;
        const int64_t out_off = LAST ? T.a3 : T.a2;
        const int tl_level = T.level;
        const int ntx = (Wo + 31) / 32, lt = wk.local();
        const int i = 8 * (lt / ntx) + ir, j = 32 * (lt % ntx) + 4 * g;
        f32x2 acc[4][8];
#pragma unroll
        for (int o = 0; o < 8; ++o)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[p][o] = bias[o];
#pragma unroll 1
        for (int cb = 0; cb < CIN; cb += kCS, buf ^= 1) {
            copies_done();
            __syncthreads();  // these channels are here, and the other buffer is free
            if (cb + kCS < CIN) {
                fetch(S.as[buf ^ 1], cb + kCS);
            } else {
                wk.step(n_tiles);
                if (wk.valid()) fetch(S.as[buf ^ 1], 0);
            }
#pragma unroll 1
            for (int c = 0; c < kCS; ++c) {
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    const uint32_t *row = S.as[buf] + (c * 17 + 2 * ir + dy) * kAP + 4 + 4 * g;
                    const uint4 u = *reinterpret_cast<const uint4 *>(row);
                    const f32x2 v0[4] = {dup2(bf_hi(row[-1])), dup2(bf_hi(u.x)), dup2(bf_hi(u.y)), dup2(bf_hi(u.z))};
                    const f32x2 v1[4] = {dup2(bf_lo(u.x)), dup2(bf_lo(u.y)), dup2(bf_lo(u.z)), dup2(bf_lo(u.w))};
                    const f32x2 v2[4] = {v0[1], v0[2], v0[3], dup2(bf_hi(u.w))};
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx) {
                        const f32x2 *v = dx == 0 ? v0 : dx == 1 ? v1 : v2;
                        const float *wp = S.ws + ((cb + c) * 9 + dy * 3 + dx) * 32 + o0;
#pragma unroll
                        for (int o = 0; o < 8; o += 2) {
                            const ulonglong2 ww = *reinterpret_cast<const ulonglong2 *>(wp + 2 * o);
#pragma unroll
                            for (int p = 0; p < 4; ++p) {
                                acc[p][o] = fma2(ww.x, v[p], acc[p][o]);
                                acc[p][o + 1] = fma2(ww.y, v[p], acc[p][o + 1]);
                            }
                        }
                    }
                }
            }
        }
        if (LAST) {  // h on the cells, channel by channel: the first two warps, then the others
            const LevelDesc &L = levels[tl_level];
            float h[4];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if ((o0 != 0) == (half != 0)) {
                    const float4 h0 = half ? S.head[tid & 63] : make_float4(bh[0], bh[0], bh[0], bh[0]);
                    h[0] = h0.x, h[1] = h0.y, h[2] = h0.z, h[3] = h0.w;
#pragma unroll
                    for (int o = 0; o < 16; ++o)
#pragma unroll
                        for (int p = 0; p < 4; ++p)
                            h[p] = fmaf(S.wh[o0 + o], fmaxf(o & 1 ? hi2(acc[p][o >> 1]) : lo2(acc[p][o >> 1]), 0.f), h[p]);
                    if (!half) S.head[tid & 63] = make_float4(h[0], h[1], h[2], h[3]);
                }
                if (!half) __syncthreads();
            }
            if (o0 && i < L.Hc) {
#pragma unroll
                for (int p = 0; p < 4; ++p)
                    if (j + p < L.Wc) hmap[(int64_t)(L.cell_row + i) * hp + j + p] = h[p];
            }
        }
        if (i < Ho && j < Po) {
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                float v[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) v[p] = fmaxf(o & 1 ? hi2(acc[p][o >> 1]) : lo2(acc[p][o >> 1]), 0.f);
                const int64_t at = out_off + ((int64_t)(o0 + o) * Ho + i) * Po + j;
                if (LAST) {
                    *reinterpret_cast<float4 *>(out32 + at) = make_float4(v[0], v[1], v[2], v[3]);
                } else {
                    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), c = __floats2bfloat162_rn(v[2], v[3]);
                    uint2 u;
                    u.x = *reinterpret_cast<const uint32_t *>(&a);
                    u.y = *reinterpret_cast<const uint32_t *>(&c);
                    *reinterpret_cast<uint2 *>(out16 + at) = u;
                }
            }
        }
    }
}

// ---- BCE with logits: per window dz = (p y (s - 1) + (1 - y) s) / N, loss
// terms; labels y = score > thr. kLossParts blocks per level, fixed-order sums.
__global__ void __launch_bounds__(256) t_loss(const TrainLevel *__restrict__ tl, const LevelDesc *__restrict__ levels,
                                              const float *__restrict__ logits, const float *__restrict__ scores,
                                              float thr, float pos_weight, float inv_n, float *__restrict__ dz,
                                              float *__restrict__ level_loss) {
    const LevelDesc &L = levels[tl[blockIdx.y].level];
    const int n = L.rows * L.cols;
    float part = 0.f;
    for (int i = blockIdx.x * 256 + threadIdx.x; i < n; i += kLossParts * 256) {
        const float z = logits[L.score_off + i];
        const float y = scores[L.score_off + i] > thr ? 1.f : 0.f;
        // log sigmoid(z) = -softplus(-z), log(1 - sigmoid(z)) = -softplus(z)
        const float sp_neg = fmaxf(-z, 0.f) + log1pf(expf(-fabsf(z)));
        const float sp_pos = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));
        part += pos_weight * y * sp_neg + (1.f - y) * sp_pos;
        const float s = 1.f / (1.f + expf(-z));
        dz[L.score_off + i] = (pos_weight * y * (s - 1.f) + (1.f - y) * s) * inv_n;
    }
    __shared__ float red[256];
    red[threadIdx.x] = part;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) level_loss[blockIdx.y * kLossParts + blockIdx.x] = red[0] * inv_n;
}

// ---- pooling backward into h: dh[c] = sum over the windows that see cell c
// of V[r][s] dz[window] (a gather: no atomics)
__global__ void t_pool_bwd_h(const TrainLevel *__restrict__ tl, const LevelDesc *__restrict__ levels,
                             const float *__restrict__ dz, const float *__restrict__ v,
                             float *__restrict__ dh, int32_t hp) {
    const LevelDesc &L = levels[tl[blockIdx.y].level];
    const int n = L.Hc * L.Wc;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        const int cy = p / L.Wc, cx = p - cy * L.Wc;
        float g = 0.f;
        for (int r = 0; r < 16; ++r) {
            const int wy = cy - r;
            if (wy < 0 || wy >= L.rows) continue;
            for (int s = 0; s < 8; ++s) {
                const int wx = cx - s;
                if (wx < 0 || wx >= L.cols) continue;
                g = fmaf(v[r * 8 + s], dz[L.score_off + (int64_t)wy * L.cols + wx], g);
            }
        }
        dh[(int64_t)(L.cell_row + cy) * hp + cx] = g;
    }
}

// Sum over a warp in a fixed order (every lane gets it).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- gradients of V, bv (32 x 16 windows per tile in shared memory, one
// thread per template position and half of the rows) and of wh, bh (32 x 8
// cells per tile, a warp per 4 channels; it also turns a3 into dz3 = wh dh (a3 > 0),
// in place, 0 outside the cells). Partial p of a block: 0..127 V,
// 128 bv, 129..160 wh, 161 bh.
constexpr int kSmallParts = 162;
__global__ void __launch_bounds__(256) t_small_grads(const TrainLevel *__restrict__ tl, int n_tl, int n_win_tiles,
                                                     int n_cell_tiles, const LevelDesc *__restrict__ levels,
                                                     const float *__restrict__ dz, const float *__restrict__ hmap,
                                                     const float *__restrict__ dh, int32_t hp,
                                                     const float *__restrict__ wh, float *__restrict__ a3,
                                                     float *__restrict__ part) {
    __shared__ float sd[16 * 32], sh[31 * 40], red[256 + 8];
    const int tid = threadIdx.x, q = tid & 127, half = tid >> 7, lane = tid & 31, warp = tid >> 5;
    const int r = q >> 3, s = q & 7;
    float acc = 0.f, accd = 0.f;
    for (Walk<4> wk(tl, n_tl, n_win_tiles); wk.valid(); wk.step(n_win_tiles)) {
        const LevelDesc &L = levels[tl[wk.k].level];
        const int ntx = (L.cols + 31) / 32, lt = wk.local();
        const int y0 = 16 * (lt / ntx), x0 = 32 * (lt % ntx);
        __syncthreads();
        for (int i = tid; i < 16 * 32; i += 256) {
            const int y = y0 + (i >> 5), x = x0 + (i & 31);
            sd[i] = y < L.rows && x < L.cols ? dz[L.score_off + (int64_t)y * L.cols + x] : 0.f;
        }
        for (int i = tid; i < 31 * 39; i += 256) {
            const int yy = i / 39, xx = i - 39 * yy;
            const int y = y0 + yy, x = x0 + xx;
            sh[yy * 40 + xx] = y < L.Hc && x < L.Wc ? hmap[(int64_t)(L.cell_row + y) * hp + x] : 0.f;
        }
        __syncthreads();
        for (int y = 8 * half; y < 8 * half + 8; ++y) {
#pragma unroll 8
            for (int x = 0; x < 32; ++x) {
                const float d = sd[y * 32 + x];
                acc = fmaf(d, sh[(y + r) * 40 + x + s], acc);
                accd += d;
            }
        }
    }
    float aw[4] = {0.f, 0.f, 0.f, 0.f}, ab = 0.f;
    const float4 wh4 = reinterpret_cast<const float4 *>(wh)[warp];
    const float who[4] = {wh4.x, wh4.y, wh4.z, wh4.w};
    for (Walk<2> wk(tl, n_tl, n_cell_tiles); wk.valid(); wk.step(n_cell_tiles)) {
        const TrainLevel &T = tl[wk.k];
        const LevelDesc &L = levels[T.level];
        const int ntx = (T.W3 + 31) / 32, lt = wk.local();
        const int y0 = 8 * (lt / ntx), x = 32 * (lt % ntx) + lane;
        const int64_t plane = (int64_t)T.H3 * T.P3;
        if (x >= T.W3) continue;
        float *src = a3 + T.a3 + 4 * warp * plane + (int64_t)y0 * T.P3 + x;
        const float *dp = dh + (int64_t)(L.cell_row + y0) * hp + x;
        float d[8], v[8][4];
#pragma unroll
        for (int yy = 0; yy < 8; ++yy) {
            d[yy] = y0 + yy < L.Hc && x < L.Wc ? dp[(int64_t)yy * hp] : 0.f;
#pragma unroll
            for (int c = 0; c < 4; ++c) v[yy][c] = y0 + yy < T.H3 ? src[c * plane + yy * T.P3] : 0.f;
        }
#pragma unroll
        for (int yy = 0; yy < 8; ++yy) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                aw[c] = fmaf(d[yy], v[yy][c], aw[c]);
                if (y0 + yy < T.H3) src[c * plane + yy * T.P3] = v[yy][c] > 0.f ? who[c] * d[yy] : 0.f;
            }
            ab += d[yy];
        }
    }
    float *out = part + (int64_t)blockIdx.x * kSmallParts;
    red[tid] = acc;
    if (q == 0) red[256 + half] = accd;
    __syncthreads();
    if (tid < 128) out[tid] = red[tid] + red[tid + 128];
    if (tid == 0) out[128] = red[256] + red[257];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const float v = warp_sum(aw[c]);
        if (lane == 0) out[129 + 4 * warp + c] = v;
    }
    ab = warp_sum(ab);
    if (tid == 0) out[161] = ab;
}

// Data gradient of a stride-2 layer for 2 x 2 quads of input positions (a quad
// is (2i, 2i+1) x (2j, 2j+1)) and 4 input channels: a quad takes 9 products per
// (output channel, input channel) from the 2 x 2 output positions it reaches. d: the
// tile's output gradients [32][dplane], row pitch DP, at (i, j); ws: [32 o][9
// taps][CIN] weights at the thread's channels.
// acc[quad row][quad column][2 * row + column][channel pair].
template <int CIN, int DP>
__device__ __forceinline__ void quad_block(const float *d, int dplane, const float *ws, f32x2 (&acc)[2][2][4][2]) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[q >> 1][q & 1][p][0] = acc[q >> 1][q & 1][p][1] = 0ull;
#pragma unroll 1
    for (int o = 0; o < 32; ++o) {
        const float *dp = d + o * dplane;
        f32x2 v[3][3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const float2 t = *reinterpret_cast<const float2 *>(dp + r * DP);
            v[r][0] = dup2(t.x);
            v[r][1] = dup2(t.y);
            v[r][2] = dup2(dp[r * DP + 2]);
        }
        const float *wo = ws + o * 9 * CIN;
        // tap, input position (2 * row + column), output position (row, column)
        constexpr int kTap[9] = {4, 3, 5, 1, 7, 0, 2, 6, 8};
        constexpr int kPos[9] = {0, 1, 1, 2, 2, 3, 3, 3, 3};
        constexpr int kRow[9] = {0, 0, 0, 1, 0, 1, 1, 0, 0};
        constexpr int kCol[9] = {0, 1, 0, 0, 0, 1, 0, 1, 0};
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(wo + kTap[k] * CIN);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const f32x2 x = v[(q >> 1) + kRow[k]][(q & 1) + kCol[k]];
                f32x2(&a)[2] = acc[q >> 1][q & 1][kPos[k]];
                a[0] = fma2(w.x, x, a[0]);
                a[1] = fma2(w.y, x, a[1]);
            }
        }
    }
}

// ---- dz2 = (a2 > 0) * data gradient of layer 3: a tile is 16 x 8 quads
// (32 x 16 layer-2 positions), 32 blocks of 2 x 2 quads x 8 groups of 4 channels.
constexpr int kD3P = 20;  // staged dz3 row pitch (17 columns)
struct Dz2Smem {
    float ws[32 * 9 * 32];           // [o][tap][c]
    float ds[2][32 * 9 * kD3P];      // dz3 [o][i][j]
    __nv_bfloat16 a2[32 * 16 * 32];  // [c][row][column] of the tile worked on
};
__global__ void __launch_bounds__(256) t_dz2(const TrainLevel *__restrict__ tl, int n_tl, int n_tiles,
                                             const float *__restrict__ dz3, const float *__restrict__ w,
                                             const __nv_bfloat16 *__restrict__ act, float *__restrict__ dz2) {
    extern __shared__ __align__(16) unsigned char smem_b[];
    Dz2Smem &S = *reinterpret_cast<Dz2Smem *>(smem_b);
    const int tid = threadIdx.x;
    for (int i = tid; i < 32 * 9 * 32; i += 256) {
        const int c = i & 31, ot = i >> 5, o = ot / 9;
        S.ws[i] = w[(o * 32 + c) * 9 + ot - 9 * o];
    }
    Walk<3> wk(tl, n_tl, n_tiles);
    auto fetch = [&](float *ds) {  // this thread's share of the tile of wk
        const TrainLevel &T = tl[wk.k];
        const int ntx = (T.W3 + 15) / 16, lt = wk.local();
        const int i0 = 8 * (lt / ntx), j0 = 16 * (lt % ntx), H3 = T.H3, W3 = T.W3, P3 = T.P3;
        const float *d = dz3 + T.a3;
        for (int e = tid; e < 32 * 9 * 5; e += 256) {
            const int oi = e / 5, q = e - 5 * oi, o = oi / 9, i = oi - 9 * o;
            copy_row16(ds + 4 * e, d + (int64_t)o * H3 * P3, i0 + i, j0 + 4 * q, H3, W3, P3);
        }
    };
    const int c0 = 4 * (tid >> 5), qx = tid & 7, qy = (tid >> 3) & 3;
    if (wk.valid()) fetch(S.ds[0]);
#pragma unroll 1
    for (int b = 0; wk.valid(); b ^= 1) {
        copies_done();
        __syncthreads();  // this tile is here, the other buffer and the mask are free
        const TrainLevel &T = tl[wk.k];
        const int H2 = T.H2, W2 = T.W2, P2 = T.P2;
        const int ntx = (T.W3 + 15) / 16, lt = wk.local();
        const int y0 = 16 * (lt / ntx), x0 = 32 * (lt % ntx);
        const __nv_bfloat16 *a2 = act + T.a2;
        float *out = dz2 + T.d2;
#pragma unroll
        for (int e = tid; e < 32 * 16 * 4; e += 256) {
            const int c = e >> 6, r = (e >> 2) & 15, q = e & 3;
            copy_row16(S.a2 + 8 * e, a2 + (int64_t)c * H2 * P2, y0 + r, x0 + 8 * q, H2, W2, P2);
        }
        wk.step(n_tiles);
        if (wk.valid()) fetch(S.ds[b ^ 1]);
        f32x2 acc[2][2][4][2];
        quad_block<32, kD3P>(S.ds[b] + 2 * qy * kD3P + 2 * qx, 9 * kD3P, S.ws + c0, acc);
        copies_done();
        __syncthreads();  // the mask is there
        const int x = x0 + 4 * qx;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int y = y0 + 4 * qy + a;
            if (y >= H2 || x >= P2) continue;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint2 m = *reinterpret_cast<const uint2 *>(S.a2 + ((c0 + c) * 16 + 4 * qy + a) * 32 + 4 * qx);
                float v[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const f32x2 s = acc[a >> 1][p >> 1][2 * (a & 1) + (p & 1)][c >> 1];
                    v[p] = c & 1 ? hi2(s) : lo2(s);
                }
                *reinterpret_cast<float4 *>(out + ((int64_t)(c0 + c) * H2 + y) * P2 + x) =
                    make_float4(bf_lo(m.x) > 0.f ? v[0] : 0.f, bf_hi(m.x) > 0.f ? v[1] : 0.f,
                                bf_lo(m.y) > 0.f ? v[2] : 0.f, bf_hi(m.y) > 0.f ? v[3] : 0.f);
            }
        }
    }
}

// ---- layer 1's weight gradient. dz1 = (a1 > 0) * data gradient of layer 2 is
// only needed for it, so a thread keeps its 4 x 4 positions x 4 channels of dz1
// in registers and adds their products with the input pixels to its own sums;
// dz1 is never written (it would be 2 x 64 bytes per position of traffic). A
// tile is 32 x 8 quads (64 x 16 layer-1 positions): 64 blocks of 2 x 2 quads x 4
// channel groups. (Two quads and 4 channels per thread on twice the warps: shared
// memory 76% busy, 0.69 ms against 0.675; two quads and 8 channels, with a ninth
// warp to copy: 168 registers, the loads of the weights waited for, 1.01 ms.)
constexpr int kD2P = 36;  // staged dz2 row pitch (33 columns)
constexpr int kW1Parts = 160;
struct Dw1Stage {
    float ds[32 * 9 * kD2P];         // dz2 [o][i][j]
    __nv_bfloat16 a1[16 * 16 * 64];  // [c][row][column]
    uint8_t raw[33 * kRawP];         // input pixels
};
struct Dw1Smem {
    float ws[32 * 9 * 16];           // [o][tap][c]
    Dw1Stage st[2];
    float E[33 * kXE], O[33 * kXO];  // input pixels
    float lut[256];
    float red[8 * 40];
};
__global__ void __launch_bounds__(256, 1) t_dw1(const TrainLevel *__restrict__ tl, int n_tl, int n_tiles,
                                                const LevelDesc *__restrict__ levels,
                                                const uint8_t *__restrict__ pyr, const float *__restrict__ in_tab,
                                                const float *__restrict__ w, const __nv_bfloat16 *__restrict__ act,
                                                const float *__restrict__ dz2, float *__restrict__ part) {
    extern __shared__ __align__(16) unsigned char smem_b[];
    Dw1Smem &S = *reinterpret_cast<Dw1Smem *>(smem_b);
    const int tid = threadIdx.x;
    S.lut[tid] = in_tab[tid];
    for (int i = tid; i < 32 * 9 * 16; i += 256) {
        const int c = i & 15, ot = i >> 4, o = ot / 9;
        S.ws[i] = w[(o * 16 + c) * 9 + ot - 9 * o];
    }
    Walk<0> wk(tl, n_tl, n_tiles);
    auto fetch = [&](Dw1Stage &st) {  // this thread's share of the tile of wk
        const TrainLevel &T = tl[wk.k];
        const LevelDesc &L = levels[T.level];
        const int ntx = (T.W2 + 31) / 32, lt = wk.local();
        const int i0 = 8 * (lt / ntx), j0 = 32 * (lt % ntx);
        for (int e = tid; e < 33 * 9; e += 256) copy_pixels(st.raw, pyr + L.img_off, L, 2 * i0, 2 * j0, e);
        const int H2 = T.H2, W2 = T.W2, P2 = T.P2, H1 = T.H1, W1 = T.W1, P1 = T.P1;
        const float *d = dz2 + T.d2;
        for (int e = tid; e < 32 * 9 * 9; e += 256) {
            const int row = e / 9, q = e - 9 * row, o = row / 9, i = row - 9 * o;
            copy_row16(st.ds + 4 * e, d + (int64_t)o * H2 * P2, i0 + i, j0 + 4 * q, H2, W2, P2);
        }
        const __nv_bfloat16 *a1 = act + T.a1;
#pragma unroll
        for (int e = tid; e < 16 * 16 * 8; e += 256) {
            const int c = e >> 7, r = (e >> 3) & 15, q = e & 7;
            copy_row16(st.a1 + 8 * e, a1 + (int64_t)c * H1 * P1, 2 * i0 + r, 2 * j0 + 8 * q, H1, W1, P1);
        }
    };
    const int c0 = 4 * (tid >> 6), qx = tid & 15, qy = (tid >> 4) & 3;
    f32x2 sum[10][2];
#pragma unroll
    for (int k = 0; k < 10; ++k) sum[k][0] = sum[k][1] = 0ull;
    if (wk.valid()) fetch(S.st[0]);
#pragma unroll 1
    for (int b = 0; wk.valid(); b ^= 1) {
        copies_done();
        __syncthreads();  // this tile is here, and the other buffer is free
        const Dw1Stage &st = S.st[b];
        {
            const TrainLevel &T = tl[wk.k];
            const LevelDesc &L = levels[T.level];
            const int ntx = (T.W2 + 31) / 32, lt = wk.local();
            spread_pixels<256>(st.raw, L, S.lut, 16 * (lt / ntx), 64 * (lt % ntx), S.E, S.O);
        }
        wk.step(n_tiles);
        if (wk.valid()) fetch(S.st[b ^ 1]);
        f32x2 acc[2][2][4][2];
        quad_block<16, kD2P>(st.ds + 2 * qy * kD2P + 2 * qx, 9 * kD2P, S.ws + c0, acc);
        // relu mask of a1 (0 outside the level)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const __nv_bfloat16 *src = st.a1 + ((c0 + 2 * c) * 16 + 4 * qy + a) * 64 + 4 * qx;
                const uint2 m0 = *reinterpret_cast<const uint2 *>(src);
                const uint2 m1 = *reinterpret_cast<const uint2 *>(src + 16 * 64);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint32_t u0 = p < 2 ? m0.x : m0.y, u1 = p < 2 ? m1.x : m1.y;
                    const bool k0 = (p & 1 ? bf_hi(u0) : bf_lo(u0)) > 0.f;
                    const bool k1 = (p & 1 ? bf_hi(u1) : bf_lo(u1)) > 0.f;
                    f32x2 &s = acc[a >> 1][p >> 1][2 * (a & 1) + (p & 1)][c];
                    s = pack2(k0 ? lo2(s) : 0.f, k1 ? hi2(s) : 0.f);
                }
            }
        }
        __syncthreads();  // the pixels are there
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) {
                const int r = 2 * (4 * qy + a) + dy;
                const float4 e = *reinterpret_cast<const float4 *>(S.E + r * kXE + 4 * qx);
                const float4 o4 = *reinterpret_cast<const float4 *>(S.O + r * kXO + 4 * qx);
                const f32x2 ev[4] = {dup2(e.x), dup2(e.y), dup2(e.z), dup2(e.w)};
                const f32x2 ov[5] = {dup2(o4.x), dup2(o4.y), dup2(o4.z), dup2(o4.w), dup2(S.O[r * kXO + 4 * qx + 4])};
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const f32x2 d = acc[a >> 1][p >> 1][2 * (a & 1) + (p & 1)][c];
                        sum[3 * dy][c] = fma2(d, ov[p], sum[3 * dy][c]);
                        sum[3 * dy + 1][c] = fma2(d, ev[p], sum[3 * dy + 1][c]);
                        sum[3 * dy + 2][c] = fma2(d, ov[p + 1], sum[3 * dy + 2][c]);
                        if (dy == 0) sum[9][c] = add2(sum[9][c], d);
                    }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 10; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float v = warp_sum(c & 1 ? hi2(sum[k][c >> 1]) : lo2(sum[k][c >> 1]));
            if ((tid & 31) == 0) S.red[(tid >> 5) * 40 + k * 4 + c] = v;
        }
    __syncthreads();
    if (tid < kW1Parts) {  // order: 144 weights [c][tap], 16 biases
        const int c = tid < 144 ? tid / 9 : tid - 144, k = tid < 144 ? tid % 9 : 9;
        const float *r = S.red + (c >> 2) * 2 * 40 + k * 4 + (c & 3);
        part[(int64_t)blockIdx.x * kW1Parts + tid] = r[0] + r[40];
    }
}

// ---- weight gradients of layers 2 and 3: dW[o][c][tap] = sum over positions
// of dz[o] a[c at the tap]. A tile is 16 x 8 positions; a thread holds one
// input channel x 8 output channels x 9 taps, in pairs of positions (so that
// the gradients pair up as they lie), and a half or a quarter of the tile's
// rows. Lanes are channels: dz is a broadcast. Activations stay two bf16
// columns to a word until they are used: taking them apart costs 12 operations
// per 4 columns and row against 6 packed multiply-adds per output channel, so a thread
// takes 8 output channels and 255 registers (4 and twice the warps: 0.76 and
// 0.39 ms, now 0.67 and 0.38). All threads fetch the next tile while they work
// on this one.
constexpr int kWAP = 20, kWAC = 17 * kWAP;  // staged activations: words per row (columns 2 j0 - 8 ..), per channel
constexpr int kWDP = 132;                   // staged dz: floats per output channel (128 positions)
static_assert(kWAC % 32 == 20, "8 channels of a row in 8 different quads of banks");
template <int CIN>
struct Dw23Stage {
    float ds[32 * kWDP];
    uint32_t as[CIN * kWAC];
};
template <int CIN>
__global__ void __launch_bounds__(256, 1) t_dw23(const TrainLevel *__restrict__ tl, int n_tl, int n_tiles,
                                              const __nv_bfloat16 *__restrict__ act, const float *__restrict__ dz,
                                              float *__restrict__ part) {
    constexpr bool LAST = CIN == 32;
    constexpr int kTeam = 4 * CIN, kParts = 256 / kTeam, kRows = 8 / kParts;  // threads of one part of the rows
    extern __shared__ __align__(16) unsigned char smem_b[];
    Dw23Stage<CIN> *st = reinterpret_cast<Dw23Stage<CIN> *>(smem_b);
    const int tid = threadIdx.x;
    const int c = tid % CIN, og = (tid / CIN) & 3, part_i = tid / kTeam;
    f32x2 acc[8][9];
    float bias = 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[u][k] = 0ull;
    constexpr int GRID = LAST ? 3 : 1;
    Walk<GRID> wk(tl, n_tl, n_tiles);
    auto fetch = [&](Dw23Stage<CIN> &S) {  // this thread's share of the tile of wk
        const TrainLevel &T = tl[wk.k];
        const int Hi = LAST ? T.H2 : T.H1, Wi = LAST ? T.W2 : T.W1, Pi = LAST ? T.P2 : T.P1;
        const int Ho = LAST ? T.H3 : T.H2, Wo = LAST ? T.W3 : T.W2, Po = LAST ? T.P3 : T.P2;
        const int ntx = (Wo + 15) / 16, lt = wk.local();
        const int i0 = 8 * (lt / ntx), j0 = 16 * (lt % ntx);
        const float *d = dz + (LAST ? T.a3 : T.d2);
#pragma unroll
        for (int e = tid; e < 32 * 8 * 4; e += 256) {
            const int o = e >> 5, i = (e >> 2) & 7, q = e & 3;
            copy_row16(S.ds + o * kWDP + i * 16 + 4 * q, d + (int64_t)o * Ho * Po, i0 + i, j0 + 4 * q, Ho, Wo, Po);
        }
        const __nv_bfloat16 *a = act + (LAST ? T.a2 : T.a1);
        for (int e = tid; e < CIN * 17 * 5; e += 256) {
            const int cr = e / 5, q = e - 5 * cr, cc = cr / 17, r = cr - 17 * cc;
            copy_row16(S.as + 4 * e, a + (int64_t)cc * Hi * Pi, 2 * i0 + r - 1, 2 * j0 - 8 + 8 * q, Hi, Wi, Pi);
        }
    };
    if (wk.valid()) fetch(st[0]);
#pragma unroll 1
    for (int b = 0; wk.valid(); b ^= 1) {
        copies_done();
        __syncthreads();  // this tile is here, and the other buffer is free
        wk.step(n_tiles);
        if (wk.valid()) fetch(st[b ^ 1]);
        const Dw23Stage<CIN> &S = st[b];
        {
            const float4 *d = reinterpret_cast<const float4 *>(S.ds + (tid >> 3) * kWDP + 4 * (tid & 7));
#pragma unroll
            for (int q = 0; q < 4; ++q) bias += (d[8 * q].x + d[8 * q].y) + (d[8 * q].z + d[8 * q].w);
        }
#pragma unroll 1
        for (int i = part_i * kRows; i < (part_i + 1) * kRows; ++i) {
            const uint32_t *ap = S.as + c * kWAC + 2 * i * kWAP + 4;
            const float *dp = S.ds + 8 * og * kWDP + 16 * i;
            uint32_t prev[3];
#pragma unroll
            for (int dy = 0; dy < 3; ++dy) prev[dy] = ap[dy * kWAP - 1];
#pragma unroll
            for (int j = 0; j < 16; j += 4) {
                ulonglong2 d[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) d[u] = *reinterpret_cast<const ulonglong2 *>(dp + u * kWDP + j);
#pragma unroll
                for (int dy = 0; dy < 3; ++dy) {
                    const uint4 w = *reinterpret_cast<const uint4 *>(ap + dy * kWAP + j);
                    const f32x2 l0 = pack2(bf_hi(prev[dy]), bf_hi(w.x)), l1 = pack2(bf_hi(w.y), bf_hi(w.z));
                    const f32x2 e0 = pack2(bf_lo(w.x), bf_lo(w.y)), e1 = pack2(bf_lo(w.z), bf_lo(w.w));
                    const f32x2 r0 = pack2(bf_hi(w.x), bf_hi(w.y)), r1 = pack2(bf_hi(w.z), bf_hi(w.w));
                    prev[dy] = w.w;
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][3 * dy] = fma2(l0, d[u].x, acc[u][3 * dy]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][3 * dy + 1] = fma2(e0, d[u].x, acc[u][3 * dy + 1]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][3 * dy + 2] = fma2(r0, d[u].x, acc[u][3 * dy + 2]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][3 * dy] = fma2(l1, d[u].y, acc[u][3 * dy]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][3 * dy + 1] = fma2(e1, d[u].y, acc[u][3 * dy + 1]);
#pragma unroll
                    for (int u = 0; u < 8; ++u) acc[u][3 * dy + 2] = fma2(r1, d[u].y, acc[u][3 * dy + 2]);
                }
            }
        }
    }
    // the parts' sums, in order
    float *x = reinterpret_cast<float *>(smem_b);
    __syncthreads();
    if (part_i) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int k = 0; k < 9; ++k) x[(u * 9 + k) * (256 - kTeam) + tid - kTeam] = lo2(acc[u][k]) + hi2(acc[u][k]);
    }
    __syncthreads();
    float *out = part + (int64_t)blockIdx.x * (32 * CIN * 9 + 32);
    if (!part_i) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                float v = lo2(acc[u][k]) + hi2(acc[u][k]);
#pragma unroll
                for (int q = 0; q + 1 < kParts; ++q) v += x[(u * 9 + k) * (256 - kTeam) + q * kTeam + tid];
                out[((8 * og + u) * CIN + c) * 9 + k] = v;
            }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) bias += __shfl_xor_sync(0xffffffffu, bias, o);
    if ((tid & 7) == 0) out[32 * CIN * 9 + (tid >> 3)] = bias;
}

// Conv weights are rounded to bf16 in the working copy the forward pass uses.
__device__ __forceinline__ float working_value(int i, float master) {
    const bool conv_w = i < kOffB1 || (i >= kOffW2 && i < kOffB2) || (i >= kOffW3 && i < kOffB3);
    return conv_w ? __bfloat162float(__float2bfloat16_rn(master)) : master;
}
__global__ void t_round(const float *__restrict__ master, float *__restrict__ wr, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        wr[i] = working_value(i, master[i]);
}

// ---- the gradient from the blocks' partials (8 warps of a block take every
// 8th partial of 32 parameters, then add up in order), Adam on the fp32 master
// parameters (lr > 0) and their working copy.
__global__ void __launch_bounds__(256) t_finish(const float *__restrict__ p1, int n1, const float *__restrict__ p2,
                                                int n2, const float *__restrict__ p3, int n3,
                                                const float *__restrict__ ps, int ns, float *__restrict__ grad,
                                                float *__restrict__ p, float *__restrict__ m, float *__restrict__ v,
                                                float *__restrict__ wr, float lr, float b1, float b2, float eps,
                                                float c1, float c2) {
    __shared__ float red[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    const float *src = nullptr;
    int n = 0, stride = 0;
    if (i < kOffW2) {  // w1, b1
        src = p1 + i; n = n1; stride = kW1Parts;
    } else if (i < kOffW3) {  // w2, b2
        src = p2 + (i - kOffW2); n = n2; stride = kOffW3 - kOffW2;
    } else if (i < kOffWh) {  // w3, b3
        src = p3 + (i - kOffW3); n = n3; stride = kOffWh - kOffW3;
    } else if (i < kCnnParams) {  // wh, bh, V, bv
        const int k = i < kOffV ? 129 + (i - kOffWh) : i - kOffV;
        src = ps + k; n = ns; stride = kSmallParts;
    }
    float s = 0.f;
#pragma unroll 4
    for (int b = warp; b < n; b += 8) s += src[(int64_t)b * stride];
    red[warp][lane] = s;
    __syncthreads();
    if (warp || i >= kCnnParams) return;
    float gi = red[0][lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) gi += red[k][lane];
    grad[i] = gi;
    if (lr > 0.f) {
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pn = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        p[i] = pn;
        wr[i] = working_value(i, pn);
    }
}

constexpr size_t conv23_smem(int cin) { return cin == 16 ? sizeof(ConvSmem<16>) : sizeof(ConvSmem<32>); }
constexpr size_t kDz2Smem = sizeof(Dz2Smem);
static_assert(2 * (kDz2Smem + 1024) <= 228 * 1024, "two blocks per SM");
constexpr size_t kDw1Smem = sizeof(Dw1Smem);
static_assert(kDw1Smem <= 227 * 1024, "one block per SM");
constexpr size_t dw23_smem(int cin) { return cin == 16 ? 2 * sizeof(Dw23Stage<16>) : 2 * sizeof(Dw23Stage<32>); }
static_assert(dw23_smem(16) >= 72 * 192 * 4 && dw23_smem(32) >= 72 * 128 * 4, "the parts' exchange fits");

}  // namespace

cudaError_t init_train() {
    cudaError_t e = cudaFuncSetAttribute(t_conv23<16, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)conv23_smem(16));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(t_conv23<32, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)conv23_smem(32));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(t_dz2, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDz2Smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(t_dw1, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDw1Smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(t_dw23<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dw23_smem(16));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(t_dw23<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dw23_smem(32));
    return e;
}

size_t train_partial_floats() {
    return (size_t)kTrainBlocks * (kW1Parts + (kOffW3 - kOffW2) + (kOffWh - kOffW3) + kSmallParts);
}

cudaError_t launch_train_step(cudaStream_t s, const TrainArgs &a) {
    const dim3 blk(256);
    const int nl = a.n_levels;
    if (nl <= 0) return cudaSuccess;
    // persistent blocks: a fixed number, so that the sums' order does not depend on the device
    constexpr int G = kTrainBlocks;
    float *p1 = a.part, *p2 = p1 + (size_t)G * kW1Parts, *p3 = p2 + (size_t)G * (kOffW3 - kOffW2),
          *ps = p3 + (size_t)G * (kOffWh - kOffW3);
    // forward
    t_conv1<<<4 * G, blk, 0, s>>>(a.tl, nl, a.tiles[0], a.levels, a.pyr, a.w.in_tab, a.wr + kOffW1, a.wr + kOffB1,
                                  a.act16);
    t_conv23<16, false><<<3 * G, 128, conv23_smem(16), s>>>(a.tl, nl, a.tiles[0], a.act16, a.wr + kOffW2,
                                                            a.wr + kOffB2, a.act16, nullptr, nullptr, nullptr, nullptr,
                                                            nullptr, 0);
    t_conv23<32, true><<<3 * G, 128, conv23_smem(32), s>>>(a.tl, nl, a.tiles[2], a.act16, a.wr + kOffW3,
                                                           a.wr + kOffB3, nullptr, a.act32, a.levels, a.wr + kOffWh,
                                                           a.wr + kOffBh, a.hmap, a.hp);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // pooling forward: the inference pooling kernel (identical sums) over the
    // batch's levels (the training levels are all levels of the batch, in order)
    CnnWeights pw = a.w;
    pw.v = a.wr + kOffV;
    pw.bv = a.wr + kOffBv;
    e = launch_cnn(s, a.levels, nl, nullptr, nullptr, 0, pw, a.hmap, a.hp, a.logits, a.pool_tiles, nullptr);  // pooling only
    if (e != cudaSuccess) return e;
    // loss and backward
    t_loss<<<dim3(kLossParts, nl), 256, 0, s>>>(a.tl, a.levels, a.logits, a.scores, a.label_thr, a.pos_weight, a.inv_n,
                                                a.dz, a.level_loss);
    t_pool_bwd_h<<<dim3(48, nl), blk, 0, s>>>(a.tl, a.levels, a.dz, a.wr + kOffV, a.dh, a.hp);
    t_small_grads<<<G, blk, 0, s>>>(a.tl, nl, a.tiles[4], a.tiles[2], a.levels, a.dz, a.hmap, a.dh, a.hp,
                                     a.wr + kOffWh, a.act32, ps);  // and a3 becomes dz3
    t_dw23<32><<<G, 256, dw23_smem(32), s>>>(a.tl, nl, a.tiles[3], a.act16, a.act32, p3);
    t_dz2<<<G, blk, kDz2Smem, s>>>(a.tl, nl, a.tiles[3], a.act32, a.wr + kOffW3, a.act16, a.dz2);
    t_dw23<16><<<G, 256, dw23_smem(16), s>>>(a.tl, nl, a.tiles[1], a.act16, a.dz2, p2);
    t_dw1<<<G, 256, kDw1Smem, s>>>(a.tl, nl, a.tiles[0], a.levels, a.pyr, a.w.in_tab, a.wr + kOffW2, a.act16, a.dz2,
                                   p1);
    t_finish<<<(kCnnParams + 31) / 32, blk, 0, s>>>(p1, G, p2, G, p3, G, ps, G, a.grad, a.master, a.m, a.v, a.wr, a.lr,
                                                    a.beta1, a.beta2, a.eps, a.c1, a.c2);
    return cudaGetLastError();
}

cudaError_t launch_round_params(cudaStream_t s, const float *master, float *wr) {
    t_round<<<64, 256, 0, s>>>(master, wr, kCnnParams);
    return cudaGetLastError();
}

}  // namespace pd
