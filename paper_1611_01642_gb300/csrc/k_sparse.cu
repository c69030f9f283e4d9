// Sparse path: which tiles the learned proposal keeps.
//
// A window is kept when its keep-logit exceeds the keep threshold. For the
// FP32 K4 one warp per window tile of its plan decides whether the tile holds
// a kept window; a kept tile marks every K2+K3 cell tile its cell region
// overlaps, and K4 computes the kept tiles (their windows are all scored
// exactly; the others get -inf, which never becomes an NMS candidate). For the
// tensor-core K4 each kept window marks only the cell tiles under its own
// 8 x 16 cells, and K4 scores every window whose cells were all computed; one
// thread per window does both this and the -inf that the skipped windows keep
// (bound by reading the logits and writing the scores). Flags are plain stores
// of 1, so they do not depend on the order of the threads. Either way every
// kept window is scored exactly, so the recall is at least that of the
// window-level proposal.
#include "pd_internal.h"

namespace pd {
namespace {

__constant__ int2 kShapeDims[kSvmShapes] = {{32, 16}, {64, 8}, {32, 8}, {64, 4}, {64, 2}, {32, 12}, {32, 4}};

__global__ void __launch_bounds__(256) k_proposal_flags(const LevelDesc *__restrict__ levels,
                                                        const SvmItem *__restrict__ s_items, int n_items,
                                                        const float *__restrict__ logits, float tau,
                                                        uint32_t *__restrict__ s_flag, uint32_t *__restrict__ c_flag) {
    const int lane = threadIdx.x & 31;
    const int item = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (item >= n_items) return;
    const SvmItem it = s_items[item];
    const LevelDesc L = levels[it.level];
    const int2 d = kShapeDims[it.shape];
    bool any = false;
    for (int i = lane; i < d.x * d.y; i += 32) {
        const int wy = it.wy0 + i / d.x, wx = it.wx0 + i % d.x;
        any |= wy < L.rows && wx < L.cols && logits[L.score_off + (int64_t)wy * L.cols + wx] > tau;
    }
    any = __any_sync(0xffffffffu, any);
    if (lane == 0) s_flag[item] = any ? 1u : 0u;
    if (!any) return;
    // cells of the tile's windows: rows wy0 .. wy0+TH+14, columns wx0 .. wx0+TW+6
    const int cy_end = min(it.wy0 + d.y + kWinBH, L.Hc), cx_end = min(it.wx0 + d.x + kWinBW, L.Wc);
    const int ty0 = it.wy0 / kCellTH, ty1 = (cy_end - 1) / kCellTH;
    const int tx0 = it.wx0 / kCellTW, tx1 = (cx_end - 1) / kCellTW;
    const int ntx = tx1 - tx0 + 1, n = (ty1 - ty0 + 1) * ntx;
    for (int k = lane; k < n; k += 32) {
        const int ty = ty0 + k / ntx, tx = tx0 + k % ntx;
        c_flag[L.citem0 + ty * L.ctx + tx] = 1u;
    }
}

// Block (x, y): every gridDim.x-th run of windows of level y.
__global__ void __launch_bounds__(256) k_window_flags(const LevelDesc *__restrict__ levels,
                                                      const float *__restrict__ logits, float tau,
                                                      uint32_t *__restrict__ c_flag, float *__restrict__ scores) {
    const LevelDesc &L = levels[blockIdx.y];
    const int n = L.rows * L.cols, cols = L.cols, ctx = L.ctx;
    const float *z = logits + L.score_off;
    float *out = scores + L.score_off;
    uint32_t *flags = c_flag + L.citem0;
    constexpr int kU = 4;  // loads in flight per thread
    for (int i0 = blockIdx.x * 256 * kU + threadIdx.x; i0 < n; i0 += gridDim.x * 256 * kU) {
        float v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) v[u] = i0 + u * 256 < n ? __ldg(z + i0 + u * 256) : -INFINITY;
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int i = i0 + u * 256;
            if (i >= n) continue;
            out[i] = -INFINITY;
            if (!(v[u] > tau)) continue;
            // cell tiles under cell rows wy .. wy+15, columns wx .. wx+7
            const int wy = i / cols, wx = i - wy * cols;
            for (int ty = wy / kCellTH; ty <= (wy + kWinBH) / kCellTH; ++ty)
                for (int tx = wx / kCellTW; tx <= (wx + kWinBW) / kCellTW; ++tx) flags[ty * ctx + tx] = 1u;
        }
    }
}

}  // namespace

cudaError_t launch_window_flags(cudaStream_t s, const LevelDesc *d_levels, int n_levels, int max_windows,
                                const float *logits, float tau, uint32_t *c_flag, float *scores) {
    if (n_levels <= 0 || max_windows <= 0) return cudaSuccess;
    const int gx = max_windows >= 32 * 1024 ? 32 : (max_windows + 1023) / 1024;
    for (int l0 = 0; l0 < n_levels; l0 += 65535) {  // grid.y limit
        const int nl = n_levels - l0 < 65535 ? n_levels - l0 : 65535;
        k_window_flags<<<dim3(gx, nl), 256, 0, s>>>(d_levels + l0, logits, tau, c_flag, scores);
    }
    return cudaGetLastError();
}

cudaError_t launch_proposal_flags(cudaStream_t s, const LevelDesc *d_levels, const SvmItem *d_items, int n_items,
                                  const float *logits, float tau, uint32_t *s_flag, uint32_t *c_flag) {
    if (n_items <= 0) return cudaSuccess;
    k_proposal_flags<<<(n_items + 7) / 8, 256, 0, s>>>(d_levels, d_items, n_items, logits, tau, s_flag, c_flag);
    return cudaGetLastError();
}

}  // namespace pd
