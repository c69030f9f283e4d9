// A CUDA runtime without a GPU, for the host code of pd_api.cu: "device" memory is host
// memory, and one in-order queue holds what was enqueued until somebody waits for it.
// That is the latest a device may run its work, so a pinned buffer that is rewritten
// before the copy out of it has been waited for shows in what the "kernels" read.
// launch_resize logs the frames and levels that the pyramid kernel would see.
// Built and run by tests/test_descriptor_upload_cpu.py.
#include <cudaTypedefs.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <vector>

#include "../../paper_1611_01642_gb300/csrc/pd_internal.h"

namespace {
using Op = std::function<void()>;
std::vector<Op> queue_;       // enqueued, not yet run
size_t done_ = 0;             // operations run
std::vector<Op> *capture_ = nullptr;
void run_to(size_t n) {
    for (; done_ < n && done_ < queue_.size(); ++done_) queue_[done_]();
}
cudaError_t put(Op f) {
    (capture_ ? *capture_ : queue_).push_back(std::move(f));
    return cudaSuccess;
}
struct Event {
    size_t at = 0;  // waits for the operations before this one
};
Event *ev(cudaEvent_t e) { return reinterpret_cast<Event *>(e); }
CUresult encode(CUtensorMap *map, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    std::memset(map, 0, sizeof *map);
    return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
cudaError_t cudaGetDevice(int *d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char *, void **p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult *q) {
    *p = reinterpret_cast<void *>(&encode);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
const char *cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaMalloc(void **p, size_t n) { return *p = std::aligned_alloc(1024, (n + 1023) / 1024 * 1024), cudaSuccess; }
cudaError_t cudaFree(void *p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void *p) { return cudaFree(p); }
cudaError_t cudaHostGetDevicePointer(void **d, void *h, unsigned) { return *d = h, cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *a, const void *) { return *a = {}, cudaErrorInvalidValue; }
cudaError_t cudaDeviceSynchronize() { return run_to(queue_.size()), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaDeviceSynchronize(); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) {
    cudaDeviceSynchronize();
    return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemset(void *d, int v, size_t n) {
    cudaDeviceSynchronize();
    return std::memset(d, v, n), cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    return put([=] { std::memcpy(d, s, n); });
}
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) {
    return put([=] { std::memset(d, v, n); });
}
cudaError_t cudaMemcpy2DAsync(void *d, size_t dp, const void *s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
    return put([=] {
        for (size_t y = 0; y < h; ++y) std::memcpy((char *)d + y * dp, (const char *)s + y * sp, w);
    });
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    return *e = reinterpret_cast<cudaEvent_t>(new Event), cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t *e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return delete ev(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { return ev(e)->at = queue_.size(), cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return run_to(ev(e)->at), cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
    return capture_ = new std::vector<Op>, cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) {
    *g = reinterpret_cast<cudaGraph_t>(capture_);
    return capture_ = nullptr, cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *x, cudaGraph_t g, unsigned long long) {
    *x = reinterpret_cast<cudaGraphExec_t>(new std::vector<Op>(*reinterpret_cast<std::vector<Op> *>(g)));
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
    for (const Op &f : *reinterpret_cast<std::vector<Op> *>(x)) put(f);
    return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return delete reinterpret_cast<std::vector<Op> *>(x), cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return delete reinterpret_cast<std::vector<Op> *>(g), cudaSuccess; }
}

namespace pd {
cudaError_t init_resize() { return cudaSuccess; }
cudaError_t init_cells_warp() { return cudaSuccess; }
cudaError_t init_svm() { return cudaSuccess; }
cudaError_t init_svm_tc() { return cudaSuccess; }
cudaError_t init_nms(bool) { return cudaSuccess; }
cudaError_t init_train() { return cudaSuccess; }
cudaError_t init_cnn() { return cudaSuccess; }
SvmShapeInfo svm_shape(int) { return {32, 16, 48, 48, 31}; }
int svm_lbp_chunk() { return 59; }
void build_tc_consts(const float *, unsigned char *) {}
int encode_tc_maps(CUtensorMap *, CUtensorMap *, const float *, int64_t, int64_t, int, const uint8_t *, int64_t, int64_t,
                   int64_t) {
    return PD_OK;
}
int nms_cluster_for(int, int, int, int64_t windows) {
    std::fprintf(stderr, "windows %ld\n", (long)windows);
    return 1;
}
int nms_launches(int, int) { return 1; }
size_t train_partial_floats() { return 0; }
size_t scheme_cells_scratch(int, int) { return 0; }
size_t scheme_scores_scratch(int, int) { return 0; }
cudaError_t launch_resize(cudaStream_t, const FrameDesc *f, const LevelDesc *l, const int32_t *, uint8_t *,
                          const ResizeItem *items, int n, bool, int, int *) {
    return put([=] {
        int last = -1;
        for (int i = 0; i < n; ++i) {
            const FrameDesc &d = f[items[i].frame];
            if (items[i].frame == last) continue;
            last = items[i].frame;
            std::printf("K1 frame %d: ptr %lx %dx%d, %d levels, last %dx%d\n", last, (unsigned long)(uintptr_t)d.ptr, d.W,
                        d.H, d.n_levels, l[d.first_level + d.n_levels - 1].Wk, l[d.first_level + d.n_levels - 1].Hk);
        }
    });
}
cudaError_t launch_cells_warp(cudaStream_t, const LevelDesc *l, const uint8_t *, CellAtlas, const StripItem *it, int n,
                              int *, int, const uint32_t *, int) {
    return put([=] {
        if (n) std::printf("K23 level %dx%d\n", l[it[0].level].Wk, l[it[0].level].Hk);
    });
}
cudaError_t launch_proposal_flags(cudaStream_t, const LevelDesc *, const SvmItem *, int, const float *, float, uint32_t *,
                                  uint32_t *) {
    return cudaSuccess;
}
cudaError_t launch_svm(cudaStream_t, const CUtensorMap *, const CUtensorMap *, const LevelDesc *, const float *, float,
                       float, float *, const SvmItem *, int, unsigned *, const uint32_t *) {
    return cudaSuccess;
}
cudaError_t launch_lbp_cells(cudaStream_t, const uint8_t *, int64_t, int, int, int, uint8_t *) { return cudaSuccess; }
cudaError_t launch_svm_tc(cudaStream_t, const CUtensorMap &, const CUtensorMap &, const LevelDesc *, const TcItem *, int,
                          int *, int, const unsigned char *, float, float, float *, const uint32_t *, unsigned *, int,
                          const CUtensorMap *) {
    return cudaSuccess;
}
cudaError_t launch_nms(cudaStream_t, const FrameDesc *, const LevelDesc *, int, const float *, float, float, float4 *,
                       int, pd_box *, int, int32_t *, int, int *, const unsigned *, unsigned *) {
    return cudaSuccess;
}
cudaError_t launch_cnn(cudaStream_t, const LevelDesc *, int, const CUtensorMap *, const CnnItem *, int,
                       const CnnWeights &, float *, int32_t, float *, int, unsigned *, float, uint32_t *, float *) {
    return cudaSuccess;
}
cudaError_t launch_train_step(cudaStream_t, const TrainArgs &) { return cudaSuccess; }
cudaError_t launch_round_params(cudaStream_t, const float *, float *) { return cudaSuccess; }
cudaError_t launch_scheme_cells(cudaStream_t, int, const uint8_t *, int, int, int, float *, int64_t, uint8_t *, int64_t,
                                int, const uint8_t *, unsigned char *, bool) {
    return cudaSuccess;
}
cudaError_t launch_scheme_scores(cudaStream_t, int, const float *, int64_t, const uint8_t *, int64_t, int, int, int,
                                 const float *, float, float, float *, unsigned char *, bool) {
    return cudaSuccess;
}
}  // namespace pd

// Arguments: the calls to make, none of them waited for: A, B (pd_detect of one or two
// frames), C (pd_cell_features of one level).
int main(int argc, char **argv) {
    pd_params p;
    pd_params_default(&p);
    p.max_frames = 2;
    p.max_width = 320;
    p.max_height = 240;
    std::vector<float> w(PD_TEMPLATE_SIZE, 0.f);
    pd_handle *h = nullptr;
    if (pd_create(&p, w.data(), 0.f, &h) != PD_OK) return 2;
    const uint8_t *fa[1] = {(const uint8_t *)0xa000}, *fb[2] = {(const uint8_t *)0xb000, (const uint8_t *)0xb800};
    const int32_t wa[1] = {320}, ha[1] = {240}, wb[2] = {200, 160}, hb[2] = {180, 150};
    std::vector<float> hog(9 * 20 * 16);
    std::vector<uint8_t> lbp(59 * 20 * 16);
    for (int i = 1; i < argc; ++i) {
        int r = PD_OK;
        if (argv[i][0] == 'A') r = pd_detect(h, nullptr, 1, fa, wa, ha, wa);
        if (argv[i][0] == 'B') r = pd_detect(h, nullptr, 2, fb, wb, hb, wb);
        if (argv[i][0] == 'C')
            r = pd_cell_features(h, nullptr, (const uint8_t *)0xc000, 128, 160, 128, hog.data(), 20 * 16, lbp.data(),
                                 20 * 16, 16);
        if (r != PD_OK) {
            std::printf("call %d: %d %s\n", i, r, pd_last_error(h));
            return 1;
        }
    }
    cudaDeviceSynchronize();
    pd_destroy(h);
    return 0;
}
