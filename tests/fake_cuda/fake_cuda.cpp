// The CUDA runtime calls and kernel launchers of the library's host code, on host memory: a batch's
// classes, launch shapes, chunks and allocations can be tested without a GPU.  "Device" memory comes
// from malloc under a budget, copies and clears happen at once, and a batch launch is not run: what
// it was given is written to a log (see Launch).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "mcpd.h"
#include "mcpd_internal.h"

namespace {
size_t g_budget = size_t(1) << 40, g_live = 0;
long long g_allocs_left = -1;          // allocations that succeed before all fail (-1: no limit)
int g_device = 0;
cudaError_t g_last = cudaSuccess;
std::map<char *, size_t> g_blocks;
// One launch: lanes, grid, warps per block, bank, total chunks, instances, words of its scratch that
// are allocated, words of marks per entry; then per instance: slots, first chunk, chunks, clones.
std::vector<long long> g_log;

size_t room_at(const void *p) {
    char *c = static_cast<char *>(const_cast<void *>(p));
    auto it = g_blocks.upper_bound(c);
    if (it == g_blocks.begin()) return 0;
    --it;
    return c < it->first + it->second ? static_cast<size_t>(it->first + it->second - c) : 0;
}
}  // namespace

extern "C" {
void fake_budget(long long bytes) { g_budget = static_cast<size_t>(bytes); }
void fake_allocs(long long left) { g_allocs_left = left; }
long long fake_live() { return static_cast<long long>(g_live); }
int fake_device(int set) { if (set >= 0) g_device = set; return g_device; }
long long fake_log(long long *out, long long cap) {
    const long long n = static_cast<long long>(g_log.size());
    for (long long i = 0; i < std::min(n, cap); ++i) out[i] = g_log[static_cast<size_t>(i)];
    return n;
}
void fake_stage(mcpd_ctx *ctx) {       // as a call of mcpd_features_batch leaves it
    ctx->stage_host = std::malloc(64);
    cudaMalloc(&ctx->stage_dev, 64);
    ctx->stage_bytes = 64;
}
void fake_clear_log() { g_log.clear(); }

cudaError_t cudaMalloc(void **p, size_t bytes) {
    if (g_live + bytes > g_budget || g_allocs_left == 0) return g_last = cudaErrorMemoryAllocation;
    if (g_allocs_left > 0) --g_allocs_left;
    char *c = static_cast<char *>(std::malloc(bytes ? bytes : 1));   // pages are taken only where they are touched
    if (!c) return g_last = cudaErrorMemoryAllocation;
    g_blocks[c] = bytes;
    g_live += bytes;
    *p = c;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (!p) return cudaSuccess;
    auto it = g_blocks.find(static_cast<char *>(p));
    if (it == g_blocks.end()) return g_last = cudaErrorInvalidValue;
    g_live -= it->second;
    g_blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) {
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void *d, int, size_t n, cudaStream_t) {
    // a clear beyond its allocation is the error that the tests look for; large ones only touch their ends
    if (room_at(d) < n) return g_last = cudaErrorInvalidValue;
    std::memset(d, 0, std::min(n, size_t(1) << 20));
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) { g_device = d; return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = g_device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = g_last; g_last = cudaSuccess; return e; }
const char *cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = reinterpret_cast<cudaGraph_t>(1); return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) {
    *e = reinterpret_cast<cudaGraphExec_t>(1);
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
int mcpd_decode_noalloc(mcpd_ctx *, const mcpd_design *, const uint8_t *, const mcpd_params *, double *, double *, mcpd_stats *) { return MCPD_ECUDA; }
}  // extern "C"

namespace mcpd {
// As the launch shapes of the kernels come out on a GB300: registers allow one block per SM.
int pairs_shape(int, int, int, bool batch, size_t tables, int wpp, size_t smem_optin, long long P, int sm_count,
                int warps, bool, bool, PairsShape *out) {
    int w = 0;
    while (w < (batch ? 16 : 20) && pairs_smem_bytes(tables, wpp, w + 1) <= smem_optin) ++w;
    if (w < 2) return MCPD_ETOO_LARGE;
    if (warps > w) return MCPD_EINVAL;
    if (warps > 0) w = warps;
    else if (P > 0) w = chunk_shape(P, sm_count, w, kBank).warps;
    out->warps = w;
    out->per_sm = 1;
    out->smem = pairs_smem_bytes(tables, wpp, w);
    return MCPD_OK;
}
int batch_kernel_degree(int coupled, int, int udeg) { return coupled && udeg >= 3 && udeg <= 8 ? udeg : 0; }
static int log_launch(const BParams &bp, int grid, int block) {
    const size_t words = room_at(bp.pair_scratch) / 8;
    for (long long v : {static_cast<long long>(bp.lanes), static_cast<long long>(grid), static_cast<long long>(block / 32),
                        static_cast<long long>(bp.bank), bp.total_units, static_cast<long long>(bp.n_inst),
                        static_cast<long long>(words), static_cast<long long>(bp.marks)})
        g_log.push_back(v);
    for (int i = 0; i < bp.n_inst; ++i)
        for (long long v : {bp.insts[i].P, bp.insts[i].unit_begin, bp.insts[i].units, static_cast<long long>(bp.insts[i].na)})
            g_log.push_back(v);
    return MCPD_OK;
}
int launch_batch(const BParams &bp, int grid, int block, size_t, void *) { return cudaGetLastError() == cudaSuccess ? log_launch(bp, grid, block) : MCPD_ECUDA; }
int launch_group(const BParams &bp, int grid, int block, size_t, void *) { return cudaGetLastError() == cudaSuccess ? log_launch(bp, grid, block) : MCPD_ECUDA; }
int launch_pairs(const KParams &kp, int grid, int block, size_t, void *) {
    if (cudaGetLastError() != cudaSuccess) return MCPD_ECUDA;
    for (long long v : {0ll, static_cast<long long>(grid), static_cast<long long>(block / 32), static_cast<long long>(kp.bank),
                        static_cast<long long>(kp.chunk), 1ll, static_cast<long long>(room_at(kp.pair_scratch) / 8), static_cast<long long>(kp.marks), kp.P, 0ll, 0ll,
                        static_cast<long long>(kp.na)})
        g_log.push_back(v);
    return MCPD_OK;
}
int launch_philox(const uint32_t *, uint32_t, uint32_t, uint32_t *, long long, void *) { return MCPD_ECUDA; }
int pairs_max_smem(int, size_t *bytes) { *bytes = 232448; return MCPD_OK; }
int set_group_smem(int, size_t) { return MCPD_OK; }
int group_occupancy(int, int, size_t, int *per_sm) { *per_sm = 1; return MCPD_OK; }
int group_max_threads(int) { return 512; }
int launch_finalize(const unsigned long long *, const unsigned long long *, const unsigned long long *, int, int, long long, long long, double *, double *, void *) { return MCPD_OK; }
int launch_finalize_batch(const InstDesc *, int, const int *, const int *, long long, double *, double *, void *) { return MCPD_OK; }
}  // namespace mcpd
