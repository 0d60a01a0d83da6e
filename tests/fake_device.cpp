// A device made of host memory, for tests of the library's host side (npx_world.cpp) without a GPU:
// two SMs, three resident blocks of any shape with the points in the slots and eight with them in
// global memory.  Launches are recorded, not run; allocations of one size can be made to fail.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <vector>

#include "../include/npx_mlp.h"
#include "../paper_2411_05799_gb300/csrc/npx_internal.h"

namespace {
std::map<char *, size_t> g_alloc;
size_t g_fail_bytes = 0;
struct Launch {
    int gp, steps, blocks, warps;
    long long room, first;   // scratch points from the launch's first one on; its address in points
};
std::vector<Launch> g_launches;
}  // namespace

extern "C" {
void fake_fail_bytes(size_t n) { g_fail_bytes = n; }
void fake_clear() { g_launches.clear(); }
int fake_launches(long long *out, int n) {
    int k = 0;
    for (const Launch &l : g_launches) {
        if (k == n) break;
        const long long v[6] = {l.gp, l.steps, l.blocks, l.warps, l.room, l.first};
        memcpy(out + 6 * k++, v, sizeof v);
    }
    return (int)g_launches.size();
}

cudaError_t cudaMalloc(void **p, size_t n) {
    if (n == g_fail_bytes) return cudaErrorMemoryAllocation;
    char *q = static_cast<char *>(aligned_alloc(256, (n + 255) & ~size_t(255)));
    g_alloc[q] = n;
    *p = q;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (p && !g_alloc.erase(static_cast<char *>(p))) return cudaErrorInvalidValue;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int *n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 2; return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t *g) { *g = nullptr; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t *e, cudaGraph_t, unsigned long long) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
}

namespace npx {
int step_blocks_per_sm(const WorldDev &, int, int, int gp, cudaError_t *err) { *err = cudaSuccess; return gp ? 8 : 3; }
bool step_fits_bare(const WorldDev &, int, int) { return true; }
bool step_has_gp(const WorldDev &W, int) { return !W.hm && !W.fric_mode && W.arena <= 1; }
cudaError_t launch_step(const WorldDev &W, const LaunchCfg &c, int n, cudaStream_t) {
    Launch l{c.gp, n, c.blocks, c.wpb, 0, 0};
    char *p = reinterpret_cast<char *>(W.pscr);
    for (const auto &a : g_alloc)
        if (c.gp && p >= a.first && p < a.first + a.second) {
            l.room = (a.first + a.second - p) / 16;
            l.first = (p - a.first) / 16;
        }
    g_launches.push_back(l);
    return c.gp && !p ? cudaErrorInvalidValue : cudaSuccess;
}
#define OK \
    { return cudaSuccess; }
cudaError_t launch_advance(long long *, int, cudaStream_t) OK
cudaError_t launch_init(const WorldDev &, const float *, const float *, const float *, const float *, cudaStream_t) OK
cudaError_t launch_refresh(const WorldDev &, cudaStream_t) OK
cudaError_t launch_scatter_state(const WorldDev &, const float *, cudaStream_t) OK
cudaError_t launch_gather_state(const WorldDev &, float *, cudaStream_t) OK
cudaError_t launch_permute_kappa(uint8_t *, const uint8_t *, const int *, int, bool, cudaStream_t) OK
cudaError_t launch_sensor_points(const WorldDev &, int *, int *, cudaStream_t) OK
cudaError_t launch_sensor_index(const WorldDev &, const SurCache &, cudaStream_t) OK
cudaError_t launch_shape_cache(const WorldDev &, const SurCache &, cudaStream_t) OK
cudaError_t launch_features(const WorldDev &, const SurCache &, const SurrogateIO &, cudaStream_t) OK
cudaError_t launch_surrogate_update(const WorldDev &, const SurCache &, const float *, int, const float *, const float *,
                                    float *, uint8_t *, uint32_t *, int *, int *, int *, int, cudaStream_t) OK
cudaError_t launch_kappa_refresh(const WorldDev &, const int *, const int *, cudaStream_t) OK
cudaError_t launch_accumulate(long long *, int *, int, cudaStream_t) OK
cudaError_t launch_points(const WorldDev &, int, float *, cudaStream_t) OK
cudaError_t launch_hm_dilate(const float *, float *, float *, int, int, int, int, cudaStream_t) OK
void encode_hm_tmap(WorldDev &, int, CUtensorMap *) {}
cudaStream_t mlp_stream(const npx_mlp *) { return nullptr; }
int mlp_max_batch(const npx_mlp *) { return 0; }
void mlp_dims(const npx_mlp *, int *, int *) {}
__nv_bfloat16 *mlp_input(npx_mlp *, int *) { return nullptr; }
int mlp_forward_packed(npx_mlp *, int, int) { return 0; }
const float *mlp_output(const npx_mlp *, int *) { return nullptr; }
}  // namespace npx
