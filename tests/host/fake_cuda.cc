// A CUDA runtime and kernel launchers for the library's host code alone, without a
// GPU: device memory is host memory (counted), launches do nothing, and a call can be
// made to fail. The tests compile it with the host sources of the library.
#include <cstdlib>
#include <cstring>
#include <map>

#include "../../paper_2007_12266_gb300/csrc/internal.h"
#include "../../paper_2007_12266_gb300/csrc/batch.h"

namespace {
std::map<void*, size_t> blocks;
size_t live = 0, peak = 0, limit = ~size_t{0};
long long launches = 0, refused = 0, uploads = 0;
int fail_in[2] = {0, 0};   // graph instantiation, graph launch: the call from now that fails
int handle = 0;
bool fails(int what) { return fail_in[what] > 0 && --fail_in[what] == 0; }
template <class T>
T next_handle() { return reinterpret_cast<T>(static_cast<size_t>(++handle) << 4); }
cudaError_t launched() {
    ++launches;
    return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_fail(int what, int nth) { fail_in[what] = nth; }
void fake_memory_limit(size_t bytes) { limit = bytes; }
void fake_reset_peak() { peak = live; }
size_t fake_peak() { return peak; }
size_t fake_live() { return live; }
long long fake_launches() { return launches; }
long long fake_refused() { return refused; }
long long fake_uploads() { return uploads; }

cudaError_t cudaMalloc(void** p, size_t n) {
    if (live + n > limit) {
        ++refused;
        return cudaErrorMemoryAllocation;
    }
    *p = std::calloc(n, 1);
    blocks[*p] = n;
    live += n;
    if (live > peak) peak = live;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    live -= blocks[p];
    blocks.erase(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* f, size_t* t) {
    *f = *t = size_t{280} << 30;
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    uploads += k == cudaMemcpyHostToDevice;
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
    std::memset(static_cast<void*>(p), 0, sizeof *p);
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorName(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "memory" : "error"; }
const char* cudaGetErrorString(cudaError_t e) { return cudaGetErrorName(e); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
    *s = next_handle<cudaStream_t>();
    return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
    *g = next_handle<cudaGraph_t>();
    return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
    if (fails(0)) return cudaErrorMemoryAllocation;
    *e = next_handle<cudaGraphExec_t>();
    return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return fails(1) ? cudaErrorUnknown : launched(); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = next_handle<cudaEvent_t>();
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.0f;
    return cudaSuccess;
}
}

namespace lbm {
cudaError_t launch_flag_pore(const uint16_t* l, long long V, int* f, cudaStream_t) {
    for (long long i = 0; i < V; ++i) f[i] = l[i] == 0;
    return cudaSuccess;
}
cudaError_t exclusive_scan(lbpm_ctx*, const int* in, int* out, long long n) {
    for (long long i = 0, s = 0; i < n; s += in[i++]) out[i] = static_cast<int>(s);
    return cudaSuccess;
}
cudaError_t copy_to_host(void* d, const void* s, size_t n, cudaStream_t st) {
    return cudaMemcpyAsync(d, s, n, cudaMemcpyDeviceToHost, st);
}
cudaError_t noalloc_setup(int) { return cudaSuccess; }
DomainView make_view(const lbpm_ctx*) { return DomainView{}; }
cudaError_t launch_measure(lbpm_ctx* c, int, const double** out, cudaStream_t) {
    static double sums[NSUM];
    *out = sums;
    return launched();
}
int batch_max_blocks(int, bool, int) { return 8; }
int batch_fused_blocks_per_sm(int, bool, int) { return 4; }
cudaError_t launch_batch_measure(bool, unsigned, cudaStream_t, const DomainView*, const int*, const BatchTile*, int,
                                 double*, const int*, int, double*) { return launched(); }
#define STUB(name, ...) \
    cudaError_t name(__VA_ARGS__) { return launched(); }
STUB(launch_scatter_sites, const lbpm_ctx*, const int*, cudaStream_t)
STUB(launch_fill_halo, const lbpm_ctx*, cudaStream_t)
STUB(launch_links, const lbpm_ctx*, cudaStream_t)
STUB(launch_affinity_table, const lbpm_ctx*, const float*, int, cudaStream_t)
STUB(launch_affinity_map, const lbpm_ctx*, const float*, cudaStream_t)
STUB(launch_slab_flags, const lbpm_ctx*, int*, cudaStream_t)
STUB(launch_slab_scatter, const lbpm_ctx*, const int*, const int*, cudaStream_t)
STUB(launch_export_index, const lbpm_ctx*, long long*, int*, cudaStream_t)
STUB(launch_init_fluids, const lbpm_ctx*, const float*, cudaStream_t)
STUB(launch_ref_sum, const lbpm_ctx*, int, cudaStream_t)
STUB(launch_phase, const lbpm_ctx*, int, bool, cudaStream_t)
STUB(launch_collide, const lbpm_ctx*, int, cudaStream_t)
STUB(launch_phase_sum, const lbpm_ctx*, int, cudaStream_t)
STUB(launch_collide_sum, const lbpm_ctx*, int, cudaStream_t)
STUB(launch_reservoir, const lbpm_ctx*, int, bool, cudaStream_t)
STUB(launch_morph, const lbpm_ctx*, int, float, int, int, float*, float*, float*, int3*, long long*, float*, int,
     unsigned long long*, cudaStream_t)
STUB(launch_field, const lbpm_ctx*, int, int, float*, cudaStream_t)
STUB(launch_export_dist, const lbpm_ctx*, int, int, float*, cudaStream_t)
STUB(launch_import_dist, const lbpm_ctx*, int, int, const float*, cudaStream_t)
STUB(launch_read_box, const lbpm_ctx*, int, int, const int*, const int*, float*, cudaStream_t)
STUB(launch_batch, int, int, int, bool, int, unsigned, cudaStream_t, const BatchLaunch&)
STUB(launch_batch_reservoir, int, bool, bool, cudaStream_t, const BatchSlabs&)
STUB(launch_batch_fused, int, bool, int, unsigned, cudaStream_t, const FusedLaunch&)
STUB(launch_barrier_probe, unsigned, unsigned, unsigned long long, unsigned*, int*, cudaStream_t)
}  // namespace lbm
