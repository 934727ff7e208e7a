// A CUDA runtime of host memory and kernels that do nothing, for tests of the library's host
// code on a machine without a GPU (test_host_alloc.py links it with the library's objects).
// Device memory is malloc'ed and zeroed, with a limit on the number of successful
// allocations; every kernel launch is recorded with its grid and the pointers that the test
// asks for.  Prototypes are those of the CUDA headers.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
std::map<char*, size_t> blocks;
long long left = -1;            // allocations until one fails (-1: none does)
size_t live_bytes = 0, peak_bytes = 0, room_bytes = size_t(270) << 30;
std::map<const void*, std::string> names;
cudaError_t last = cudaSuccess;
struct Launch {
    std::string name;
    unsigned grid;
    std::vector<void*> ptrs;   // see record()
};
std::vector<Launch> launches;
struct Config {
    dim3 grid, block;
    size_t smem;
    cudaStream_t s;
};
std::vector<Config> configs;

cudaError_t set(cudaError_t e) {
    if (e != cudaSuccess) last = e;
    return e;
}

// Tables in a Toeplitz kernel's arguments: TzArgs starts with tiles, twiddle, ptw, H; the
// persistent kernel has its own tables, spectra and scratch behind three integers.  Of a
// batched dot product the vectors and the result.
void record(const void* f, dim3 grid, void** args) {
    Launch l{names.count(f) ? names[f] : "?", grid.x * grid.y * grid.z, {}};
    auto word = [&](int arg, int at) { return *reinterpret_cast<void**>(static_cast<char*>(args[arg]) + 8 * at); };
    if (l.name.find("toeplitz_ws") != std::string::npos) l.ptrs = {word(0, 0), word(4, 0), word(5, 0), word(6, 0)};
    else if (l.name.find("toeplitz_os") != std::string::npos) l.ptrs = {word(0, 0), word(0, 3)};
    else if (l.name.find("dot_batch_kernel") != std::string::npos) l.ptrs = {word(0, 0), word(2, 0)};
    launches.push_back(l);
}

bool inside(const void* p) {
    auto it = blocks.upper_bound(const_cast<char*>(static_cast<const char*>(p)));
    if (it == blocks.begin()) return false;
    --it;
    return static_cast<const char*>(p) < it->first + it->second;
}
}  // namespace

extern "C" {

// ---- for the test
int fake_fail_after(long long n) {   // whether the failure asked for before has not come about
    const int pending = left >= 0;
    left = n;
    return pending;
}
long long fake_live_bytes() { return (long long)live_bytes; }
long long fake_peak_bytes(int reset) {
    if (reset) peak_bytes = live_bytes;
    return (long long)peak_bytes;
}
void fake_room(long long bytes) { room_bytes = (size_t)bytes; }   // free memory that is reported
void fake_clear_launches() { launches.clear(); }
int fake_launches() { return (int)launches.size(); }
const char* fake_launch_name(int i) { return launches[(size_t)i].name.c_str(); }
unsigned fake_launch_grid(int i) { return launches[(size_t)i].grid; }
// table pointers of launch i that do not point into live memory
int fake_launch_dead(int i) {
    int n = 0;
    for (void* p : launches[(size_t)i].ptrs) n += !inside(p);
    return n;
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t bytes) {
    if (left == 0) {
        left = -1;
        return set(cudaErrorMemoryAllocation);
    }
    if (left > 0) --left;
    char* q = static_cast<char*>(std::calloc(bytes + 256, 1));
    blocks[q] = bytes;
    live_bytes += bytes;
    if (live_bytes > peak_bytes) peak_bytes = live_bytes;
    *p = q;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
    auto it = blocks.find(static_cast<char*>(p));
    if (it == blocks.end()) std::abort();   // freed twice
    live_bytes -= it->second;
    blocks.erase(it);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) {
    *p = std::calloc(bytes, 1);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
    if (d == nullptr || s == nullptr) return set(cudaErrorInvalidValue);
    std::memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
    return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
    if (d == nullptr) return set(cudaErrorInvalidValue);
    std::memset(d, v, n);
    return cudaSuccess;
}
cudaError_t cudaMemGetInfo(size_t* room, size_t* total) {
    *total = size_t(280) << 30;
    *room = room_bytes;
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    std::memset(a, 0, sizeof *a);
    a->type = inside(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
    *p = const_cast<void*>(symbol);
    return cudaSuccess;
}

// ---- device, streams, events, errors
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char* cudaGetErrorString(cudaError_t) { return "error of the fake runtime"; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return set(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return set(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return set(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return set(cudaErrorNotSupported); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
    *e = reinterpret_cast<cudaEvent_t>(8);
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
    *ms = 1.f;
    return cudaSuccess;
}

// ---- kernels
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    record(f, c->gridDim, args);
    return cudaSuccess;
}
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 grid, dim3, void** args, size_t, cudaStream_t) {
    record(f, grid, args);
    return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
    configs.push_back({grid, block, smem, s});
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
    const Config c = configs.back();
    configs.pop_back();
    *grid = c.grid;
    *block = c.block;
    *smem = c.smem;
    *static_cast<cudaStream_t*>(s) = c.s;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
    return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void** args, size_t, cudaStream_t) {
    record(k, grid, args);
    return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* device, int, uint3*, uint3*, dim3*, dim3*, int*) {
    names[host] = device;
}
}
