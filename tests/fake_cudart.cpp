// A CUDA runtime that runs nothing: what the library's host code asks of it is written down, so that the order of its calls
// can be tested without a GPU.  Linked with the library's own objects in place of the real runtime.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {
std::map<const void*, std::string> names;                   // host stub -> device name
std::map<std::pair<int, const void*>, size_t> smem_allowed; // (device, kernel), as cudaFuncSetAttribute left it
std::set<std::pair<int, const void*>> in_flight;            // (device, target): work on the default stream that the host has not waited for
int device = 0, capturing = 0;
std::string events;
void* last_alloc = nullptr;
std::vector<std::pair<char*, size_t>> allocations;

void note(const std::string& s) { events += s + "\n"; }

cudaError_t refused_in_capture(const char* what) {
    if (!capturing) return cudaSuccess;
    note(std::string("refused ") + what);
    return cudaErrorStreamCaptureUnsupported;
}

cudaError_t launch(const void* f, size_t smem, cudaStream_t stream) {
    const auto allowed = smem_allowed.find({device, f});
    if (smem > (allowed == smem_allowed.end() ? 48u * 1024u : allowed->second)) {
        note("shared memory not allowed: " + names[f]);
        return cudaErrorInvalidValue;
    }
    size_t unordered = 0;                                   // (a stream of the caller's own need not wait for the default stream)
    for (const auto& c : in_flight) unordered += stream != nullptr && c.first == device;
    note("launch " + names[f] + " device " + std::to_string(device) + " unordered " + std::to_string(unordered));
    return cudaSuccess;
}
}  // namespace

extern "C" {
// for the test
void fake_reset() { events.clear(); capturing = 0; }
void fake_capture(int on) { capturing = on; }
void* fake_last_alloc() { return last_alloc; }
const char* fake_events() { return events.c_str(); }

// registration, called when the library is loaded
void** __cudaRegisterFatBinary(void*) { static void* handle; return &handle; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names[host] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void* stream) {
    *smem = 0;
    *static_cast<cudaStream_t*>(stream) = nullptr;
    return cudaSuccess;
}

cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { device = d; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) smem_allowed[{device, f}] = (size_t)v;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) { *n = 4; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 32; return cudaSuccess; }

cudaError_t cudaMalloc(void** p, size_t n) {
    const cudaError_t e = refused_in_capture("cudaMalloc");
    if (e == cudaSuccess) {
        *p = last_alloc = std::calloc(1, n);
        allocations.push_back({static_cast<char*>(*p), n});
    }
    return e;
}
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) {           // returns before the device has done it
    std::memset(d, v, n);
    in_flight.insert({device, d});
    return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { static char array[1 << 20]; *p = last_alloc = array; return cudaSuccess; }
// from pageable memory: returns when the source has been staged, not when the device has the bytes
cudaError_t cudaMemcpyToSymbol(const void* symbol, const void*, size_t, size_t, cudaMemcpyKind) {
    const cudaError_t e = refused_in_capture("cudaMemcpyToSymbol");
    if (e == cudaSuccess) in_flight.insert({device, symbol});
    return e;
}
cudaError_t cudaStreamSynchronize(cudaStream_t stream) {
    const cudaError_t e = refused_in_capture("cudaStreamSynchronize");
    if (e == cudaSuccess && stream == nullptr)
        for (auto it = in_flight.begin(); it != in_flight.end();) it = it->first == device ? in_flight.erase(it) : std::next(it);
    return e;
}

cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t smem, cudaStream_t stream) {
    if (names[f].find("bucket_norm_kernel") != std::string::npos) {     // where the norms go: which allocation, which byte of it
        const char* norms = *static_cast<char**>(args[4]);
        for (size_t i = 0; i < allocations.size(); ++i)
            if (norms >= allocations[i].first && norms < allocations[i].first + allocations[i].second)
                note("norms in allocation " + std::to_string(i) + " of " + std::to_string(allocations.size()));
    }
    return launch(f, smem, stream);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->dynamicSmemBytes, c->stream); }
}
