// Activations of the host-buffer calls from page-locked memory to the device stage, by a kernel.
//
// A decode step's inputs are a few KB.  A copy-engine transfer of that size costs two hand-overs between engine and SMs, about
// 10 us in a stream of 3 to 6 us kernels; here the SMs read the mapped buffer over the bus themselves (one 16-byte load per
// thread: the bus latency once) and the layer kernel behind is already resident, filling up with weights, under programmatic
// dependent launch.  A 7B-shaped decoder layer of seven projections in four calls: 90 us with copies, 60 so.
// Letting the layer kernel read host memory itself is slower still (194 us): every CTA fetches its slices over the bus.
#include "rabit_internal.h"

namespace {

constexpr int kThreads = 256;

struct FetchParams {
    const uint4* src[8];
    uint4* dst[8];
    int end[8];                     // running totals in 16-byte units
    int n;
};

__global__ void __launch_bounds__(kThreads) rabit_fetch_kernel(const __grid_constant__ FetchParams P) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int i = (int)(blockIdx.x * kThreads + threadIdx.x);
    int s = 0;
    while (s < P.n && i >= P.end[s]) ++s;
    asm volatile("griddepcontrol.wait;" ::: "memory");               // the stage may still be read by earlier work of the stream
    if (s >= P.n) return;
    const int at = i - (s > 0 ? P.end[s - 1] : 0);
    uint4 v;
    asm volatile("ld.volatile.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(P.src[s] + at) : "memory");
    P.dst[s][at] = v;
}

}  // namespace

// n copies (at most 8) of bytes[i] bytes each, a multiple of 16, from device-visible host addresses.
cudaError_t rabit_launch_fetch(const void* const* src, void* const* dst, const size_t* bytes, int n, cudaStream_t stream) {
    if (n < 1 || n > 8) return cudaErrorInvalidValue;
    FetchParams P;
    size_t total = 0;
    for (int i = 0; i < 8; ++i) {
        if (i < n) {
            if ((bytes[i] | (size_t)(uintptr_t)src[i] | (size_t)(uintptr_t)dst[i]) & 15u) return cudaErrorInvalidValue;
            total += bytes[i] / 16;
            if (total > (1u << 30)) return cudaErrorInvalidValue;
        }
        P.src[i] = reinterpret_cast<const uint4*>(i < n ? src[i] : nullptr);
        P.dst[i] = reinterpret_cast<uint4*>(i < n ? dst[i] : nullptr);
        P.end[i] = (int)total;
    }
    P.n = n;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned int)((total + kThreads - 1) / kThreads));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, rabit_fetch_kernel, P);
}
