// When a grid that is launched behind a call may start.  Test code: it is compiled by tests/test_one_kernel_calls.py, not part of the
// library.  hold_kernel lets the grid behind it start at once and then takes a given time; mark_kernel, launched with programmatic
// stream serialization behind the call, says when it has started.  Neither waits for anybody.
#include <cuda_runtime.h>
#include <stdint.h>

namespace {

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__global__ void hold_kernel(unsigned long long ns, unsigned long long* end)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const unsigned long long from = now_ns();
    for (uint32_t i = 0; i < (1u << 16) && now_ns() - from < ns; ++i) __nanosleep(1000);
    *end = now_ns();
}

__global__ void mark_kernel(unsigned long long* start)
{
    *start = now_ns();
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace

extern "C" int launch_hold(unsigned long long ns, void* end, void* stream)
{
    hold_kernel<<<1, 1, 0, static_cast<cudaStream_t>(stream)>>>(ns, static_cast<unsigned long long*>(end));
    return (int)cudaGetLastError();
}

extern "C" int launch_mark(void* start, void* stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1); cfg.blockDim = dim3(1); cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return (int)cudaLaunchKernelEx(&cfg, mark_kernel, static_cast<unsigned long long*>(start));
}
