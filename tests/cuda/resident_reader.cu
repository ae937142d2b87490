// A stand-in for a consumer of the early outputs on another stream than the calls'.  Test code: it is compiled by
// tests/test_one_kernel_calls.py, not part of the library.  Copies the rows that were resident before the call (positions with a slot
// whose `arriving` flag is 0), a warp a row, in blocks that can be given much shared memory.  It waits for nobody: what it reads is final
// when it starts.
#include <cuda_runtime.h>
#include <stdint.h>

namespace {

__global__ void __launch_bounds__(256) resident_reader_kernel(const int32_t* slots, const uint8_t* arriving, uint32_t positions, uint32_t per_table,
                                                              const uint8_t* rows, uint32_t S, uint32_t row_bytes, uint8_t* out)
{
    const uint32_t lane = threadIdx.x & 31u, warps = blockDim.x / 32u;
    for (uint32_t i = blockIdx.x * warps + threadIdx.x / 32u; i < positions; i += gridDim.x * warps) {
        const int32_t j = __ldcg(slots + i);
        if (j < 0 || (uint32_t)j >= S || __ldcg(arriving + i)) continue;
        const uint8_t* src = rows + ((size_t)(i / per_table) * S + (uint32_t)j) * row_bytes;
        for (uint32_t b = lane; b < row_bytes; b += 32u) out[(size_t)i * row_bytes + b] = __ldcg(src + b);
    }
}

}  // namespace

extern "C" int launch_resident_reader(const void* slots, const void* arriving, uint32_t positions, uint32_t per_table, const void* rows,
                                      uint32_t S, uint32_t row_bytes, void* out, uint32_t shared_bytes, void* stream)
{
    if (cudaFuncSetAttribute(resident_reader_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shared_bytes) != cudaSuccess) return -1;
    resident_reader_kernel<<<148, 256, shared_bytes, static_cast<cudaStream_t>(stream)>>>(
        static_cast<const int32_t*>(slots), static_cast<const uint8_t*>(arriving), positions, per_table, static_cast<const uint8_t*>(rows), S,
        row_bytes, static_cast<uint8_t*>(out));
    return (int)cudaGetLastError();
}
