// Which host buffers of a call the kernels may use in place.
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

namespace avsg {

// Device-visible address of a caller's host buffer of `count` elements, or null: it has to be page-locked and mapped from
// its first byte to its last, at device addresses that go on as the host's do (a copy checks its whole range, a kernel's
// access beyond what is mapped would be a fault).
template <typename T>
T* mapped(T* p, size_t count)
{
    const uint8_t* host[2] = {reinterpret_cast<const uint8_t*>(p), reinterpret_cast<const uint8_t*>(p + count) - 1};
    uint8_t* dev[2];
    for (int i = 0; i < 2; ++i) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, host[i]) != cudaSuccess) { cudaGetLastError(); return nullptr; }
        if (at.type != cudaMemoryTypeHost || at.devicePointer == nullptr) return nullptr;
        dev[i] = static_cast<uint8_t*>(at.devicePointer);
    }
    return dev[1] - dev[0] == host[1] - host[0] ? reinterpret_cast<T*>(dev[0]) : nullptr;
}

}  // namespace avsg
