// Host buffers that are page-locked in part, against a stand-in for the runtime that knows three registered ranges.
#include <stdio.h>
#include "host_buffers.h"

struct Range { uint64_t host, bytes, dev; cudaMemoryType type; };
static const Range ranges[] = {{0x10000, 0x1000, 0x910000, cudaMemoryTypeHost},      // two that the device sees side by side,
                               {0x11000, 0x1000, 0x911000, cudaMemoryTypeHost},
                               {0x12000, 0x1000, 0x700000, cudaMemoryTypeHost},      // one that lies elsewhere there,
                               {0x13000, 0x1000, 0x13000, cudaMemoryTypeDevice}};    // and no host memory

extern "C" cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* at, const void* p)
{
    const uint64_t a = reinterpret_cast<uint64_t>(p);
    *at = cudaPointerAttributes();
    at->type = cudaMemoryTypeUnregistered;
    for (const Range& r : ranges)
        if (a >= r.host && a < r.host + r.bytes) {
            at->type = r.type;
            at->devicePointer = reinterpret_cast<void*>(r.dev + (a - r.host));
        }
    return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }

static int failed = 0;
template <typename T>
static void expect(uint64_t host, size_t count, uint64_t dev)
{
    const uint64_t got = reinterpret_cast<uint64_t>(avsg::mapped(reinterpret_cast<T*>(host), count));
    if (got != dev) { printf("%llx + %zu: %llx, not %llx\n", (unsigned long long)host, count, (unsigned long long)got, (unsigned long long)dev); failed = 1; }
}

int main()
{
    expect<int32_t>(0x10000, 1024, 0x910000);            // all of a range, and its last elements
    expect<int32_t>(0x10ff8, 2, 0x910ff8);
    expect<uint8_t>(0x10fff, 1, 0x910fff);
    expect<int32_t>(0x10800, 1024, 0x910800);            // into a range that goes on
    expect<int32_t>(0x11ffc, 1, 0x911ffc);
    expect<int32_t>(0x11ffc, 2, 0);                      // into one that does not
    expect<int32_t>(0x12800, 1024, 0);                   // the end is no host memory
    expect<uint8_t>(0xffff, 2, 0);                       // the start is not page-locked
    expect<int32_t>(0x13000, 4, 0);
    expect<int32_t>(0x20000, 4, 0);
    expect<int32_t>(0x10000, 1 << 20, 0);                // the end is pageable
    return failed;
}
