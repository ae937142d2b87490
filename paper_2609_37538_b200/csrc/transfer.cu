// Stage Two of the AVSG operator: miss-only host -> device gather (Sec. 3.4).
//
// The step's miss list is segmented by table (token order, then position
// order inside a table).  Every thread block recomputes the exclusive prefix
// sum of the segment lengths, which gives N_miss, and takes floor(N_miss/C)
// or ceil(N_miss/C) consecutive misses (Eq. 6, C = number of blocks); inside
// a block the warps take rows round-robin.  One warp moves one row: its lanes
// read the host row in place (mapped pinned memory) with 16-byte loads, so a
// warp-wide load covers 512 contiguous bytes of ONE row, and store it into
// the reserved slot.  Keeping a warp inside one row matters: the host link
// is bound by the number of read requests, and 16-byte units that straddle
// two rows produce more, smaller requests (measured 43.5 vs 47.5 GB/s).
//
// request_level = 1 gives the comparator S1 of App. D: block b serves
// segment b alone.
//
// avsg_transfer_overlap_kernel is the same gather started per token while
// Stage One still runs (App. G, latency hiding; described at the kernel), and
// avsg_transfer_positions_kernel is the comparator S2 of App. D.
#include "avsg_kernels.cuh"

namespace avsg {
namespace {

constexpr int CHUNKS_PER_PASS = 4;     // 16-byte loads a lane keeps in flight (covers rows up to 2 KiB per pass)

// 16-byte global load / store in the order written (volatile asm statements keep their relative order).
__device__ __forceinline__ int4 ld16(uint64_t addr)
{
    int4 v;
    asm volatile("ld.global.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(addr));
    return v;
}
__device__ __forceinline__ void st16(uint64_t addr, const int4& v)
{
    asm volatile("st.global.v4.s32 [%0], {%1, %2, %3, %4};" :: "l"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// One warp moves one row: 16-byte loads from the (host) source, all issued before the 16-byte stores into the slot.
// Rows of up to 1 KiB (two loads per lane) take the short path, whose instruction order is fixed by hand: both
// loads of a lane are in flight together.
__device__ __forceinline__ void copy_row(uint64_t src, uint64_t dst, uint32_t cpr, uint32_t lane)
{
    if (cpr <= 64u) {
        const bool p0 = lane < cpr, p1 = lane + 32u < cpr;
        int4 a = make_int4(0, 0, 0, 0), b = make_int4(0, 0, 0, 0);
        if (p0) a = ld16(src + 16ull * lane);
        if (p1) b = ld16(src + 16ull * (lane + 32u));
        if (p0) st16(dst + 16ull * lane, a);
        if (p1) st16(dst + 16ull * (lane + 32u), b);
        return;
    }
    for (uint32_t c0 = lane; c0 < cpr; c0 += 32u * CHUNKS_PER_PASS) {
        int4 v[CHUNKS_PER_PASS];
#pragma unroll
        for (int k = 0; k < CHUNKS_PER_PASS; ++k) {
            const uint32_t c = c0 + 32u * k;
            if (c < cpr) v[k] = *reinterpret_cast<const int4*>(src + 16ull * c);
        }
#pragma unroll
        for (int k = 0; k < CHUNKS_PER_PASS; ++k) {
            const uint32_t c = c0 + 32u * k;
            if (c < cpr) *reinterpret_cast<int4*>(dst + 16ull * c) = v[k];
        }
    }
}

// The share of worker w of W (32 threads each) of the call's outputs, to host memory: 16 bytes a lane where the caller's
// pointer allows it.  The stores are posted: nothing waits for them but the end of the grid.  One 32-table call (0.5 MB of
// slots, 131 KB of flags) with ids read and outputs written by the kernels: 130.4 us where the calls queue, 145 alone;
// with copies and events on a side stream 147.4 and 154.  (Stage One writing them to the host itself: 165, its hand-over
// fences wait for the link.)
__device__ __forceinline__ void put_out(const uint8_t* src, uint8_t* dst, uint32_t bytes, uint32_t w, uint32_t W, uint32_t lane)
{
    const uint32_t wide = (reinterpret_cast<uint64_t>(dst) & 15u) == 0 ? bytes / 16u : 0u;
    for (uint32_t i = w * 32u + lane; i < wide; i += W * 32u)
        reinterpret_cast<int4*>(dst)[i] = __ldcg(reinterpret_cast<const int4*>(src) + i);
    const uint32_t words = (reinterpret_cast<uint64_t>(dst) & 3u) == 0 ? bytes / 4u : 0u;
    for (uint32_t i = wide * 4u + w * 32u + lane; i < words; i += W * 32u)
        reinterpret_cast<int32_t*>(dst)[i] = __ldcg(reinterpret_cast<const int32_t*>(src) + i);
    for (uint32_t i = (words ? words * 4u : wide * 16u) + w * 32u + lane; i < bytes; i += W * 32u) dst[i] = __ldcg(src + i);
}
__device__ __forceinline__ void put_outputs(const HostOut& o, uint32_t w, uint32_t W, uint32_t lane)
{
    put_out(reinterpret_cast<const uint8_t*>(o.slots), reinterpret_cast<uint8_t*>(o.host_slots), o.n_slots * 4u, w, W, lane);
    if (o.n_hit) put_out(o.hit, o.host_hit, o.n_hit, w, W, lane);
    if (o.n_count)
        put_out(reinterpret_cast<const uint8_t*>(o.count), reinterpret_cast<uint8_t*>(o.host_count), o.n_count * 4u, w, W, lane);
}

__global__ void __launch_bounds__(1024, 1) avsg_transfer_kernel(const __grid_constant__ XferParams p)
{
    __shared__ uint32_t s_pref[XFER_MAX_SEG + 1];
    __shared__ uint32_t s_w[40];

    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u;
    const uint32_t n_seg = p.n_seg;

    // Programmatic dependent launch: the blocks may already be resident while Stage One still runs; the miss
    // list is read only after that grid has completed.  The kernel after this one may start its prologue.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (p.t_range && tid == 0) atomicMin(p.t_range, global_ns());

    if (p.out.n_slots) put_outputs(p.out, blockIdx.x * (nt >> 5) + (tid >> 5), gridDim.x * (nt >> 5), lane);

    // global miss prefix sum (every block computes the same one)
    uint32_t running = 0;
    for (uint32_t base = 0; base < n_seg; base += nt) {
        const uint32_t i = base + tid;
        const uint32_t c = i < n_seg ? p.seg[i].count : 0u;
        uint32_t total;
        const uint32_t excl = block_excl_scan(c, s_w, total);
        if (i < n_seg) s_pref[i] = running + excl;
        running += total;
        __syncthreads();
    }
    if (tid == 0) s_pref[n_seg] = running;
    __syncthreads();

    uint32_t m0, m1;                                           // this block's share of the miss list
    if (p.request_level) {
        m0 = s_pref[blockIdx.x];
        m1 = s_pref[blockIdx.x + 1];
    } else {
        const uint32_t C = gridDim.x, c = blockIdx.x, q = running / C, r = running % C;
        m0 = c * q + (c < r ? c : r);
        m1 = m0 + q + (c < r ? 1u : 0u);
    }

    const uint32_t cpr = p.row_bytes >> 4;                     // 16-byte chunks per row
    bool first_row = p.t_range != nullptr;                     // timing: when the copy starts, when its first row is in
    if (first_row && tid == 0 && m1 > m0) atomicMin(p.t_range + 2, global_ns());
    for (uint32_t m = m0 + (tid >> 5); m < m1; m += nt >> 5) {
        uint32_t lo = 0, hi = n_seg;                           // largest lo with s_pref[lo] <= m
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_pref[mid] <= m) lo = mid; else hi = mid;
        }
        const uint32_t local = m - s_pref[lo];
        if (local >= p.list_stride) {
            if (lane == 0) atomicOr(p.status, ST_BAD_SEGMENT);
            continue;
        }
        const int2 e = __ldg(p.miss_list + (size_t)lo * p.list_stride + local);
        if (e.x < 0) continue;                                 // padding entry of the transfer-all-K comparator
        if (e.y < 0 || (uint32_t)e.y >= p.S) {
            if (lane == 0) atomicOr(p.status, ST_BAD_SLOT);
            continue;
        }
        const uint64_t src = __ldg(&p.seg[lo].src_base) + (uint64_t)(uint32_t)e.x * __ldg(&p.seg[lo].src_stride);
        const uint64_t dst = __ldg(&p.seg[lo].dst_base) + (uint64_t)(uint32_t)e.y * p.row_bytes;
        copy_row(src, dst, cpr, lane);
        if (first_row) {
            if (tid == 0) atomicMin(p.t_range + 3, global_ns());
            first_row = false;
        }
    }
    if (p.t_range) {
        __syncthreads();
        if (tid == 0) {
            const unsigned long long t = global_ns();
            atomicMax(p.t_range + 1, t);
            if (m1 > m0) atomicMin(p.t_range + 4, t);          // the earliest block to finish: the tail starts here
        }
    }
}

// Stage Two that overlaps Stage One (the latency-hiding direction of App. G).  The grid is launched with programmatic
// stream serialization and does NOT wait for Stage One to complete: its blocks become resident once every Stage One
// block has started, and copy each token's misses as soon as Stage One has placed that token of all tables.  Stage One
// raises a flag per table and token, carrying the miss count, after making those miss-list entries visible; it has taken
// all flags down before this grid could start.
//
// A call is walked in phases, one per token.  The last warp of a block polls the phase's flags - with a bound -,
// prefix-sums the counts over the tables and raises s_ready; the other warps copy (Eq. 6 per phase: the misses are cut
// evenly over the blocks, and a block's over its warps).  In a small call no barrier ties the warps together and phases
// go round over the blocks and warps: a row is a round trip of 2 us, and a warp without one in this phase is already at
// work on the next (one request, 230 rows in two tokens: 17.3 us a call where the block met after every phase and found
// its last block with a counter, 15.8 now).  With more rows per block than warps the copying warps do meet: rows of a
// later phase that mix with this one's cost 1 % where the link is the limit (128 tables in one call: 392 us against
// 394), and 5 % where translations on the way to 11 GB of host memory are.
//
// A call is one round unless it has so many tables that Stage One, with a block per table, would take most of the SMs:
// then Stage One runs with round_size blocks that serve the tables round by round, and this grid follows them.  Every
// Stage One block is resident before this grid starts and never waits for it, so it always makes progress; if a wait
// still runs out the block sets ST_WAIT_TIMEOUT and stops copying.  Before leaving, every block waits for the
// completion of the Stage One grid, so that the completion of this grid implies it.  The kernel arguments hold nothing
// that changes from call to call (a captured call can be replayed).  All reads of data written by the running Stage One go to L2 (ld.cg / acquire).
constexpr uint32_t GAVE_UP = 0xFFFFFFFFu;
constexpr uint32_t READY_SPIN_LIMIT = 1u << 24;              // far above the polling warp's own limit

template <int CAP>
__global__ void __launch_bounds__(1024, 1) avsg_transfer_overlap_kernel(const __grid_constant__ XferOverlapParamsT<CAP> p)
{
    extern __shared__ uint32_t s_phase[];        // per phase: prefix sums [round_size + 1], first list entries [round_size]
    __shared__ volatile uint32_t s_ready;        // phases whose prefix sums are there
    __shared__ uint32_t s_copied;

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, W = (blockDim.x >> 5) - 1u;   // W warps copy
    const uint32_t n = p.n, rounds = (n + p.round_size - 1u) / p.round_size, phases = rounds * p.n_q;
    const uint32_t stride = 2u * p.round_size + 1u;

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (p.t_range && tid == 0) atomicMin(p.t_range, global_ns());
    if (tid == 0) { s_ready = 0; s_copied = 0; }
    __syncthreads();

    if (warp == W) {
        for (uint32_t ph = 0, base = 0, g = 0; ph < phases; ++ph) {
            const uint32_t nr = n - base < p.round_size ? n - base : p.round_size;       // tables [base, base + nr)
            uint32_t* pref = s_phase + ph * stride;
            uint32_t* off = pref + p.round_size + 1u;
            uint32_t running = 0;
            bool ok = true;
            for (uint32_t i = lane; i - lane < nr && ok; i += 32u) {
                uint32_t c = 0, spin = 0;
                if (i < nr) {
                    const uint32_t* f = p.flags + (size_t)(base + i) * p.n_q + g;
                    for (; spin < OVERLAP_SPIN_LIMIT; ++spin) {
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(f) : "memory");
                        if (c) break;
                        __nanosleep(64);
                    }
                    c -= c ? 1u : 0u;                                   // the table's misses of this phase
                }
                ok = __all_sync(0xffffffffu, spin < OVERLAP_SPIN_LIMIT);
                const uint32_t incl = warp_incl_scan(c, lane);
                if (i < nr) {
                    pref[i] = running + incl - c;
                    off[i] = g == 0 ? 0u : off[(int)i - (int)stride] + pref[(int)i + 1 - (int)stride] - pref[(int)i - (int)stride];
                }
                running += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (!ok) {
                if (lane == 0) { atomicOr(p.status, ST_WAIT_TIMEOUT); s_ready = GAVE_UP; }
                break;
            }
            if (lane == 0) pref[nr] = running;
            __threadfence_block();
            __syncwarp();
            if (lane == 0) s_ready = ph + 1u;
            if (++g == p.n_q) { g = 0; base += p.round_size; }
        }
    } else {
        const uint32_t C = gridDim.x, cpr = p.row_bytes >> 4;
        bool first_row = p.t_range != nullptr;
        uint32_t block_from = 0, warp_from = 0;                        // where the next phase's shares start
        for (uint32_t ph = 0, base = 0, g = 0; ph < phases; ++ph) {
            const uint32_t nr = n - base < p.round_size ? n - base : p.round_size;
            const uint32_t* pref = s_phase + ph * stride;
            const uint32_t* off = pref + p.round_size + 1u;
            uint32_t ready = s_ready;
            for (uint32_t spin = 0; ready <= ph && spin < READY_SPIN_LIMIT; ++spin) {
                __nanosleep(32);
                ready = s_ready;
            }
            ready = __shfl_sync(0xffffffffu, ready, 0);                // one decision for the warp
            if (ready <= ph || ready == GAVE_UP) {
                if (ready != GAVE_UP && lane == 0) atomicOr(p.status, ST_WAIT_TIMEOUT);
                break;
            }
            __threadfence_block();
            if (p.out.n_slots && ph + 1u == phases)                    // the call's last token is placed: outputs are final
                put_outputs(p.out, blockIdx.x * W + warp, C * W, lane);
            const uint32_t total = pref[nr], q = total / C, rem = total % C;
            const uint32_t cb = blockIdx.x >= block_from ? blockIdx.x - block_from : blockIdx.x + C - block_from;
            const uint32_t m0 = cb * q + (cb < rem ? cb : rem), count = q + (cb < rem ? 1u : 0u);
            block_from = q > 0 ? 0u : block_from + rem < C ? block_from + rem : block_from + rem - C;
            if (first_row && lane == 0 && count) { atomicMin(p.t_range + 2, global_ns()); s_copied = 1; }
            for (uint32_t k = warp >= warp_from ? warp - warp_from : warp + W - warp_from; k < count; k += W) {
                const uint32_t m = m0 + k;
                uint32_t lo = 0, hi = nr;                              // largest lo with pref[lo] <= m
                while (hi - lo > 1) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (pref[mid] <= m) lo = mid; else hi = mid;
                }
                const uint32_t t = base + lo;                          // the table, within the call
                const uint32_t local = off[lo] + (m - pref[lo]);       // entry of the table's miss list
                if (local >= p.list_stride) {
                    if (lane == 0) atomicOr(p.status, ST_BAD_SEGMENT);
                    continue;
                }
                const int2 e = __ldcg(p.miss_list + (size_t)t * p.list_stride + local);
                if (e.x < 0) continue;
                if (e.y < 0 || (uint32_t)e.y >= p.S) {
                    if (lane == 0) atomicOr(p.status, ST_BAD_SLOT);
                    continue;
                }
                const uint64_t src = p.kv_base[t] + (uint64_t)(uint32_t)e.x * p.kv_stride[t];
                const uint64_t dst = reinterpret_cast<uint64_t>(p.buffer) +
                                     ((uint64_t)p.table_id[t] * p.S + (uint32_t)e.y) * p.row_bytes;
                copy_row(src, dst, cpr, lane);
                if (first_row) {
                    if (lane == 0) atomicMin(p.t_range + 3, global_ns());
                    first_row = false;
                }
            }
            if (q < W) {
                warp_from = (warp_from + count) % W;
            } else {
                warp_from = 0;
                asm volatile("bar.sync 1, %0;" :: "r"(W * 32u) : "memory");        // (q is the same in all of them)
            }
            if (++g == p.n_q) { g = 0; base += p.round_size; }
        }
    }
    __syncthreads();
    const unsigned long long t_copied = p.t_range ? global_ns() : 0ull;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.t_range && tid == 0) {
        atomicMax(p.t_range + 1, global_ns());                         // the block's end, the wait for Stage One included
        if (s_copied) atomicMin(p.t_range + 4, t_copied);
    }
}

// Comparator S2 (App. D, Eq. 14): the n * N_q * K selected positions of the call are flattened and cut into
// gridDim.x near-equal contiguous ranges regardless of hit or miss; a block walks its range, one warp per
// position, and copies the row of every position that missed.  Work per block = misses in its range (Eq. 15).
__global__ void __launch_bounds__(1024) avsg_transfer_positions_kernel(const __grid_constant__ PosParams p)
{
    const uint32_t lane = threadIdx.x & 31u, warps = blockDim.x >> 5;
    const uint64_t P = (uint64_t)p.n * p.per_table, C = gridDim.x, c = blockIdx.x;
    const uint64_t begin = c * P / C, end = (c + 1) * P / C;
    const uint32_t cpr = p.row_bytes >> 4;
    for (uint64_t q = begin + (threadIdx.x >> 5); q < end; q += warps) {
        const int32_t x = __ldg(p.indices + q);
        if (x < 0 || __ldg(p.hit + q)) continue;                 // padding or hit: nothing to move
        const int32_t o = __ldg(p.slots + q);
        if (o < 0) continue;                                     // an id Stage One refused (beyond the host rows)
        if ((uint32_t)o >= p.S) {
            if (lane == 0) atomicOr(p.status, ST_BAD_SLOT);
            continue;
        }
        const uint32_t ti = (uint32_t)(q / p.per_table);
        const uint64_t src = __ldg(&p.seg[ti].src_base) + (uint64_t)(uint32_t)x * __ldg(&p.seg[ti].src_stride);
        const uint64_t dst = __ldg(&p.seg[ti].dst_base) + (uint64_t)(uint32_t)o * p.row_bytes;
        copy_row(src, dst, cpr, lane);
    }
}

}  // namespace

cudaError_t launch_transfer_positions(const PosParams& p, uint32_t blocks, uint32_t threads, cudaStream_t stream)
{
    avsg_transfer_positions_kernel<<<blocks, threads, 0, stream>>>(p);
    return cudaGetLastError();
}

namespace {
template <int CAP>
cudaError_t launch_transfer_overlap_t(const XferOverlapParamsT<CAP>& p, uint32_t blocks, uint32_t threads, cudaStream_t stream)
{
    const uint32_t phases = (p.n + p.round_size - 1) / p.round_size * p.n_q;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads + 32 < 1024 ? threads + 32 : 1024);        // the copying warps and the one that polls
    cfg.dynamicSmemBytes = phases * (2 * p.round_size + 1) * sizeof(uint32_t);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, avsg_transfer_overlap_kernel<CAP>, p);
}
}  // namespace

cudaError_t launch_transfer_overlap(const XferOverlapParams& p, uint32_t blocks, uint32_t threads, cudaStream_t stream)
{
    return launch_transfer_overlap_t(p, blocks, threads, stream);
}

cudaError_t launch_transfer_overlap(const XferOverlapParamsBig& p, uint32_t blocks, uint32_t threads, cudaStream_t stream)
{
    return launch_transfer_overlap_t(p, blocks, threads, stream);
}

cudaError_t launch_transfer(const XferParams& p, uint32_t blocks, uint32_t threads, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, avsg_transfer_kernel, p);
}

// Loads this file's kernels (see stage_one_prepare() on why that is not left to their first launch).
cudaError_t transfer_prepare()
{
    const void* kernels[] = {reinterpret_cast<const void*>(avsg_transfer_overlap_kernel<S1_MAX_TABLES>),
                             reinterpret_cast<const void*>(avsg_transfer_overlap_kernel<S1_BIG_TABLES>),
                             reinterpret_cast<const void*>(avsg_transfer_kernel),
                             reinterpret_cast<const void*>(avsg_transfer_positions_kernel)};
    for (const void* k : kernels) {
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
    }
    // a call in 32 rounds of 32 tables and eight tokens has 256 phases
    for (int k = 0; k < 2; ++k) {
        cudaError_t e = cudaFuncSetAttribute(kernels[k], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(OVERLAP_MAX_TABLES / S1_ROUND_BLOCKS * OVERLAP_MAX_TOKENS *
                                                   (2 * S1_ROUND_BLOCKS + 1) * sizeof(uint32_t)));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace avsg
