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
#include "follow_stage_one.cuh"

namespace avsg {
namespace {

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
// A call is one round unless it has so many tables that Stage One, with a block per table, would take most of the SMs:
// then Stage One runs with round_size blocks that serve the tables round by round, and this grid follows them.  Every
// Stage One block is resident before this grid starts and never waits for it, so it always makes progress; if a wait
// still runs out the block sets ST_WAIT_TIMEOUT and stops copying.  Before leaving, every block waits for the
// completion of the Stage One grid, so that the completion of this grid implies it.  The kernel arguments hold nothing
// that changes from call to call (a captured call can be replayed).  All reads of data written by the running Stage One
// go to L2 (ld.cg / acquire).
template <int CAP>
__global__ void __launch_bounds__(1024, 1) avsg_transfer_overlap_kernel(const __grid_constant__ XferOverlapParamsT<CAP> p)
{
    extern __shared__ uint32_t s_phase[];

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (p.t_range && threadIdx.x == 0) atomicMin(p.t_range, global_ns());
    const bool copied = follow_stage_one(p, p.n, p.n_q, p.round_size, blockIdx.x, gridDim.x, p.t_range, s_phase,
        [&](uint32_t t, uint32_t g, uint32_t& count) {                 // the flag of table t and token g
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(count) : "l"(p.flags + (size_t)t * p.n_q + g) : "memory");
            const bool raised = count >= p.announcers * ANNOUNCED;
            count &= ANNOUNCED - 1u;
            return raised;
        });
    const unsigned long long t_copied = p.t_range ? global_ns() : 0ull;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.t_range && threadIdx.x == 0) {
        atomicMax(p.t_range + 1, global_ns());                         // the block's end, the wait for Stage One included
        if (copied) atomicMin(p.t_range + 4, t_copied);
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
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads + 32 < 1024 ? threads + 32 : 1024);        // the copying warps and the one that polls
    cfg.dynamicSmemBytes = follow_words(p.n, p.n_q, p.round_size) * sizeof(uint32_t);
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
                                             (int)(follow_words(OVERLAP_MAX_TABLES, OVERLAP_MAX_TOKENS, S1_ROUND_BLOCKS) *
                                                   sizeof(uint32_t)));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace avsg
