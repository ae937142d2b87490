// The copy of a row and the outputs of calls with host buffers, shared by every kernel that copies; and the overlapped
// transfer kernel's way through a call.
#pragma once
#include "avsg_kernels.cuh"

namespace avsg {

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

// A row of up to ROW_CHUNKS 16-byte pieces in a warp's registers, for a kernel that asks for it before it knows where it goes.
// (By cp.async into shared memory, which would need no registers, 32 tables take 245 us past L1 and 125 through it, and not 117:
// those requests are smaller.)
constexpr uint32_t ROW_CHUNKS = 96;
struct Row { int4 v[ROW_CHUNKS / 32]; };
__device__ __forceinline__ void load_row(Row& r, uint64_t src, uint32_t chunks, uint32_t lane)
{
    // (One statement, predicated inside: with a branch around it a piece would have an old and a new value, and a copy from register
    // to register where these meet would wait for the load.  The pieces' loads follow one another without anything in between.)
    static_assert(ROW_CHUNKS == 96, "three loads");
    asm volatile("{\n\t.reg .pred p, q, r;\n\t"
                 "setp.gt.u32 p, %14, %13;\n\tsetp.gt.u32 q, %15, %13;\n\tsetp.gt.u32 r, %16, %13;\n\t"
                 "@p ld.global.v4.s32 {%0, %1, %2, %3}, [%12];\n\t"
                 "@q ld.global.v4.s32 {%4, %5, %6, %7}, [%12 + 512];\n\t"
                 "@r ld.global.v4.s32 {%8, %9, %10, %11}, [%12 + 1024];\n\t}"
                 : "=r"(r.v[0].x), "=r"(r.v[0].y), "=r"(r.v[0].z), "=r"(r.v[0].w), "=r"(r.v[1].x), "=r"(r.v[1].y), "=r"(r.v[1].z), "=r"(r.v[1].w),
                   "=r"(r.v[2].x), "=r"(r.v[2].y), "=r"(r.v[2].z), "=r"(r.v[2].w)
                 : "l"(src + 16ull * lane), "r"(lane), "r"(chunks), "r"(chunks > 32u ? chunks - 32u : 0u), "r"(chunks > 64u ? chunks - 64u : 0u));
    __syncwarp();                      // (the compiler may move plain loads behind a wait, but not behind this)
}
__device__ __forceinline__ void store_row(const Row& r, uint64_t dst, uint32_t cpr, uint32_t lane)
{
#pragma unroll
    for (uint32_t k = 0; k < ROW_CHUNKS / 32; ++k)
        if (lane + 32u * k < cpr) st16(dst + 16ull * (lane + 32u * k), r.v[k]);
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
    const uint64_t odd = reinterpret_cast<uint64_t>(dst) | reinterpret_cast<uint64_t>(src);
    const uint32_t wide = (odd & 15u) == 0 ? bytes / 16u : 0u;
    for (uint32_t i = w * 32u + lane; i < wide; i += W * 32u)
        reinterpret_cast<int4*>(dst)[i] = __ldcg(reinterpret_cast<const int4*>(src) + i);
    const uint32_t words = (odd & 3u) == 0 ? bytes / 4u : 0u;
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
// The outputs of the ti-th table alone: `ids` positions, `tokens` counts.
__device__ __forceinline__ void put_outputs_of(HostOut o, uint32_t ti, uint32_t ids, uint32_t tokens, uint32_t w, uint32_t W, uint32_t lane)
{
    o.slots += (size_t)ti * ids; o.host_slots += (size_t)ti * ids; o.n_slots = ids;
    if (o.n_hit) { o.hit += (size_t)ti * ids; o.host_hit += (size_t)ti * ids; o.n_hit = ids; }
    if (o.n_count) { o.count += (size_t)ti * tokens; o.host_count += (size_t)ti * tokens; o.n_count = tokens; }
    put_outputs(o, w, W, lane);
}

// Copies what Stage One announces, in one of `blocks` thread blocks.  A call is walked in phases, one per announcement.
// The last warp of a block polls the phase's flags (`flag(table, phase, count)`: raised?) - with a bound -, prefix-sums
// the counts over the tables and raises s_ready; the other warps copy (Eq. 6 per phase: the misses are cut evenly over the
// blocks, and a block's over its warps).  With few rows no barrier ties the warps together and phases go round over the
// blocks and warps: a row is a round trip of 2 us, and a warp without one in this phase is already at work on the next
// (230 rows in two tokens: 17.3 us a call where the block met after every phase and found its last block with a counter,
// 15.8 now).  With more rows per block than warps
// the copying warps do meet: rows of a later phase that mix with this one's cost 5 % where translations on the way to 11 GB of
// host memory are the limit (where the link is, no difference was found).
constexpr uint32_t READY_SPIN_LIMIT = 1u << 28;              // over 10 s: the polling warp ends the wait long before

// Words of shared memory that the phases of a call take: prefix sums [round_size + 1] and first list entries [round_size].
__host__ __device__ inline uint32_t follow_words(uint32_t n, uint32_t n_pub, uint32_t round_size)
{
    return (n + round_size - 1u) / round_size * n_pub * (2u * round_size + 1u);
}

// n tables in rounds of round_size, n_pub announcements each.  Ends with a block barrier; returns whether the block copied
// anything (known with t_range only).
template <typename P, typename F>
__device__ __forceinline__ bool follow_stage_one(const P& p, uint32_t n, uint32_t n_pub, uint32_t round_size, uint32_t block,
                                                 uint32_t blocks, unsigned long long* t_range, uint32_t* s_phase, F flag)
{
    __shared__ volatile uint32_t s_ready, s_gave_up;     // phases whose prefix sums are there; no more will come
    __shared__ uint32_t s_copied;

    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, W = (blockDim.x >> 5) - 1u;   // W warps copy
    const uint32_t phases = (n + round_size - 1u) / round_size * n_pub, stride = 2u * round_size + 1u;
    if (tid == 0) { s_ready = s_gave_up = 0; s_copied = 0; }
    __syncthreads();

    if (warp == W) {
        for (uint32_t ph = 0, base = 0, g = 0; ph < phases; ++ph) {
            const uint32_t nr = n - base < round_size ? n - base : round_size;       // tables [base, base + nr)
            uint32_t* pref = s_phase + ph * stride;
            uint32_t* off = pref + round_size + 1u;
            uint32_t running = 0;
            bool ok = true;
            for (uint32_t i = lane; i - lane < nr && ok; i += 32u) {
                uint32_t c = 0, spin = 0;                               // c: the table's misses of this phase
                if (i < nr)
                    for (; spin < OVERLAP_SPIN_LIMIT && !flag(base + i, g, c); ++spin) __nanosleep(64);
                ok = __all_sync(0xffffffffu, spin < OVERLAP_SPIN_LIMIT);
                const uint32_t incl = warp_incl_scan(c, lane);
                if (i < nr) {
                    pref[i] = running + incl - c;
                    off[i] = g == 0 ? 0u : off[(int)i - (int)stride] + pref[(int)i + 1 - (int)stride] - pref[(int)i - (int)stride];
                }
                running += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (!ok) {
                if (lane == 0) { atomicOr(p.status, ST_WAIT_TIMEOUT); s_gave_up = 1; }
                break;
            }
            if (lane == 0) pref[nr] = running;
            __threadfence_block();
            __syncwarp();
            if (lane == 0) s_ready = ph + 1u;
            if (++g == n_pub) { g = 0; base += round_size; }
        }
    } else {
        const uint32_t C = blocks, cpr = p.row_bytes >> 4;
        bool first_row = t_range != nullptr;
        uint32_t block_from = 0, warp_from = 0;               // where the next phase's shares start
        for (uint32_t ph = 0, base = 0, g = 0; ph < phases; ++ph) {
            const uint32_t nr = n - base < round_size ? n - base : round_size;
            const uint32_t* pref = s_phase + ph * stride;
            const uint32_t* off = pref + round_size + 1u;
            // (s_ready stays what it is once s_gave_up is set: every warp of the block goes through the same phases)
            uint32_t gave_up = 0;
            for (uint32_t spin = 0; s_ready <= ph && !gave_up && spin < READY_SPIN_LIMIT; ++spin) {
                __nanosleep(32);
                gave_up = s_gave_up;
            }
            __threadfence_block();
            if (__shfl_sync(0xffffffffu, s_ready, 0) <= ph) break;     // one decision for the warp
            __threadfence_block();
            if (p.out.n_slots && ph + 1u == phases)                    // the call's last token is placed: outputs are final
                put_outputs(p.out, block * W + warp, C * W, lane);
            const uint32_t total = pref[nr], q = total / C, rem = total % C;
            const uint32_t cb = block >= block_from ? block - block_from : block + C - block_from;
            const uint32_t m0 = cb * q + (cb < rem ? cb : rem), count = q + (cb < rem ? 1u : 0u);
            block_from = q > 0 ? 0u : block_from + rem < C ? block_from + rem : block_from + rem - C;
            if (first_row && lane == 0 && count) { atomicMin(t_range + 2, global_ns()); s_copied = 1; }
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
                    if (lane == 0) atomicMin(t_range + 3, global_ns());
                    first_row = false;
                }
            }
            if (q < W) {
                warp_from = (warp_from + count) % W;
            } else {                                                   // (all of them come: q and the phases are the same)
                warp_from = 0;
                asm volatile("bar.sync 1, %0;" :: "r"(W * 32u) : "memory");
            }
            if (++g == n_pub) { g = 0; base += round_size; }
        }
    }
    __syncthreads();
    return s_copied != 0;
}

}  // namespace avsg
