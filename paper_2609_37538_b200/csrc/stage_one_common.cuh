// Device helpers of the Stage One kernels: thread-block clusters, packed lifetimes, warp ranks and the hand-over to the
// overlapped Stage Two, shared by all of them; id loads, the range check and the lifetime histogram of the paper-literal one.
#pragma once
#include "avsg_kernels.cuh"

namespace avsg {

__host__ __device__ inline uint32_t align16(uint32_t n) { return (n + 15u) & ~15u; }

constexpr int32_t PRIV_HIST_MAX_L = 30;   // private byte-counter histogram up to this L (32 rows)

// ---- thread-block clusters ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r; asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r)); return r;
}
// the address of the same shared-memory location in block `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank)
{
    uint32_t r; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank)); return r;
}
__device__ __forceinline__ void stc_u32(uint32_t a, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void addc_u32(uint32_t a, uint32_t v)
{
    asm volatile("red.shared::cluster.add.u32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
// Four or eight bytes into another block's shared memory, counted there by an mbarrier: no fence on either side.
__device__ __forceinline__ void send_async(uint32_t a, int32_t x, int32_t y, uint32_t mbar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];"
                 :: "r"(a), "r"(x), "r"(y), "r"(mbar) : "memory");
}
__device__ __forceinline__ void send_async(uint32_t a, uint32_t v, uint32_t mbar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" :: "r"(a), "r"(v), "r"(mbar) : "memory");
}
// Another block's mbarrier: its one arrival, with the bytes that are sent to it.
__device__ __forceinline__ void arrive_expect(uint32_t mbar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t arrivals)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n\tfence.mbarrier_init.release.cluster;" :: "r"(mbar), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar)              // the block's own
{
    asm volatile("{\n\t.reg .b64 s;\n\tmbarrier.arrive.release.cta.shared::cta.b64 s, [%0];\n\t}" :: "r"(mbar) : "memory");
}
__device__ __forceinline__ bool mbar_done(uint32_t mbar)
{
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0, %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(mbar), "r"(1000u) : "memory");     // (asked for 1 us, suspended 4)
    return done != 0;
}
// All threads of all blocks of the cluster; earlier (distributed) shared-memory and global writes of the cluster
// are visible to every thread of the cluster afterwards.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }

__device__ __forceinline__ uint32_t hash_id(int32_t x, uint32_t logH)
{
    return ((uint32_t)x * 2654435769u) >> (32u - logH);
}

// life <- max(life - d, -1) on four packed signed bytes
__device__ __forceinline__ uint32_t decay4(uint32_t w, uint32_t d)
{
    return __vmaxs4(__vsubss4(w, d * 0x01010101u), 0xFFFFFFFFu);
}

// The lifetimes of a thread's SPT consecutive slots (2, 4, 8 or 16), packed one signed byte each, four to a word; unused
// bytes carry 0x7F (never counted, never dead).  GLOBAL: from global memory, past L1; WIDE: `at` is a multiple of SPT.
template <int SPT, bool GLOBAL = false, bool WIDE = true>
__device__ __forceinline__ void life_words(const int8_t* at, bool own, uint32_t (&w)[(SPT + 3) / 4])
{
#pragma unroll
    for (int q = 0; q < (SPT + 3) / 4; ++q) w[q] = 0x7F7F7F7Fu;
    if (!own) return;
    if constexpr (!WIDE) {
#pragma unroll
        for (int k = 0; k < SPT; ++k) {
            const uint32_t v = (uint8_t)__ldcg(reinterpret_cast<const signed char*>(at) + k);
            w[k / 4] = (w[k / 4] & ~(0xFFu << (8 * (k & 3)))) | v << (8 * (k & 3));
        }
    } else if constexpr (SPT == 16) {
        const uint4 v = GLOBAL ? __ldcg(reinterpret_cast<const uint4*>(at)) : *reinterpret_cast<const uint4*>(at);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else if constexpr (SPT == 8) {
        const uint2 v = GLOBAL ? __ldcg(reinterpret_cast<const uint2*>(at)) : *reinterpret_cast<const uint2*>(at);
        w[0] = v.x; w[1] = v.y;
    } else if constexpr (SPT == 4) {
        w[0] = GLOBAL ? __ldcg(reinterpret_cast<const uint32_t*>(at)) : *reinterpret_cast<const uint32_t*>(at);
    } else {
        w[0] = 0x7F7F0000u | (GLOBAL ? __ldcg(reinterpret_cast<const uint16_t*>(at)) : *reinterpret_cast<const uint16_t*>(at));
    }
}

template <int SPT, bool WIDE = true>
__device__ __forceinline__ void life_words_store(int8_t* at, bool own, const uint32_t (&w)[(SPT + 3) / 4])
{
    if (!own) return;
    if constexpr (!WIDE) {
#pragma unroll
        for (int k = 0; k < SPT; ++k) at[k] = (int8_t)(w[k / 4] >> (8 * (k & 3)));
    }
    else if constexpr (SPT == 16) *reinterpret_cast<uint4*>(at) = make_uint4(w[0], w[1], w[2], w[3]);
    else if constexpr (SPT == 8) *reinterpret_cast<uint2*>(at) = make_uint2(w[0], w[1]);
    else if constexpr (SPT == 4) *reinterpret_cast<uint32_t*>(at) = w[0];
    else *reinterpret_cast<uint16_t*>(at) = (uint16_t)w[0];
}

// ---- the chained index id -> slot (see stage_one.cu): nodes {id, slot << 16 | next node}, chains' first nodes ----
// The thread's q-th vector of ids is that of the slots from 4 (tid + q blockDim.x) on; node n < S is slot n.
template <int NV>
__device__ __forceinline__ void index_slots(const int4 (&t4)[NV], uint2* s_node, uint32_t* s_head, uint32_t S, uint32_t log_heads, uint32_t nil)
{
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (threadIdx.x + q * blockDim.x < S / 4) {
            const uint32_t j = 4u * (threadIdx.x + q * blockDim.x);
            const int32_t x[4] = {t4[q].x, t4[q].y, t4[q].z, t4[q].w};
            uint32_t next[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) next[c] = x[c] >= 0 ? atomicExch(&s_head[hash_id(x[c], log_heads)], j + c) : nil;
#pragma unroll
            for (int c = 0; c < 4; c += 2)
                reinterpret_cast<uint4*>(s_node)[(j + c) / 2] = make_uint4((uint32_t)x[c], (j + c) << 16 | next[c],
                                                                           (uint32_t)x[c + 1], (j + c + 1) << 16 | next[c + 1]);
        }
    }
}

// The slots of M ids (-1: none; an id of -1 is not looked for).
template <int M>
__device__ __forceinline__ void find_slots(const int32_t (&x)[M], const uint2* s_node, const uint32_t* s_head,
                                           uint32_t log_heads, uint32_t nil, uint32_t* status, int32_t (&slot)[M])
{
    uint32_t node[M];
#pragma unroll
    for (int k = 0; k < M; ++k) {
        slot[k] = -1;
        node[k] = nil;
        if (x[k] >= 0) node[k] = s_head[hash_id(x[k], log_heads)];
    }
    uint32_t open = 1;
    for (uint32_t it = 0; open && it <= nil; ++it) {                   // all chains of the warp side by side
        uint2 v[M];
#pragma unroll
        for (int k = 0; k < M; ++k) v[k] = s_node[node[k]];
        open = 0;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const bool found = (int32_t)v[k].x == x[k];
            slot[k] = found ? (int32_t)(v[k].y >> 16) : slot[k];
            node[k] = found ? nil : v[k].y & 0xFFFFu;
            open |= node[k] ^ nil;
        }
        open = __any_sync(0xffffffffu, open);
    }
    if (open) atomicOr(status, ST_PROBE_EXHAUSTED);
}

// The same index where nodes of eight bytes do not fit (tables of 16384 slots): ids, links of two bytes, and the slots of the nodes
// from S on, each in a place of its own; as many chains as there is room for.
struct PackedIndex {
    int32_t*  id;                        // [nil + 1]
    uint16_t* link;                      // [nil + 1]
    uint16_t* slot;                      // [nil - S]: of node S, S + 1, ...
    uint32_t* head;                      // [heads]
    uint32_t  heads, nil, S;
    __device__ __forceinline__ uint32_t* chain(int32_t x) const { return head + __umulhi((uint32_t)x * 2654435769u, heads); }
};

template <int NV>
__device__ __forceinline__ void index_slots(const int4 (&t4)[NV], const PackedIndex& ix)
{
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (threadIdx.x + q * blockDim.x < ix.S / 4) {
            const uint32_t j = 4u * (threadIdx.x + q * blockDim.x);
            const int32_t x[4] = {t4[q].x, t4[q].y, t4[q].z, t4[q].w};
            uint32_t next[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) next[c] = x[c] >= 0 ? atomicExch(ix.chain(x[c]), j + c) : ix.nil;
            reinterpret_cast<int4*>(ix.id)[j / 4] = t4[q];
            reinterpret_cast<uint2*>(ix.link)[j / 4] = make_uint2(next[0] | next[1] << 16, next[2] | next[3] << 16);
        }
    }
}

template <int M>
__device__ __forceinline__ void find_slots(const int32_t (&x)[M], const PackedIndex& ix, uint32_t* status, int32_t (&slot)[M])
{
    uint32_t node[M];
#pragma unroll
    for (int k = 0; k < M; ++k) {
        slot[k] = -1;
        node[k] = ix.nil;
        if (x[k] >= 0) node[k] = *ix.chain(x[k]);
    }
    uint32_t open = 1;
    for (uint32_t it = 0; open && it <= ix.nil; ++it) {
        int32_t id[M];
        uint32_t next[M];
#pragma unroll
        for (int k = 0; k < M; ++k) { id[k] = ix.id[node[k]]; next[k] = ix.link[node[k]]; }
        open = 0;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const bool found = id[k] == x[k];
            slot[k] = found ? (int32_t)node[k] : slot[k];
            node[k] = found ? ix.nil : next[k];
            open |= node[k] ^ ix.nil;
        }
        open = __any_sync(0xffffffffu, open);
    }
    if (open) atomicOr(status, ST_PROBE_EXHAUSTED);
#pragma unroll
    for (int k = 0; k < M; ++k)
        if (slot[k] >= (int32_t)ix.S) slot[k] = ix.slot[slot[k] - (int32_t)ix.S];
}

// With lifetimes above L on entry a slot that one token of a call reserves may be reserved again by a later one.  Nothing orders
// the copies of a call's rows, so only the last reservation's row may be copied: the entries {id, slot (and more, from bit
// LIST_SLOT_BITS on)} of a table's list whose slots hold another id by now become padding.  All threads of the block, behind a
// barrier; thread t has the entries t, t + blockDim.x, ...  Lifetimes above L come with a caller's own state only, so with no
// Stage Two that already follows the list.
constexpr uint32_t LIST_SLOT_BITS = 13;                  // S <= 8192 here
__device__ __forceinline__ void drop_lost_rows(int2* list, uint32_t count, const uint2* s_node)
{
    for (uint32_t e = threadIdx.x; e < count; e += blockDim.x) {
        const int2 v = list[e];
        if ((int32_t)s_node[(uint32_t)v.y & ((1u << LIST_SLOT_BITS) - 1u)].x != v.x) list[e].x = -1;
    }
}

// Bits 0 .. 3: the sign bits of a word's four bytes.
__device__ __forceinline__ uint32_t signs(uint32_t w) { return (((w >> 7) & 0x01010101u) * 0x10204080u) >> 28; }

// A thread's slots as bits.
template <int SPT> struct SlotBits { using type = uint8_t; };
template <> struct SlotBits<16> { using type = uint16_t; };

// The thread's lifetimes to shared memory, its dead slots as bits, the warp's number of them.
template <int SPT>
__device__ __forceinline__ void store_lifetimes(int8_t* s_life, typename SlotBits<SPT>::type* s_bits, uint32_t* s_ndead, bool own,
                                                const uint32_t (&w)[(SPT + 3) / 4])
{
    uint32_t bits = 0;
#pragma unroll
    for (int q = 0; q < (SPT + 3) / 4; ++q) bits |= signs(w[q]) << (4 * q);
    life_words_store<SPT>(s_life + threadIdx.x * SPT, own, w);
    s_bits[threadIdx.x] = (typename SlotBits<SPT>::type)bits;
    const uint32_t n = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(bits));
    if ((threadIdx.x & 31u) == 0) s_ndead[threadIdx.x >> 5] = n;
}

// The while-loop of Alg. 1 in closed form: the fewest unit decays after which n_g of the block's lifetimes are negative
// (L + 1 where even those are too few; lifetimes are <= L).  All threads of the block; s_cnt: 4 x 32 words.
template <int NV>
__device__ __forceinline__ uint32_t decays_until(const uint32_t (&w)[NV], uint32_t n_g, uint32_t L, uint32_t* s_cnt)
{
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t lo = 0, hi = L + 1u, buf = 0;               // lo decays are too few, hi are enough
    while (hi - lo > 1u) {                               // (L >= 1: at least once, so every warp has read the old counts)
        uint32_t c[4];                                   // candidates in (lo, hi), ascending; small ones first
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) {
            c[i] = lo == 0 ? 1u << i : lo + ((i + 1u) * (hi - lo)) / 5u;
            c[i] = c[i] <= lo ? lo + 1u : (c[i] >= hi ? hi - 1u : c[i]);
        }
        uint32_t n01 = 0, n23 = 0;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            n01 += __popc(__vsubss4(w[q], c[0] * 0x01010101u) & 0x80808080u) |
                   (__popc(__vsubss4(w[q], c[1] * 0x01010101u) & 0x80808080u) << 16);
            n23 += __popc(__vsubss4(w[q], c[2] * 0x01010101u) & 0x80808080u) |
                   (__popc(__vsubss4(w[q], c[3] * 0x01010101u) & 0x80808080u) << 16);
        }
        n01 = __reduce_add_sync(0xffffffffu, n01);
        n23 = __reduce_add_sync(0xffffffffu, n23);
        if (lane == 0) { s_cnt[buf + warp] = n01; s_cnt[buf + 32u + warp] = n23; }
        __syncthreads();
        n01 = __reduce_add_sync(0xffffffffu, lane < nw ? s_cnt[buf + lane] : 0u);
        n23 = __reduce_add_sync(0xffffffffu, lane < nw ? s_cnt[buf + 32u + lane] : 0u);
        const uint32_t n[4] = {n01 & 0xFFFFu, n01 >> 16, n23 & 0xFFFFu, n23 >> 16};
#pragma unroll
        for (int i = 3; i >= 0; --i) if (n[i] >= n_g) hi = c[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) if (n[i] < n_g) lo = c[i];
        buf ^= 64u;
    }
    return hi;
}

// Exclusive prefix over the lanes and total of a count 0 .. MAX that every lane of the warp has: one ballot per bit.
template <int MAX>
__device__ __forceinline__ void warp_rank(uint32_t n, uint32_t below, uint32_t& rank, uint32_t& total)
{
    rank = total = 0;
#pragma unroll
    for (int bit = 0; (1 << bit) <= MAX; ++bit) {
        const uint32_t v = __ballot_sync(0xffffffffu, (n >> bit) & 1u);
        rank += __popc(v & below) << bit;
        total += __popc(v) << bit;
    }
}

// The ids a thread handles for one token: positions i0 .. i0+ipt-1.
__device__ __forceinline__ void load_ids(const int32_t* X, uint32_t i0, uint32_t ipt, uint32_t K, int32_t (&xs)[MAX_IPT])
{
    if ((ipt & 3u) == 0 && (K & 3u) == 0 && ((reinterpret_cast<uintptr_t>(X) & 15u) == 0)) {
#pragma unroll
        for (uint32_t q = 0; q < (uint32_t)MAX_IPT / 4; ++q) {
            if (4 * q < ipt && i0 + 4 * q < K) {
                const int4 v = __ldg(reinterpret_cast<const int4*>(X + i0) + q);
                xs[4 * q] = v.x; xs[4 * q + 1] = v.y; xs[4 * q + 2] = v.z; xs[4 * q + 3] = v.w;
            }
        }
    } else if (ipt == 2 && (K & 1u) == 0 && ((reinterpret_cast<uintptr_t>(X) & 7u) == 0)) {
        if (i0 < K) {
            const int2 v = __ldg(reinterpret_cast<const int2*>(X + i0));
            xs[0] = v.x; xs[1] = v.y;
        }
    } else {
#pragma unroll
        for (uint32_t k = 0; k < (uint32_t)MAX_IPT; ++k)
            if (k < ipt && i0 + k < K) xs[k] = __ldg(X + i0 + k);
    }
}

// Ids at or beyond the table's host row count (or, with the direct index, beyond its index) are never read from
// host memory: they are reported in the status word and then handled like padding.
__device__ __forceinline__ void check_ids(int32_t (&xs)[MAX_IPT], uint32_t i0, uint32_t ipt, uint32_t K, uint32_t limit,
                                          uint32_t* status)
{
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)MAX_IPT; ++k)
        if (k < ipt && i0 + k < K && xs[k] >= 0 && (uint32_t)xs[k] >= limit) {
            atomicOr(status, ST_BAD_ID);
            xs[k] = -1;
        }
}

// Lifetime histogram of the table: s_hist[v + 1] = number of slots with lifetime v, v = -1 .. L.
// s_hist must be zero on entry.  w0/w1 are the thread's packed lifetimes (life_load).
__device__ __forceinline__ void count_lifetimes(uint32_t w0, uint32_t w1, uint32_t spt, bool own, int32_t L,
                                                uint8_t* s_priv, uint32_t priv_stride, uint32_t* s_hist)
{
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u;
    if (s_priv) {
        // private byte counters: row = lifetime value + 1, column = thread; no atomics
        if (own) {
#pragma unroll
            for (uint32_t k = 0; k < (uint32_t)MAX_SPT; ++k) {
                if (k < spt) {
                    const uint32_t byte = ((k < 4 ? w0 >> (8 * k) : w1 >> (8 * (k - 4))) + 1u) & 0xFFu;   // value + 1
                    s_priv[byte * priv_stride + tid] += 1;
                }
            }
        }
        __syncthreads();
        // one warp per row: sum nt byte counters with dp4a and clear them for the next use
        const uint32_t words = nt >> 2;
        for (uint32_t row = tid >> 5; row <= (uint32_t)L + 1u; row += nt >> 5) {
            uint32_t* r = reinterpret_cast<uint32_t*>(s_priv + row * priv_stride);
            uint32_t acc = 0;
            for (uint32_t i = lane; i < words; i += 32u) {
                acc = __dp4a(r[i], 0x01010101u, acc);
                r[i] = 0;
            }
            acc = __reduce_add_sync(0xffffffffu, acc);
            if (lane == 0) s_hist[row] = acc;
        }
    } else {
        for (int32_t v = -1; v <= L; ++v) {
            const uint32_t vv = (uint32_t)(v & 0xFF) * 0x01010101u;
            uint32_t c = (__popc(__vcmpeq4(w0, vv)) + __popc(__vcmpeq4(w1, vv))) >> 3;
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0 && c) atomicAdd(&s_hist[v + 1], c);
        }
    }
}

// Takes down the hand-over flags of the block's tables, once the previous call of the context has completed
// (griddepcontrol.wait); `tables` of this launch, every `step`-th from `from` on.  The next kernel of the stream may start
// when every block has called start_dependents() with what this returned: so no flag of an earlier call is ever seen, and
// nothing has to be counted or zeroed behind a call.  Atomic exchanges, because their results say that they are done: a
// store and a fence in their place held up the block's first warp, and so its first barrier, by 0.5 us.
template <typename P>
__device__ __forceinline__ uint32_t take_flags_down(const P& p, uint32_t from, uint32_t step, uint32_t tables)
{
    uint32_t seen = 0;
    if (p.flags && threadIdx.x < 32u) {                  // lane: (table, token); at most eight tokens
        const uint32_t at_once = 32u / p.n_q, i = threadIdx.x / p.n_q, g = threadIdx.x % p.n_q;
        if (i < at_once)
            for (uint32_t bt = from + i * step; bt < tables; bt += at_once * step)
                seen |= atomicExch(p.flags + (size_t)(p.first + bt) * p.n_q + g, 0u);
    }
    return seen;
}

__device__ __forceinline__ void start_dependents(uint32_t seen)
{
    if (threadIdx.x < 32u && __all_sync(0xffffffffu, seen != 0xFFFFFFFFu) && threadIdx.x == 0)     // (no flag has that value)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Calls that asked for it (host buffers in the overlapped mode, or a caller's own signal word): the block that arrives last
// after the call's last token announces that every table of the call has written its slot table, hit mask and miss counts.
// The arrivals are counted in a word of their own that wraps to zero by itself (atomicInc).  One thread per block.
template <typename P>
__device__ __forceinline__ void announce_call(const P& p, bool announce)
{
    if (announce && atomicInc(p.done_ctr, p.expect - 1u) == p.expect - 1u) {
        __threadfence();
        *reinterpret_cast<volatile unsigned long long*>(p.done_seq) = p.host_seq;
    }
}

// Tells the overlapped transfer kernel, which is already resident (p.flags set), that token g of this table is placed:
// `count` more entries of the table's miss list are final.  Called by every thread of the block after a barrier behind
// the list writes; one thread then fences (the barrier makes the fence cover the whole block's earlier writes, as in a
// grid-wide barrier) and raises the table's flag.  SHARED: one of several blocks that place the table, each for itself.
template <bool SHARED = false, typename P>
__device__ __forceinline__ void announce_token(const P& p, uint32_t ti, uint32_t g, uint32_t count)
{
    const bool announce = p.done_seq && g + 1 == p.n_q;
    if ((!p.flags && !announce) || threadIdx.x != 0) return;
    __threadfence();
    if (p.flags) {
        if constexpr (SHARED) atomicAdd(p.flags + (size_t)ti * p.n_q + g, ANNOUNCED + count);
        else *reinterpret_cast<volatile uint32_t*>(p.flags + (size_t)ti * p.n_q + g) = ANNOUNCED + count;
    }
    announce_call(p, announce);
}

// The same with the barrier in front.
template <typename P>
__device__ __forceinline__ void publish_token(const P& p, uint32_t ti, uint32_t g, uint32_t count)
{
    if (!p.flags && !(p.done_seq && g + 1 == p.n_q)) return;
    __syncthreads();
    announce_token(p, ti, g, count);
}

}  // namespace avsg
