// Stage One of the AVSG operator: match + reserve, one thread block per table.
//
// Follows Algorithm 1 (refresh / classify / allocate) with the lifetime operations of Algorithm 3, for the N_q tokens
// of one iteration in order (Algorithm 4), and the end-of-step invalidation of Algorithm 4.
//
// The whole table lives in shared memory for the step:
//   s_node[n]  {id, slot << 16 | next node}: node n < S is slot n with its cached id; an id that comes in before the
//              last token gets a node of its own behind those, because its slot's node still hangs in the chain of the
//              id that it replaces (where it is passed over, its id being another one); the last node closes every chain
//   s_head[2S] the chains' first nodes: the index id -> slot, built from the cached ids at the start of every step
//   s_life[S]  lifetime per slot, one signed byte;  s_bits: one bit per slot, set where it is dead (lifetime < 0)
// The index is private to the kernel: a hit is "some slot holds the id" (Eq. 1), whatever node found it, so both
// exact index modes of the interface run it (AVSG_INDEX_DIRECT only adds the bound on the ids).
//
// What bounds it: nothing but latency.  A 32-table call touches 4 MB, 0.6 us of HBM time; the rest is a chain of
// dependent passes over shared memory on one SM per table.  So the passes are few and short:
//   * The index is chained and not open-addressed: an insert is one exchange whatever it meets, so a thread has all of
//     its eight in flight, and a chain is 1.25 nodes long on average where linear probing at half load goes through
//     clusters; what a warp pays for is the longest of its 32 lanes.  A step along a chain is one 8-byte read without a
//     branch: a lane that is through reads the closing node again.
//   * Three block barriers per token: lookups | misses and dead slots listed | install |.  Misses are ranked by ballots
//     (a warp takes 32 consecutive positions at a time, so lane order is position order) and the block prefix is two
//     warp reductions that every warp does for itself, over the warps' totals.  The dead slots of a warp are counted
//     when lifetimes decay; hits that revive one and slots that are handed out are taken off.  Only the warps that
//     hold some of the first n_g dead slots rank them, and the compacted misses are installed by a few warps: an SM
//     issues instructions for 32 warps here, and what all of them execute is what takes the time.
//   * The decay loop of Algorithm 1 ("decay all, CollectDead, until enough slots are dead") in closed form: d = the
//     smallest number of unit decays after which n_g lifetimes are negative, found by counting the lifetimes below up
//     to four candidate values at a time.
//   * Only what changed is written back: installed ids, the lifetimes, and ids that verification makes empty.
// Measured inside the kernel, 32 tables of 8192 slots, K = 2048, two tokens: 8.6 us.  With the open-addressing index of
// 4-byte keys and 2-byte slots, eight barriers and a lifetime histogram it was 30.0 us, and 12.7 us with a table of one
// 2-byte entry per context position in device memory; K = 256, S = 1024, one token: 2.5 us against 7.8.
//
// When Stage Two overlaps Stage One (S1Params::flags set), the block announces every token as soon as its misses are
// placed: see announce_token().
#include "avsg_kernels.cuh"
#include "follow_stage_one.cuh"
#include "stage_one_common.cuh"

namespace avsg {
namespace {

// Shared memory of one block, in bytes from its start (every part on a 16-byte boundary).
struct S1Layout {
    uint32_t head, life, bits, tot, ndead, cnt, sum, miss, pos, dead, total;
};
__host__ __device__ inline S1Layout s1_layout(uint32_t S, uint32_t K, uint32_t n_q, uint32_t nt)
{
    S1Layout o;
    uint32_t a = align16((S + (n_q - 1u) * K + 1u) * 8u);      // nodes first
    o.head = a;  a += 2u * S * 4u;
    o.life = a;  a += align16(S);
    o.bits = a;  a += align16(nt);
    o.tot = a;   a += 2u * 32u * 4u;                           // warps' miss totals, by parity
    o.ndead = a; a += 2u * 32u * 4u;                           // warps' dead slots, by parity
    o.cnt = a;   a += 2u * 2u * 32u * 4u;                      // warps' counts of the decay search, by parity
    o.sum = a;   a += 16u;                                     // valid ids of the call
    o.miss = a;  a += align16(K * 4u);                         // misses in position order: ids,
    o.pos = a;   a += align16(K * 2u);                         //   positions
    o.dead = a;  a += align16(K * 2u);                         // dead slots in slot order
    o.total = a;
    return o;
}

// SPT slots per thread (a power of two): S <= SPT * blockDim.x.  IPT: the most ids a thread has to look up per token
// (K <= S, so SPT is always enough).  CAP: tables the argument block has room for.  The block serves the tables block,
// block + blocks, ... of the launch.  WIDE: the state is aligned (state_is_aligned()).
template <int SPT, int IPT, bool WIDE, int CAP>
__device__ __forceinline__ void stage_one(const S1ParamsT<CAP>& p, const uint32_t block, const uint32_t blocks, unsigned char* smem)
{
    constexpr int NV = (SPT + 3) / 4;                    // 4-slot vectors of ids / words of lifetimes per thread
    const uint32_t S = p.S, K = p.K, H = 2u * S, L = p.L;
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u, warp = tid >> 5, nw = nt >> 5;
    const uint32_t below = (1u << lane) - 1u;            // the lanes before this one
    const uint32_t NIL = S + (p.n_q - 1u) * K;           // the closing node

    const S1Layout lay = s1_layout(S, K, p.n_q, nt);
    uint2*    s_node = reinterpret_cast<uint2*>(smem);
    uint32_t* s_head = reinterpret_cast<uint32_t*>(smem + lay.head);
    int8_t*   s_life = reinterpret_cast<int8_t*>(smem + lay.life);
    uint8_t*  s_bits = smem + lay.bits;                  // a thread's slots: set where dead
    uint32_t* s_tot  = reinterpret_cast<uint32_t*>(smem + lay.tot);
    uint32_t* s_ndead = reinterpret_cast<uint32_t*>(smem + lay.ndead);
    uint32_t* s_cnt  = reinterpret_cast<uint32_t*>(smem + lay.cnt);
    uint32_t* s_sum  = reinterpret_cast<uint32_t*>(smem + lay.sum);
    int32_t*  s_miss = reinterpret_cast<int32_t*>(smem + lay.miss);
    uint16_t* s_pos  = reinterpret_cast<uint16_t*>(smem + lay.pos);
    uint16_t* s_dead = reinterpret_cast<uint16_t*>(smem + lay.dead);

    auto clear_index = [&] {
        for (uint32_t i = tid; i < H / 4; i += nt) reinterpret_cast<uint4*>(s_head)[i] = make_uint4(NIL, NIL, NIL, NIL);
    };
    // slot j is no longer dead (the count follows the bit, so that an id that comes twice is counted once)
    auto revive = [&](uint32_t j, uint32_t par) {
        const uint32_t owner = j / SPT, bit = 1u << ((owner & 3u) * 8u + j % SPT);
        if (atomicAnd(reinterpret_cast<uint32_t*>(s_bits) + owner / 4u, ~bit) & bit)
            atomicSub(&s_ndead[par + owner / 32u], 1u);
    };
    const uint32_t ipt = (K + nt - 1) / nt;              // ids per thread
    const uint32_t i0 = warp * ipt * 32u + lane;         // position of the thread's k-th id: i0 + 32 k, below i1
    const uint32_t i1 = (warp + 1u) * ipt * 32u < K ? (warp + 1u) * ipt * 32u : K;
    int32_t xs[IPT];
    auto load_token = [&](uint32_t ti, uint32_t g) {
        const int32_t* ids = p.indices + ((size_t)ti * p.n_q + g) * K;
#pragma unroll
        for (int k = 0; k < IPT; ++k)
            xs[k] = i0 + 32u * k < i1 ? (p.host_ids ? __ldcv(ids + i0 + 32u * k) : __ldcg(ids + i0 + 32u * k)) : -1;
    };
    // the first table's arguments and the clearing come before the wait: under the previous kernel's tail
    uint32_t bt = block, table = p.table_id[bt], id_limit = p.id_limit[bt];
    int32_t N = p.verified_len[bt];
    clear_index();
    if (tid == 0) s_node[NIL] = make_uint2(0xFFFFFFFEu, NIL);          // an id that nobody looks for
    // Ids in host memory are there when the call is made, and nothing on the device writes them: a call that queues
    // behind another fetches its first ones while that one's rows travel (32 tables: 5 us of link time and a round trip).
    if (p.host_ids) load_token(p.first + bt, 0);

    // Programmatic dependent launch: this grid may have been started while the previous kernel of the stream
    // was still running; nothing that the device writes is read before that kernel has completed.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.t_range && tid == 0) atomicMin(p.t_range, global_ns());

    const uint32_t j0 = tid * SPT;                       // first of the thread's slots
    const bool own = j0 < S;

    // A block usually serves one table.  A call with many tables and an overlapped Stage Two is launched with fewer
    // blocks than tables: a block then serves the tables bt = block, block + blocks, ... one after the
    // other, so that Stage One stays on a few SMs and publishes its tables round by round while the transfer grid,
    // resident on the other SMs, already copies the earlier rounds' misses.
    for (;;) {
        const uint32_t ti = p.first + bt;                // table index within the call
        int32_t* g_tok = p.tok + (size_t)table * S;
        int8_t*  g_life = p.life + (size_t)table * S;

        // ---- every global load is issued first: cached ids, lifetimes, the first token's ids ----
        int4 t4[NV];
        uint32_t w[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if (tid + q * nt < S / 4) {
                const int32_t* at = g_tok + 4u * (tid + q * nt);
                if constexpr (WIDE) t4[q] = __ldcg(reinterpret_cast<const int4*>(at));
                else t4[q] = make_int4(__ldcg(at), __ldcg(at + 1), __ldcg(at + 2), __ldcg(at + 3));
            }
        life_words<SPT, true, WIDE>(g_life + j0, own, w);
        if (!p.host_ids || bt != block) load_token(ti, 0);
        if (p.verified_len_dev) N = __ldg(p.verified_len_dev + ti);
        const uint32_t seen = bt == block ? take_flags_down(p, bt, blocks, p.n_launch) : 0u;
        if (tid == 0) s_sum[0] = 0;
        __syncthreads();                                 // the index is empty

        // ---- ids to shared memory and into the index; global pre-decay of the lifetimes (Alg. 1 Pass 1) ----
        bool stale_ids = false;                          // ids that are no longer verified (the caller took tokens back)
#pragma unroll
        for (int q = 0; q < NV; ++q)
            if (tid + q * nt < S / 4) stale_ids = stale_ids || t4[q].x >= N || t4[q].y >= N || t4[q].z >= N || t4[q].w >= N;
        index_slots(t4, s_node, s_head, S, p.logH, NIL);
        uint32_t high = 0;                               // lifetimes above L (only a caller's own state can have them)
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            if (own) high |= __vcmpgts4(w[q], L * 0x01010101u) & (SPT == 2 ? 0xFFFFu : 0xFFFFFFFFu);
            w[q] = decay4(w[q], 1);
        }
        store_lifetimes<SPT>(s_life, s_bits, s_ndead, own, w);
        const bool unusual = __syncthreads_or(high != 0);

        uint32_t list_off = 0, sum_miss = 0, sum_decay = 0, valid = 0;
        int2* list = p.miss_list + (size_t)ti * p.list_stride;

        for (uint32_t g = 0; g < p.n_q; ++g) {
            const bool last = g + 1 == p.n_q;
            const uint32_t par = 32u * (g & 1u);
            const size_t row = ((size_t)ti * p.n_q + g) * K;
            int32_t* O = p.slots + row;
            uint8_t* Hm = p.hit ? p.hit + row : nullptr;

            // ---- lookups; hits: lifetime <- L, slot and flag out (Pass 1 + Pass 2) ----
            // (pass after pass over the thread's ids, so that their reads are in flight together)
            uint32_t rank[IPT], missing = 0, wmiss = 0;
            int32_t slot[IPT], was[IPT];
            bool bad = false;
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const bool ok = (uint32_t)xs[k] < id_limit;
                bad = bad || (!ok && xs[k] >= 0);
                xs[k] = ok ? xs[k] : -1;
                valid += ok;
            }
            if (bad) atomicOr(p.status, ST_BAD_ID);                    // not fetched: reported and taken as padding
            find_slots(xs, s_node, s_head, p.logH, NIL, p.status, slot);
            // with lifetimes above L on entry a slot reserved in this step may go to yet another id: its first node is stale
            if (unusual) {
#pragma unroll
                for (int k = 0; k < IPT; ++k)
                    if (slot[k] >= 0 && (int32_t)s_node[slot[k]].x != xs[k]) slot[k] = -1;
            }
#pragma unroll
            for (int k = 0; k < IPT; ++k) was[k] = slot[k] >= 0 ? s_life[slot[k]] : 0;
            bool revived = false;
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const bool miss = xs[k] >= 0 && slot[k] < 0, store = !miss && i0 + 32u * k < i1;
                const uint32_t votes = __ballot_sync(0xffffffffu, miss);
                rank[k] = wmiss + __popc(votes & below);               // within the warp, in position order
                wmiss += __popc(votes);
                missing |= miss ? 1u << k : 0u;
                if (slot[k] >= 0) s_life[slot[k]] = (int8_t)L;
                if (store) O[i0 + 32u * k] = slot[k];
                if (store && Hm) Hm[i0 + 32u * k] = slot[k] >= 0;
                revived = revived || was[k] < 0;
            }
            if (revived) {
#pragma unroll
                for (int k = 0; k < IPT; ++k)
                    if (was[k] < 0) revive((uint32_t)slot[k], par);
            }
            if (last) {
                valid = __reduce_add_sync(0xffffffffu, valid);
                if (lane == 0 && valid) atomicAdd(s_sum, valid);
            }
            if (lane == 0) s_tot[par + warp] = wmiss;
            if (g == 0 && bt == block && (p.flags || p.early)) start_dependents(seen);
            __syncthreads();

            // ---- CollectDead and the misses, each in order; the prefix over the warps: lane l looks at warp l ----
            uint32_t t = lane < nw ? s_ndead[par + lane] | s_tot[par + lane] << 16 : 0u;
            const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u);
            const uint32_t all = __reduce_add_sync(0xffffffffu, t);
            const uint32_t n_g = all >> 16;
            uint32_t dtotal = all & 0xFFFFu, dead_before = before & 0xFFFFu, d = 0;
            sum_miss += n_g;
            if (tid == 0 && p.miss_count) p.miss_count[(size_t)ti * p.n_q + g] = (int32_t)n_g;
            if (missing) {
#pragma unroll
                for (int k = 0; k < IPT; ++k) {
                    if (missing & (1u << k)) {
                        s_miss[(before >> 16) + rank[k]] = xs[k];
                        s_pos[(before >> 16) + rank[k]] = (uint16_t)(i0 + 32u * k);
                    }
                }
            }
            if (!last) load_token(ti, g + 1);                              // arrives while this token's misses are placed

            // Pass 3, the while-loop of Alg. 1: decay until n_g slots are dead
            if (dtotal < n_g) {
                life_words<SPT>(s_life + j0, own, w);
                d = decays_until(w, n_g, L, s_cnt);
#pragma unroll
                for (int q = 0; q < NV; ++q) w[q] = decay4(w[q], d);
                store_lifetimes<SPT>(s_life, s_bits, s_ndead + par, own, w);
                __syncthreads();
                t = lane < nw ? s_ndead[par + lane] : 0u;
                dead_before = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u);
                dtotal = __reduce_add_sync(0xffffffffu, t);
                if (dtotal < n_g && tid == 0) atomicOr(p.status, ST_NO_DEAD_SLOTS);
            }
            const uint32_t n_take = n_g < dtotal ? n_g : dtotal;
            if (dead_before < n_take) {                  // some of the first n_g dead slots are this warp's
                uint32_t bits = s_bits[tid], r, unused;
                warp_rank<SPT>(__popc(bits), below, r, unused);
                for (r += dead_before; bits && r < n_take; bits &= bits - 1u, ++r) s_dead[r] = (uint16_t)(j0 + __ffs((int)bits) - 1);
                s_bits[tid] = (uint8_t)bits;              // what is handed out is dead no more
            }
            uint32_t left = __shfl_sync(0xffffffffu, t & 0xFFFFu, (int)warp);          // the warp's dead slots for the next token
            if (dead_before < n_take) left = left > n_take - dead_before ? left - (n_take - dead_before) : 0u;
            if (lane == 0) s_ndead[32u - par + warp] = left;
            __syncthreads();

            // ---- install: the k-th miss in position order takes the k-th dead slot ----
            for (uint32_t k = tid; k < n_g; k += nt) {
                const uint32_t i = s_pos[k];
                const int32_t x = s_miss[k];
                const int32_t j = k < n_take ? s_dead[k] : -1;
                if (k < n_take) {
                    s_node[j].x = (uint32_t)x;
                    s_life[j] = (int8_t)L;
                    list[list_off + k] = make_int2(x, j);
                    g_tok[j] = x >= N ? -1 : x;                        // speculative ids are forgotten (end of Alg. 4)
                    if (!last) {
                        const uint32_t n = S + list_off + k;
                        s_node[n] = make_uint2((uint32_t)x, (uint32_t)j << 16 | atomicExch(&s_head[hash_id(x, p.logH)], n));
                    }
                }
                O[i] = j;
                if (Hm) Hm[i] = 0;
            }
            list_off += n_take;
            sum_decay += d;
            __syncthreads();
            announce_token(p, ti, g, n_take);
        }

        if (unusual) drop_lost_rows(list, list_off, s_node);

        // ---- write back: lifetimes; resident ids that are no longer verified become empty (Alg. 4) ----
        life_words<SPT>(s_life + j0, own, w);
        life_words_store<SPT, WIDE>(g_life + j0, own, w);
        if (stale_ids) {
            for (uint32_t q = 0; q < NV; ++q)
                for (uint32_t j = 4u * (tid + q * nt); j < 4u * (tid + q * nt) + 4u && j < S; ++j)
                    if ((int32_t)s_node[j].x >= N) g_tok[j] = -1;
        }
        if (tid == 0) {
            SegDesc sd;
            sd.src_base = p.kv_base[bt];
            sd.src_stride = p.kv_stride[bt];
            sd.dst_base = reinterpret_cast<uint64_t>(p.buffer + (size_t)table * S * p.row_bytes);
            sd.count = list_off;
            sd.pad = 0;
            p.seg[ti] = sd;
            TableStats* st = p.stats + table;            // (reductions: nothing waits for the old values)
            atomicAdd(&st->steps, 1ull);
            atomicAdd(&st->tokens, (unsigned long long)p.n_q);
            atomicAdd(&st->hits, (unsigned long long)(s_sum[0] - sum_miss));
            atomicAdd(&st->misses, (unsigned long long)sum_miss);
            atomicAdd(&st->rows, (unsigned long long)list_off);
            atomicAdd(&st->extra_decays, (unsigned long long)sum_decay);
        }
        bt += blocks;
        if (bt >= p.n_launch) break;
        table = p.table_id[bt]; id_limit = p.id_limit[bt]; N = p.verified_len[bt];
        __syncthreads();                                 // this table's last reads of shared memory are over
        clear_index();
    }
    if (p.t_range) {
        __syncthreads();
        if (tid == 0) atomicMax(p.t_range + 1, global_ns());
    }
}

template <int SPT, int IPT, int CAP, bool WIDE = true>
__global__ void __launch_bounds__(1024, 1) avsg_stage_one_kernel(const __grid_constant__ S1ParamsT<CAP> p)
{
    extern __shared__ __align__(16) unsigned char smem[];
    stage_one<SPT, IPT, WIDE>(p, blockIdx.x, gridDim.x, smem);
}

// A request ended: its tables become empty (id -1) and dead (lifetime -1) again, their counters and rows zero;
// in the paper-literal mode every bucket word returns to (lifetime -1, invalid, fingerprint 0, slot 0).  Grid (blocks per table, tables).
// What bounds it is the 43 MB of rows that eight tables have, at the rate of stores; so the device is filled with blocks
// whatever the number of tables, and the grid starts under the kernel before it and lets the next one start under itself
// (programmatic launch): eight tables in 7.5 us and not 10.4.
__global__ void __launch_bounds__(RESET_THREADS) avsg_reset_tables_kernel(const __grid_constant__ ResetParams p)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const size_t table = p.table_id[blockIdx.y];
    const size_t S = p.S, tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, nth = (size_t)gridDim.x * blockDim.x;
    int4* rows = reinterpret_cast<int4*>(p.buffer + table * S * p.row_bytes);
    const size_t chunks = S * (p.row_bytes >> 4);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (size_t i = tid; i < chunks; i += nth) rows[i] = make_int4(0, 0, 0, 0);
    for (size_t j = tid; j < S / 4; j += nth) {
        reinterpret_cast<int4*>(p.tok + table * S)[j] = make_int4(-1, -1, -1, -1);
        reinterpret_cast<uint32_t*>(p.life + table * S)[j] = 0xFFFFFFFFu;
        if (p.qword) reinterpret_cast<uint4*>(p.qword + table * S)[j] = make_uint4(0xFF800000u, 0xFF800000u, 0xFF800000u, 0xFF800000u);
    }
    if (tid == 0) p.stats[table] = TableStats{0, 0, 0, 0, 0, 0};
}

// ---------------------------------------------------------------------------------------------------------------
// Paper-literal Hash-State mode (Sec. 3.2-3.3, Eq. 2-4, Eq. 8-11, Algorithm 2): 64-bit entries (c_j, q_j) with
// q_j = [lifetime 8 | invalid 1 | fingerprint 23-m | slot m], double hashing with retry budget R, fingerprint
// check and lazy reclamation of stale bucket words.  Lossy by design: a resident id whose bucket word was
// overwritten is missed and fetched again.  Where Algorithm 2 leaves open which of several writers of one bucket
// wins, the miss with the highest position wins (an atomicMax on a per-bucket tag), so results are reproducible.
// ---------------------------------------------------------------------------------------------------------------
__device__ __forceinline__ void pack_life_bytes(const uint32_t* q, uint32_t j0, uint32_t spt, bool own,
                                                uint32_t& w0, uint32_t& w1)
{
    w0 = w1 = 0x7F7F7F7Fu;
    if (!own) return;
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)MAX_SPT; ++k) {
        if (k < spt) {
            const uint32_t b = q[j0 + k] >> 24;
            if (k < 4) w0 = (w0 & ~(0xFFu << (8 * k))) | (b << (8 * k));
            else w1 = (w1 & ~(0xFFu << (8 * (k - 4)))) | (b << (8 * (k - 4)));
        }
    }
}

__device__ __forceinline__ void unpack_life_bytes(uint32_t* q, uint32_t j0, uint32_t spt, bool own, uint32_t w0, uint32_t w1)
{
    if (!own) return;
#pragma unroll
    for (uint32_t k = 0; k < (uint32_t)MAX_SPT; ++k) {
        if (k < spt) {
            const uint32_t b = k < 4 ? (w0 >> (8 * k)) & 0xFFu : (w1 >> (8 * (k - 4))) & 0xFFu;
            q[j0 + k] = (q[j0 + k] & 0x00FFFFFFu) | (b << 24);
        }
    }
}

__global__ void __launch_bounds__(1024, 1) avsg_stage_one_paper_kernel(const __grid_constant__ S1Params p)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t S = p.S, K = p.K, Kp = (K + 7u) & ~7u, m = p.logH - 1u, Fm = (1u << (23u - m)) - 1u;
    const uint32_t tid = threadIdx.x, nt = blockDim.x, R = p.probe_retries, a1 = p.hash_a1, a2 = p.hash_a2;
    const int32_t L = (int32_t)p.L;

    int32_t*  s_c        = reinterpret_cast<int32_t*>(smem);
    uint32_t* s_q        = reinterpret_cast<uint32_t*>(s_c + S);
    uint32_t* s_win      = s_q + S;                                   // per-bucket winner tag of UpdateState
    int32_t*  s_miss_x   = reinterpret_cast<int32_t*>(s_win + S);
    uint16_t* s_miss_pos = reinterpret_cast<uint16_t*>(s_miss_x + Kp);
    uint16_t* s_dead     = s_miss_pos + Kp;
    uint16_t* s_bucket   = s_dead + Kp;                               // bit 15: a reusable bucket was found
    uint32_t* s_hist     = reinterpret_cast<uint32_t*>(s_bucket + Kp);
    uint32_t* s_scan_a   = s_hist + 128;
    uint32_t* s_scan_b   = s_scan_a + 40;
    const uint32_t priv_stride = nt + 4u;
    uint8_t*  s_priv     = L <= PRIV_HIST_MAX_L ? reinterpret_cast<uint8_t*>(s_scan_b + 40) : nullptr;

    const uint32_t ti = p.first + blockIdx.x, table = p.table_id[blockIdx.x];
    int32_t*  g_c = p.tok + (size_t)table * S;
    uint32_t* g_q = p.qword + (size_t)table * S;
    int8_t*   g_life = p.life + (size_t)table * S;
    const uint32_t spt = S >= nt ? S / nt : 1u, j0 = tid * spt;
    const bool own = j0 < S;
    const uint32_t ipt = (K + nt - 1) / nt, i0 = tid * ipt;

    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.t_range && threadIdx.x == 0) atomicMin(p.t_range, global_ns());

    start_dependents(take_flags_down(p, blockIdx.x, gridDim.x, p.n_launch));
    // ---- load the table; global pre-decay ----
    if (own)
        for (uint32_t k = 0; k < spt; ++k) {
            s_c[j0 + k] = __ldg(g_c + j0 + k);
            s_q[j0 + k] = __ldg(g_q + j0 + k);
            s_win[j0 + k] = 0;
        }
    if (s_priv)
        for (uint32_t i = tid; i < ((uint32_t)(L + 2) * priv_stride + 15u) / 16u; i += nt)
            reinterpret_cast<int4*>(s_priv)[i] = make_int4(0, 0, 0, 0);
    int32_t xs[MAX_IPT];
    load_ids(p.indices + (size_t)ti * p.n_q * K, i0, ipt, K, xs);
    __syncthreads();
    {
        uint32_t w0, w1;
        pack_life_bytes(s_q, j0, spt, own, w0, w1);
        unpack_life_bytes(s_q, j0, spt, own, decay4(w0, 1), decay4(w1, 1));
    }
    __syncthreads();

    uint32_t list_off = 0, sum_valid = 0, sum_miss = 0, sum_decay = 0;
    int2* list = p.miss_list + (size_t)ti * p.list_stride;

    for (uint32_t g = 0; g < p.n_q; ++g) {
        const size_t row = ((size_t)ti * p.n_q + g) * K;
        int32_t* O = p.slots + row;
        uint8_t* Hm = p.hit ? p.hit + row : nullptr;
        if (tid < 128) s_hist[tid] = 0;

        // ---- Probe (Eq. 8-11): at most R + 1 buckets; the full id is compared ----
        uint32_t missmask = 0, nmiss = 0, nvalid = 0;
        check_ids(xs, i0, ipt, K, p.id_limit[blockIdx.x], p.status);
#pragma unroll
        for (uint32_t k = 0; k < (uint32_t)MAX_IPT; ++k) {
            const uint32_t i = i0 + k;
            if (k < ipt && i < K) {
                const int32_t x = xs[k];
                if (x >= 0) {
                    ++nvalid;
                    uint32_t h = (a1 * (uint32_t)x) & (S - 1u);
                    const uint32_t d = ((a2 * (uint32_t)x) & (S - 1u)) | 1u;
                    int32_t j = -1;
                    for (uint32_t r = 0; r <= R; ++r) {
                        const uint32_t o = s_q[h] & (S - 1u);
                        if (s_c[o] == x) { j = (int32_t)o; break; }
                        if (r < R) h = (h + d) & (S - 1u);
                    }
                    if (j >= 0) {
                        reinterpret_cast<uint8_t*>(s_q)[4u * (uint32_t)j + 3u] = (uint8_t)L;    // lifetime <- L
                        O[i] = j;
                        if (Hm) Hm[i] = 1;
                    } else {
                        missmask |= 1u << k;
                        ++nmiss;
                    }
                } else {
                    O[i] = -1;
                    if (Hm) Hm[i] = 0;
                }
            }
        }
        uint32_t total;
        uint32_t off = block_excl_scan(nmiss | (nvalid << 16), s_scan_a, total) & 0xFFFFu;
        const uint32_t n_g = total & 0xFFFFu;
        sum_valid += total >> 16;
        sum_miss += n_g;
#pragma unroll
        for (uint32_t k = 0; k < (uint32_t)MAX_IPT; ++k) {
            if (missmask & (1u << k)) {
                s_miss_x[off] = xs[k];
                s_miss_pos[off] = (uint16_t)(i0 + k);
                ++off;
            }
        }
        if (g + 1 < p.n_q) load_ids(p.indices + row + K, i0, ipt, K, xs);
        if (tid == 0 && p.miss_count) p.miss_count[(size_t)ti * p.n_q + g] = (int32_t)n_g;
        if (n_g == 0) { __syncthreads(); publish_token(p, ti, g, 0); continue; }
        __syncthreads();

        // ---- CollectDead / decay until n_g slots are dead ----
        uint32_t w0, w1;
        pack_life_bytes(s_q, j0, spt, own, w0, w1);
        uint32_t sg0 = w0 & 0x80808080u, sg1 = w1 & 0x80808080u;
        uint32_t dtotal, d = 0;
        uint32_t doff = block_excl_scan(__popc(sg0) + __popc(sg1), s_scan_b, dtotal);
        if (dtotal < n_g) {
            count_lifetimes(w0, w1, spt, own, L, s_priv, priv_stride, s_hist);
            __syncthreads();
            uint32_t cum = 0;
            bool found = false;
            d = (uint32_t)L + 1u;
            for (uint32_t b = 0; b <= (uint32_t)L + 1u; ++b) {
                cum += s_hist[b];
                if (cum >= n_g) { d = b; found = true; break; }
            }
            if (!found && tid == 0) atomicOr(p.status, ST_NO_DEAD_SLOTS);
            w0 = decay4(w0, d);
            w1 = decay4(w1, d);
            unpack_life_bytes(s_q, j0, spt, own, w0, w1);
            sg0 = w0 & 0x80808080u; sg1 = w1 & 0x80808080u;
            doff = block_excl_scan(__popc(sg0) + __popc(sg1), s_scan_b, dtotal);
        }
#pragma unroll
        for (uint32_t k = 0; k < (uint32_t)MAX_SPT; ++k) {
            const uint32_t bit = k < 4 ? (sg0 >> (8 * k + 7)) & 1u : (sg1 >> (8 * (k - 4) + 7)) & 1u;
            if (bit) {
                if (doff < n_g) s_dead[doff] = (uint16_t)(j0 + k);
                ++doff;
            }
        }
        __syncthreads();
        const uint32_t n_take = n_g < dtotal ? n_g : dtotal;

        // ---- UpdateState (1): every miss looks for a reusable bucket on the table as it stands (Eq. 4) ----
        for (uint32_t k = tid; k < n_take; k += nt) {
            const int32_t x = s_miss_x[k];
            uint32_t h = (a1 * (uint32_t)x) & (S - 1u);
            const uint32_t dd = ((a2 * (uint32_t)x) & (S - 1u)) | 1u;
            uint32_t v = 0;
            for (uint32_t r = 0; r <= R; ++r) {
                const uint32_t qh = s_q[h], o = qh & (S - 1u);
                const uint32_t invalid = (qh >> 23) & 1u, fp = (qh >> m) & Fm;
                const int32_t life_o = (int32_t)(int8_t)(s_q[o] >> 24);
                v = invalid | (uint32_t)(life_o < 0) | (uint32_t)(fp != ((uint32_t)s_c[o] & Fm));
                if (v || r == R) break;
                h = (h + dd) & (S - 1u);
            }
            s_bucket[k] = (uint16_t)(h | (v ? 0x8000u : 0u));
        }
        __syncthreads();
        // ---- (2): ids and lifetimes go into the allocated slots ----
        for (uint32_t k = tid; k < n_take; k += nt) {
            const uint32_t j = s_dead[k], i = s_miss_pos[k];
            const int32_t x = s_miss_x[k];
            if (j < S && i < K) {
                s_c[j] = x;
                reinterpret_cast<uint8_t*>(s_q)[4u * j + 3u] = (uint8_t)L;
                O[i] = (int32_t)j;
                if (Hm) Hm[i] = 0;
                list[list_off + k] = make_int2(x, (int32_t)j);
                if (s_bucket[k] & 0x8000u) atomicMax(&s_win[s_bucket[k] & 0x7FFFu], ((g + 1u) << 16) | k);
            } else {
                list[list_off + k] = make_int2(-1, -1);
                atomicOr(p.status, ST_BAD_SLOT);
            }
        }
        __syncthreads();
        // ---- (3): the bucket word keeps its slot's lifetime, takes fingerprint and slot, becomes valid ----
        for (uint32_t k = tid; k < n_take; k += nt) {
            const uint32_t hb = s_bucket[k];
            if ((hb & 0x8000u) && s_win[hb & 0x7FFFu] == (((g + 1u) << 16) | k)) {
                const uint32_t h = hb & 0x7FFFu;
                s_q[h] = (s_q[h] & 0xFF000000u) | (((uint32_t)s_miss_x[k] & Fm) << m) | (uint32_t)s_dead[k];
            }
        }
        list_off += n_take;
        sum_decay += d;
        __syncthreads();
        publish_token(p, ti, g, n_take);
    }

    // ---- write back; speculative entries (id >= N) become empty ----
    const int32_t N = p.verified_len_dev ? __ldg(p.verified_len_dev + ti) : p.verified_len[blockIdx.x];
    if (own)
        for (uint32_t k = 0; k < spt; ++k) {
            const int32_t v = s_c[j0 + k];
            g_c[j0 + k] = v >= N ? -1 : v;
            g_q[j0 + k] = s_q[j0 + k];
            g_life[j0 + k] = (int8_t)(s_q[j0 + k] >> 24);
        }
    if (tid == 0) {
        SegDesc sd;
        sd.src_base = p.kv_base[blockIdx.x];
        sd.src_stride = p.kv_stride[blockIdx.x];
        sd.dst_base = reinterpret_cast<uint64_t>(p.buffer + (size_t)table * S * p.row_bytes);
        sd.count = list_off;
        sd.pad = 0;
        p.seg[ti] = sd;
        TableStats* st = p.stats + table;
        st->steps += 1;
        st->tokens += p.n_q;
        st->hits += sum_valid - sum_miss;
        st->misses += sum_miss;
        st->rows += list_off;
        st->extra_decays += sum_decay;
    }
    if (p.t_range) {
        __syncthreads();
        if (tid == 0) atomicMax(p.t_range + 1, global_ns());
    }
}

// "KV offload" comparator: every selected row moves, position (g, i) -> slot g*K + i.
__global__ void __launch_bounds__(256) avsg_all_k_prepare_kernel(const __grid_constant__ AllKParams p)
{
    __shared__ uint32_t s_valid;
    const uint32_t g = blockIdx.x, b = blockIdx.y, ti = p.first + b, K = p.K;
    const uint32_t table = p.table_id[b];
    if (threadIdx.x == 0) s_valid = 0;
    __syncthreads();
    const size_t row = ((size_t)ti * p.n_q + g) * K;
    int2* list = p.miss_list + (size_t)ti * p.list_stride + (size_t)g * K;
    uint32_t valid = 0;
    for (uint32_t i = threadIdx.x; i < K; i += blockDim.x) {
        int32_t x = __ldg(p.indices + row + i);
        if (x >= 0 && (uint32_t)x >= p.id_limit[b]) {             // beyond the table's host rows: not fetched
            atomicOr(p.status, ST_BAD_ID);
            x = -1;
        }
        const int32_t o = x >= 0 ? (int32_t)(g * K + i) : -1;
        p.slots[row + i] = o;
        if (p.hit) p.hit[row + i] = 0;
        list[i] = make_int2(x, o);
        valid += x >= 0;
    }
    valid = __reduce_add_sync(0xffffffffu, valid);
    if ((threadIdx.x & 31u) == 0 && valid) atomicAdd(&s_valid, valid);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (p.miss_count) p.miss_count[(size_t)ti * p.n_q + g] = (int32_t)s_valid;
        TableStats* st = p.stats + table;
        atomicAdd(&st->tokens, 1ull);
        atomicAdd(&st->misses, (unsigned long long)s_valid);
        atomicAdd(&st->rows, (unsigned long long)s_valid);
        if (g == 0) {
            SegDesc sd;
            sd.src_base = p.kv_base[b];
            sd.src_stride = p.kv_stride[b];
            sd.dst_base = reinterpret_cast<uint64_t>(p.buffer + (size_t)table * p.S * p.row_bytes);
            sd.count = p.n_q * K;
            sd.pad = 0;
            p.seg[ti] = sd;
            atomicAdd(&st->steps, 1ull);
        }
    }
}

}  // namespace

size_t stage_one_smem_bytes(uint32_t S, uint32_t K, uint32_t n_q)
{
    return s1_layout(S, K, n_q, stage_one_threads(S, K)).total;
}

static uint32_t stage_one_paper_threads(uint32_t S)
{
    const uint32_t t = S / 2;
    return t < 128 ? 128 : (t > 1024 ? 1024 : t);
}

size_t stage_one_paper_smem_bytes(uint32_t S, uint32_t K, uint32_t L)
{
    const size_t Kp = (K + 7u) & ~7u;
    size_t n = S * 12 + Kp * 4 + Kp * 2 * 3 + (128 + 40 + 40) * 4;
    if ((int32_t)L <= PRIV_HIST_MAX_L) n += ((size_t)(L + 2) * (stage_one_paper_threads(S) + 4) + 15) / 16 * 16;
    return n;
}

// Eight slots per thread when that leaves a thread at most two ids of a token, else four (at most 1024 threads).
// Measured inside the kernel, eight / four slots per thread: S = 4096, K = 1000: 3.9 / 4.5 us; S = 2048, K = 512, two
// tokens: 4.8 / 5.0; S = 4096, K = 2048, two tokens: 13.1 / 10.7; S = K = 2048: 8.3 / 6.8; S = 1024, K = 512, two
// tokens: 8.4 / 5.6 (two slots per thread: 6.4).
uint32_t stage_one_threads(uint32_t S, uint32_t K)
{
    const uint32_t t = K <= S / 4 ? S / 8 : S / 4;
    return t < 128 ? 128 : (t > 1024 ? 1024 : t);
}

cudaError_t stage_one_prepare(size_t max_smem)
{
    const void* kernels[] = {
        reinterpret_cast<const void*>(avsg_stage_one_kernel<2, 2, S1_MAX_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<4, 2, S1_MAX_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<4, 4, S1_MAX_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 2, S1_MAX_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 4, S1_MAX_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 8, S1_MAX_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<2, 2, S1_MAX_TABLES, false>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<4, 4, S1_MAX_TABLES, false>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 8, S1_MAX_TABLES, false>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<2, 2, S1_BIG_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<4, 2, S1_BIG_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<4, 4, S1_BIG_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 2, S1_BIG_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 4, S1_BIG_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_kernel<8, 8, S1_BIG_TABLES>),
        reinterpret_cast<const void*>(avsg_stage_one_paper_kernel)};
    for (const void* k : kernels) {
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(max_smem - fa.sharedSizeBytes));
        if (e != cudaSuccess) return e;
    }
    // The other kernels of this file are loaded now as well: the runtime loads a kernel at its first use, which may
    // have to wait for every stream of the device - forever, if a stream is waiting for something that very launch
    // would produce (a caller who arms a wait for a call's stage_one_done word before its first call).
    const void* others[] = {reinterpret_cast<const void*>(avsg_all_k_prepare_kernel),
                            reinterpret_cast<const void*>(avsg_reset_tables_kernel)};
    for (const void* k : others) {
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

namespace {
template <int CAP>
cudaError_t launch_stage_one_t(const S1ParamsT<CAP>& p, uint32_t n_blocks, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_blocks);
    cfg.blockDim = dim3(stage_one_threads(p.S, p.K));
    cfg.dynamicSmemBytes = stage_one_smem_bytes(p.S, p.K, p.n_q);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const uint32_t ipt = (p.K + cfg.blockDim.x - 1) / cfg.blockDim.x;      // ids per thread
    if constexpr (CAP == S1_MAX_TABLES)
        if (!state_is_aligned(p.tok, p.life))
            switch (p.S / cfg.blockDim.x) {
                case 8:  return cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<8, 8, CAP, false>, p);
                case 4:  return cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<4, 4, CAP, false>, p);
                default: return cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<2, 2, CAP, false>, p);
            }
    switch (p.S / cfg.blockDim.x) {
        case 8:  return ipt <= 2 ? cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<8, 2, CAP>, p)
                      : ipt <= 4 ? cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<8, 4, CAP>, p)
                                 : cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<8, 8, CAP>, p);
        case 4:  return ipt <= 2 ? cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<4, 2, CAP>, p)
                                 : cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<4, 4, CAP>, p);
        default: return cudaLaunchKernelEx(&cfg, avsg_stage_one_kernel<2, 2, CAP>, p);
    }
}
}  // namespace

cudaError_t launch_stage_one(const S1Params& p, uint32_t n_tables, cudaStream_t stream)
{
    if (p.qword == nullptr) return launch_stage_one_t(p, n_tables, stream);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_tables);
    cfg.blockDim = dim3(stage_one_paper_threads(p.S));
    cfg.dynamicSmemBytes = stage_one_paper_smem_bytes(p.S, p.K, p.L);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, avsg_stage_one_paper_kernel, p);
}

cudaError_t launch_stage_one(const S1ParamsBig& p, uint32_t n_tables, cudaStream_t stream)
{
    return launch_stage_one_t(p, n_tables, stream);
}

cudaError_t launch_reset_tables(const ResetParams& p, uint32_t n_tables, uint32_t sm_count, cudaStream_t stream)
{
    const uint32_t per_sm = 2048 / RESET_THREADS;        // blocks
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((sm_count * per_sm + n_tables - 1) / n_tables, n_tables);
    cfg.blockDim = dim3(RESET_THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, avsg_reset_tables_kernel, p);
}

cudaError_t launch_all_k_prepare(const AllKParams& p, uint32_t n_tables, cudaStream_t stream)
{
    avsg_all_k_prepare_kernel<<<dim3(p.n_q, n_tables), 256, 0, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace avsg
