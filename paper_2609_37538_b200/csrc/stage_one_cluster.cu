// Stage One of the AVSG operator across a thread-block cluster: one table per cluster of C blocks (C = 2, 4, 8), for
// tables that one SM's shared memory does not hold (S up to 32768 slots; of 16384 slots those calls that avsg_step_kernel does
// not serve).
//
// Same results as the single-block kernel (Algorithm 1 with the lifetime operations of Algorithm 3, the tokens of an
// iteration in order as in Algorithm 4, the end-of-step invalidation), and the same index, bits and passes; see there.
//
// What bounds it is again latency, and here above all what crosses blocks.  So block r of the cluster owns the slots
// [r S/C, (r+1) S/C) with an index of its own over the ids in them, and looks up EVERY position of a token in it: no
// lookup, hit or install touches another block's shared memory.  (Before, positions were split over the blocks and ids,
// lifetimes and buckets of other blocks were read and written through distributed shared memory, with three cluster
// barriers per token.)  What the blocks tell one another, once per token, goes by remote stores and additions that
// nobody waits for, followed by ONE cluster barrier:
//   * a bit per position that is a hit in the block (block 0 also sets those of padding): what no block has set is a
//     miss, and every block sees the whole token's misses in position order;
//   * the number of dead slots that the block's hits have revived.  The dead slots of every block are known to all at
//     any time: a decay announces them anew, and how many of them a token takes follows from the same numbers.
// So every block computes for itself how many slots have to be taken and which of the misses are its own: the k-th dead
// slot in slot order (block order, then the block's) takes the k-th miss in position order, and the block that owns the
// slot selects that miss from the bits and installs it.  A decay adds a barrier per four candidate values of d and one
// for the new dead counts.  For an overlapped Stage Two every block announces its own misses of a token, on one flag that
// they add to: where block 0 announced them all behind one more barrier of the cluster, Stage One took 25.4 us beside the
// transfer grid and not 23.6 (16 tables, four tokens), and the call 108.7 us and not 108.2.
// Measured inside the kernel, 16 tables, K = 2048, four tokens: S = 16384 (C = 2) 22.3 us, S = 32768 (C = 4) 21.8 us.  With
// positions split over the blocks: 85 and 70 us with a distributed open-addressing index, 40 and 42 with an entry per
// context position in device memory.  S = 32768, K = 8192, three tokens, four tables: 35 us against 133.
#include "avsg_kernels.cuh"
#include "stage_one_common.cuh"

namespace avsg {
namespace {

constexpr uint32_t MAX_CL = 8;          // largest cluster (the portable limit)
constexpr uint32_t SMEM_LIMIT = 227u << 10;

// Shared-memory layout of one block (the same in every block of the cluster, so that a location's address in another
// block follows from the local one).  Nodes come first; a call takes each of the block's slots once at most.
struct Layout {
    uint32_t heads, nil;                                        // numbers, not offsets: chains, the closing node
    uint32_t head, life, bits, ndead, dead, pref, mask, rev, cnt, sum, total;
};
__host__ __device__ inline Layout make_layout(uint32_t S, uint32_t K, uint32_t n_q, uint32_t C, uint32_t nt)
{
    const uint32_t Sc = S / C, W = (K + 31u) / 32u, extra = (n_q - 1u) * K < Sc ? (n_q - 1u) * K : Sc;
    Layout o;
    o.heads = 2u * Sc;
    o.nil = Sc + extra;
    for (;;) {
        uint32_t a = align16((o.nil + 1u) * 8u);
        o.head = a;  a += o.heads * 4u;
        o.life = a;  a += align16(Sc);
        o.bits = a;  a += align16(nt);
        o.ndead = a; a += 2u * 32u * 4u;                        // warps' dead slots, by parity
        o.dead = a;  a += align16((K < Sc ? K : Sc) * 2u);      // the block's dead slots that are taken
        o.pref = a;  a += align16(W * 2u);                      // misses before each word of the mask
        o.mask = a;  a += align16(2u * C * W * 4u);             // received: positions that are no miss [parity][block][word]
        o.rev = a;   a += 2u * MAX_CL * 4u;                     // received: revived slots [parity][block]
        o.cnt = a;   a += 3u * (2u + MAX_CL) * 4u;              // received: counts of the decay search, dead slots, in turn
        o.sum = a;   a += 16u;
        o.total = a;
        if (a <= SMEM_LIMIT || o.heads <= Sc) return o;
        o.heads = Sc;                                           // (longer chains where the rest needs the room)
    }
}

constexpr int IPT = 2;                  // words of 32 positions that a warp looks up at a time

// SPT: the block's slots per thread (a power of two); CAP: tables the argument block has room for.
template <int SPT, int CAP>
__global__ void __launch_bounds__(1024, 1) avsg_stage_one_cluster_kernel(const __grid_constant__ S1ParamsT<CAP> p)
{
    constexpr int NV = (SPT + 3) / 4;
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t rank = cluster_rank(), C = cluster_size();
    const uint32_t S = p.S, K = p.K, L = p.L, Sc = S / C, W = (K + 31u) / 32u;
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u, warp = tid >> 5, nw = nt >> 5;
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t j_base = rank * Sc;                           // the block's first slot

    const Layout lay = make_layout(S, K, p.n_q, C, nt);
    const uint32_t NIL = lay.nil, logH = 31u - (uint32_t)__clz((int)lay.heads);
    uint2*    s_node = reinterpret_cast<uint2*>(smem);
    uint32_t* s_head = reinterpret_cast<uint32_t*>(smem + lay.head);
    int8_t*   s_life = reinterpret_cast<int8_t*>(smem + lay.life);
    uint8_t*  s_bits = smem + lay.bits;
    uint32_t* s_ndead = reinterpret_cast<uint32_t*>(smem + lay.ndead);
    uint16_t* s_dead = reinterpret_cast<uint16_t*>(smem + lay.dead);
    uint16_t* s_pref = reinterpret_cast<uint16_t*>(smem + lay.pref);
    uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + lay.mask);
    uint32_t* s_rev  = reinterpret_cast<uint32_t*>(smem + lay.rev);
    uint32_t* s_cnt  = reinterpret_cast<uint32_t*>(smem + lay.cnt);
    uint32_t* s_sum  = reinterpret_cast<uint32_t*>(smem + lay.sum);

    const uint32_t bt = blockIdx.x / C;                          // table of this cluster within the launch
    const uint32_t ti = p.first + bt, table = p.table_id[bt], id_limit = p.id_limit[bt];
    int32_t N = p.verified_len[bt];
    int32_t* g_tok = p.tok + (size_t)table * S + j_base;
    int8_t*  g_life = p.life + (size_t)table * S + j_base;
    const int32_t* ids = p.indices + (size_t)ti * p.n_q * K;
    const uint32_t j0 = tid * SPT;                               // first of the thread's slots, counted in the block
    const bool own = j0 < Sc;

    int32_t xs[IPT];
    auto load_ids = [&](uint32_t g, uint32_t w0) {               // positions of the words w0 + warp IPT + k
#pragma unroll
        for (int k = 0; k < IPT; ++k) {
            const uint32_t i = (w0 + warp * IPT + k) * 32u + lane;
            xs[k] = i < K ? __ldcg(ids + (size_t)g * K + i) : -1;
        }
    };
    auto revive = [&](uint32_t j, uint32_t par) -> bool {        // the slot is no longer dead; false: it was not
        const uint32_t owner = j / SPT, bit = 1u << ((owner & 3u) * 8u + j % SPT);
        if (!(atomicAnd(reinterpret_cast<uint32_t*>(s_bits) + owner / 4u, ~bit) & bit)) return false;
        atomicSub(&s_ndead[par + owner / 32u], 1u);
        return true;
    };

    for (uint32_t i = tid; i < lay.heads / 4; i += nt) reinterpret_cast<uint4*>(s_head)[i] = make_uint4(NIL, NIL, NIL, NIL);
    if (tid == 0) { s_node[NIL] = make_uint2(0xFFFFFFFEu, NIL); s_sum[0] = s_sum[1] = 0; }      // an id that nobody looks for
    if (tid < 2u * MAX_CL) s_rev[tid] = 0;
    if (tid < 3u * (2u + MAX_CL)) s_cnt[tid] = 0;
    cluster_arrive();                                            // what the other blocks write to is ready (waited for below)

    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (p.t_range && tid == 0) atomicMin(p.t_range, global_ns());

    // ---- every global load is issued first: the block's cached ids and lifetimes, the first token's ids ----
    int4 t4[NV];
    uint32_t w[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (tid + q * nt < Sc / 4) t4[q] = __ldcg(reinterpret_cast<const int4*>(g_tok) + tid + q * nt);
    life_words<SPT, true>(g_life + j0, own, w);
    load_ids(0, 0);
    if (p.verified_len_dev) N = __ldg(p.verified_len_dev + ti);
    const uint32_t seen = take_flags_down(p, bt, gridDim.x, rank == 0 ? p.n_launch : 0u);      // (a cluster serves one table)
    cluster_wait();                                              // (the index is empty, too)

    // ---- ids to shared memory and into the index; global pre-decay of the lifetimes (Alg. 1 Pass 1) ----
    bool stale_ids = false;                                      // ids that are no longer verified
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (tid + q * nt < Sc / 4) {
            const uint32_t j = 4u * (tid + q * nt);
            const int32_t x[4] = {t4[q].x, t4[q].y, t4[q].z, t4[q].w};
            uint32_t next[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                next[c] = x[c] >= 0 ? atomicExch(&s_head[hash_id(x[c], logH)], j + c) : NIL;
                stale_ids = stale_ids || x[c] >= N;
            }
#pragma unroll
            for (int c = 0; c < 4; c += 2)
                reinterpret_cast<uint4*>(s_node)[(j + c) / 2] = make_uint4((uint32_t)x[c], (j + c) << 16 | next[c],
                                                                           (uint32_t)x[c + 1], (j + c + 1) << 16 | next[c + 1]);
        }
    }
    // the block's dead slots are added up in the s_cnt buffers of all blocks; buffers take turns so that one can be
    // zeroed while the next is in use: `turn` counts their uses, with a cluster barrier behind each
    uint32_t turn = 0;
    auto cnt_of = [&](uint32_t t) { return (t % 3u) * (2u + MAX_CL); };
    auto store_life = [&](uint32_t par) {                        // lifetimes, dead bits, dead slots of warp and block
        uint32_t bits = 0;
#pragma unroll
        for (int q = 0; q < NV; ++q) bits |= signs(w[q]) << (4 * q);
        life_words_store<SPT>(s_life + j0, own, w);
        s_bits[tid] = (uint8_t)bits;
        const uint32_t n = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(bits));
        if (lane == 0) s_ndead[par + warp] = n;
        if (lane < C && n) addc_u32(map_rank(smem_u32(s_cnt + cnt_of(turn) + 2u + rank), lane), n);
        if (tid < 2u + MAX_CL) s_cnt[cnt_of(turn + 1u) + tid] = 0;
        ++turn;
    };
#pragma unroll
    for (int q = 0; q < NV; ++q) w[q] = decay4(w[q], 1);
    store_life(0);
    __syncthreads();

    uint32_t list_off = 0, sum_miss = 0, sum_decay = 0, valid = 0;
    uint32_t dead_of = 0;                                        // lane q < C: dead slots of block q; set after the barrier
    bool fresh = true;                                           // ... from s_cnt, the first time
    int2* list = p.miss_list + (size_t)ti * p.list_stride;

    for (uint32_t g = 0; g < p.n_q; ++g) {
        const bool last = g + 1 == p.n_q;
        const uint32_t par = 32u * (g & 1u);
        const size_t row = ((size_t)ti * p.n_q + g) * K;
        int32_t* O = p.slots + row;
        uint8_t* Hm = p.hit ? p.hit + row : nullptr;
        uint32_t* mask = s_mask + (g & 1u) * C * W;

        // ---- lookups of all positions in the block's own index; hits: lifetime <- L, slot and flag out ----
        for (uint32_t w0 = 0; w0 < W; w0 += nw * IPT) {
            if (w0) load_ids(g, w0);
            uint32_t node[IPT], revived = 0;
            int32_t slot[IPT], was[IPT];
            bool bad = false;
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const bool ok = (uint32_t)xs[k] < id_limit;
                bad = bad || (!ok && xs[k] >= 0);
                xs[k] = ok ? xs[k] : -1;
                valid += ok;
                slot[k] = -1;
                node[k] = NIL;
                if (ok) node[k] = s_head[hash_id(xs[k], logH)];
            }
            if (bad && rank == 0) atomicOr(p.status, ST_BAD_ID);       // not fetched: reported and taken as padding
            uint32_t open = 1;
            for (uint32_t it = 0; open && it <= NIL; ++it) {           // all chains of the warp side by side
                uint2 v[IPT];
#pragma unroll
                for (int k = 0; k < IPT; ++k) v[k] = s_node[node[k]];
                open = 0;
#pragma unroll
                for (int k = 0; k < IPT; ++k) {
                    const bool found = (int32_t)v[k].x == xs[k];
                    slot[k] = found ? (int32_t)(v[k].y >> 16) : slot[k];
                    node[k] = found ? NIL : v[k].y & 0xFFFFu;
                    open |= node[k] ^ NIL;
                }
                open = __any_sync(0xffffffffu, open);
            }
            if (open) atomicOr(p.status, ST_PROBE_EXHAUSTED);
#pragma unroll
            for (int k = 0; k < IPT; ++k) was[k] = slot[k] >= 0 ? s_life[slot[k]] : 0;
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                const uint32_t wi = w0 + warp * IPT + k, i = wi * 32u + lane;
                const bool hit = slot[k] >= 0, pad = xs[k] < 0 && rank == 0;
                const uint32_t votes = __ballot_sync(0xffffffffu, hit || pad);
                if (lane < C && wi < W) stc_u32(map_rank(smem_u32(mask + rank * W + wi), lane), votes);
                if (hit) s_life[slot[k]] = (int8_t)L;
                if ((hit || pad) && i < K) {
                    O[i] = hit ? (int32_t)j_base + slot[k] : -1;
                    if (Hm) Hm[i] = hit;
                }
                const bool back = hit && was[k] < 0 && revive((uint32_t)slot[k], par);
                revived += __popc(__ballot_sync(0xffffffffu, back));
            }
            if (revived && lane < C) addc_u32(map_rank(smem_u32(s_rev + (g & 1u) * MAX_CL + rank), lane), revived);
        }
        if (last && rank == 0) {
            valid = __reduce_add_sync(0xffffffffu, valid);
            if (lane == 0 && valid) atomicAdd(s_sum, valid);
        }
        if (!last) load_ids(g + 1, 0);                                 // arrives while this token's misses are placed
        if (g == 0 && (p.flags || p.early)) start_dependents(seen);
        cluster_sync();

        // ---- the token's misses, and the dead slots of the blocks ----
        uint32_t n_g = 0;
        for (uint32_t w0 = 0; w0 < W; w0 += 32u) {
            const uint32_t wi = w0 + lane;
            uint32_t m = 0xFFFFFFFFu;
            if (wi < W) {
                m = 0;
                for (uint32_t q = 0; q < C; ++q) m |= mask[q * W + wi];
            }
            const uint32_t c = __popc(~m);
            if (warp == 0) {                                           // (the other warps need the sum alone)
                const uint32_t incl = warp_incl_scan(c, lane);
                if (wi < W) s_pref[wi] = (uint16_t)(n_g + incl - c);
                n_g += __shfl_sync(0xffffffffu, incl, 31);
            } else {
                n_g += __reduce_add_sync(0xffffffffu, c);
            }
        }
        if (fresh) dead_of = lane < C ? s_cnt[cnt_of(turn - 1u) + 2u + lane] : 0u;
        fresh = false;
        if (lane < C) dead_of -= s_rev[(g & 1u) * MAX_CL + lane];
        uint32_t dtotal = __reduce_add_sync(0xffffffffu, dead_of), d = 0;
        sum_miss += n_g;
        if (rank == 0 && tid == 0 && p.miss_count) p.miss_count[(size_t)ti * p.n_q + g] = (int32_t)n_g;

        // Pass 3, the while-loop of Alg. 1: decay until n_g slots are dead (every block takes the same decisions)
        if (dtotal < n_g) {
            life_words<SPT>(s_life + j0, own, w);
            uint32_t lo = 0, hi = L + 1u;                // lo decays are too few, hi are enough
            while (hi - lo > 1u) {
                uint32_t c[4];                           // candidates in (lo, hi), ascending; small ones first
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
                uint32_t* cnt = s_cnt + cnt_of(turn);
                if (lane < C && n01) addc_u32(map_rank(smem_u32(cnt), lane), n01);           // (S <= 32768: 16 bits are enough)
                if (lane < C && n23) addc_u32(map_rank(smem_u32(cnt + 1), lane), n23);
                if (tid < 2u + MAX_CL) s_cnt[cnt_of(turn + 1u) + tid] = 0;
                ++turn;
                cluster_sync();
                const uint32_t n[4] = {cnt[0] & 0xFFFFu, cnt[0] >> 16, cnt[1] & 0xFFFFu, cnt[1] >> 16};
#pragma unroll
                for (int i = 3; i >= 0; --i) if (n[i] >= n_g) hi = c[i];
#pragma unroll
                for (int i = 0; i < 4; ++i) if (n[i] < n_g) lo = c[i];
            }
            d = hi;
#pragma unroll
            for (int q = 0; q < NV; ++q) w[q] = decay4(w[q], d);
            store_life(par);
            cluster_sync();
            dead_of = lane < C ? s_cnt[cnt_of(turn - 1u) + 2u + lane] : 0u;
            dtotal = __reduce_add_sync(0xffffffffu, dead_of);
            if (dtotal < n_g && rank == 0 && tid == 0) atomicOr(p.status, ST_NO_DEAD_SLOTS);
        }
        const uint32_t n_take = n_g < dtotal ? n_g : dtotal;
        const uint32_t first = __reduce_add_sync(0xffffffffu, lane < rank ? dead_of : 0u);       // dead slots of the blocks before
        {   // what the token takes of every block's dead slots
            const uint32_t before = warp_incl_scan(dead_of, lane) - dead_of;
            const uint32_t taken = before < n_take ? (n_take - before < dead_of ? n_take - before : dead_of) : 0u;
            dead_of -= taken;
        }
        // the block's dead slots that are taken, in increasing order
        const uint32_t t = lane < nw ? s_ndead[par + lane] : 0u;
        const uint32_t dead_before = first + __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u);
        if (dead_before < n_take) {
            uint32_t bits = s_bits[tid], r, unused;
            warp_rank<SPT>(__popc(bits), below, r, unused);
            for (r += dead_before; bits && r < n_take; bits &= bits - 1u, ++r) s_dead[r - first] = (uint16_t)(j0 + __ffs((int)bits) - 1);
            s_bits[tid] = (uint8_t)bits;                 // what is handed out is dead no more
        }
        uint32_t left = __shfl_sync(0xffffffffu, t, (int)warp);        // the warp's dead slots for the next token
        if (dead_before < n_take) left = left > n_take - dead_before ? left - (n_take - dead_before) : 0u;
        if (lane == 0) s_ndead[32u - par + warp] = left;
        __syncthreads();
        if (tid < MAX_CL) s_rev[(g & 1u) * MAX_CL + tid] = 0;          // (read by all; added to again two tokens on)

        // ---- install: the k-th miss in position order takes the k-th dead slot ----
        const uint32_t own_total = __reduce_add_sync(0xffffffffu, t);
        const uint32_t mine = first < n_take ? (n_take - first < own_total ? n_take - first : own_total) : 0u;
        for (uint32_t k = tid; k < mine + (rank == 0 ? n_g - n_take : 0u); k += nt) {
            const uint32_t r = k < mine ? first + k : n_take + (k - mine);
            uint32_t lo = 0, hi = W;                                   // largest lo with s_pref[lo] <= r
            while (hi - lo > 1u) {
                const uint32_t mid = (lo + hi) >> 1;
                if (s_pref[mid] <= r) lo = mid; else hi = mid;
            }
            uint32_t m = 0;
            for (uint32_t q = 0; q < C; ++q) m |= mask[q * W + lo];
            m = ~m;
            for (uint32_t skip = r - s_pref[lo]; skip && m; --skip) m &= m - 1u;
            const uint32_t i = lo * 32u + (uint32_t)__ffs((int)m) - 1u;
            if (m == 0 || i >= K) { atomicOr(p.status, ST_BAD_SLOT); continue; }
            int32_t j = -1;
            if (k < mine) {
                const int32_t x = __ldcg(ids + (size_t)g * K + i);
                const uint32_t jl = s_dead[k];
                j = (int32_t)(j_base + jl);
                s_node[jl].x = (uint32_t)x;
                s_life[jl] = (int8_t)L;
                list[list_off + r] = make_int2(x, j);
                g_tok[jl] = x >= N ? -1 : x;                           // speculative ids are forgotten (end of Alg. 4)
                if (!last) {                                           // a node of its own: the slot's is in the old id's chain
                    const uint32_t n = atomicAdd(&s_sum[1], 1u) + Sc;
                    if (n < NIL) s_node[n] = make_uint2((uint32_t)x, jl << 16 | atomicExch(&s_head[hash_id(x, logH)], n));
                    else atomicOr(p.status, ST_PROBE_EXHAUSTED);
                }
            }
            O[i] = j;
            if (Hm) Hm[i] = 0;
        }
        list_off += n_take;
        sum_decay += d;
        __syncthreads();
        announce_token<true>(p, ti, g, mine);
    }

    // ---- write back: lifetimes; resident ids that are no longer verified become empty (Alg. 4) ----
    life_words<SPT>(s_life + j0, own, w);
    life_words_store<SPT>(g_life + j0, own, w);
    if (stale_ids) {
        for (uint32_t q = 0; q < NV; ++q)
            for (uint32_t j = 4u * (tid + q * nt); j < 4u * (tid + q * nt) + 4u && j < Sc; ++j)
                if ((int32_t)s_node[j].x >= N) g_tok[j] = -1;
    }
    if (rank == 0 && tid == 0) {
        SegDesc sd;
        sd.src_base = p.kv_base[bt];
        sd.src_stride = p.kv_stride[bt];
        sd.dst_base = reinterpret_cast<uint64_t>(p.buffer + (size_t)table * S * p.row_bytes);
        sd.count = list_off;
        sd.pad = 0;
        p.seg[ti] = sd;
        TableStats* st = p.stats + table;
        atomicAdd(&st->steps, 1ull);
        atomicAdd(&st->tokens, (unsigned long long)p.n_q);
        atomicAdd(&st->hits, (unsigned long long)(s_sum[0] - sum_miss));
        atomicAdd(&st->misses, (unsigned long long)sum_miss);
        atomicAdd(&st->rows, (unsigned long long)list_off);
        atomicAdd(&st->extra_decays, (unsigned long long)sum_decay);
    }
    if (p.t_range) {
        __syncthreads();
        if (tid == 0) atomicMax(p.t_range + 1, global_ns());
    }
    // (nothing is written to another block's shared memory behind the last token's barrier: a block may leave)
}

template <int CAP>
const void* kernel_of(uint32_t Sc, uint32_t nt)
{
    switch (Sc / nt) {
        case 8:  return reinterpret_cast<const void*>(avsg_stage_one_cluster_kernel<8, CAP>);
        case 4:  return reinterpret_cast<const void*>(avsg_stage_one_cluster_kernel<4, CAP>);
        default: return reinterpret_cast<const void*>(avsg_stage_one_cluster_kernel<2, CAP>);
    }
}

}  // namespace

// Every block looks up all K ids of a token, so the threads follow from the block's slots and K as for a table of S / C.
size_t stage_one_cluster_smem_bytes(uint32_t S, uint32_t K, uint32_t n_q, uint32_t C)
{
    return make_layout(S, K, n_q, C, stage_one_threads(S / C, K)).total;
}

cudaError_t stage_one_cluster_prepare(size_t max_smem)
{
    for (uint32_t spt : {2u, 4u, 8u})
        for (const void* k : {kernel_of<S1_MAX_TABLES>(spt, 1), kernel_of<S1_BIG_TABLES>(spt, 1)}) {
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

namespace {
void cluster_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, uint32_t n_tables, uint32_t S, uint32_t K, uint32_t n_q,
                    uint32_t C)
{
    cfg.gridDim = dim3(n_tables * C);
    cfg.blockDim = dim3(stage_one_threads(S / C, K));
    cfg.dynamicSmemBytes = stage_one_cluster_smem_bytes(S, K, n_q, C);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

template <int CAP>
cudaError_t launch_cluster_t(const S1ParamsT<CAP>& p, uint32_t n_tables, uint32_t C, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cluster_config(cfg, attr, n_tables, p.S, p.K, p.n_q, C);
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    void* args[] = {const_cast<S1ParamsT<CAP>*>(&p)};
    return cudaLaunchKernelExC(&cfg, kernel_of<CAP>(p.S / C, cfg.blockDim.x), args);
}
}  // namespace

// How many clusters of this shape the device can hold at once (0: the shape cannot be launched at all).
int stage_one_cluster_max_active(uint32_t S, uint32_t K, uint32_t n_q, uint32_t C)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cluster_config(cfg, attr, 1, S, K, n_q, C);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel_of<S1_MAX_TABLES>(S / C, cfg.blockDim.x), &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_stage_one_cluster(const S1Params& p, uint32_t n_tables, uint32_t C, cudaStream_t stream)
{
    return launch_cluster_t(p, n_tables, C, stream);
}

cudaError_t launch_stage_one_cluster(const S1ParamsBig& p, uint32_t n_tables, uint32_t C, cudaStream_t stream)
{
    return launch_cluster_t(p, n_tables, C, stream);
}

}  // namespace avsg
