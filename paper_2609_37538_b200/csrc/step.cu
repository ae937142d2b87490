// Both stages of a call in one kernel: a thread-block cluster per table.
//
// The first block of a cluster runs Stage One (match + reserve: Algorithm 1 with the lifetime operations of Algorithm 3,
// the tokens of an iteration in order as in Algorithm 4, the end-of-step invalidation); the others copy the rows of the
// misses, in one of two ways.
//
// Rows asked for early (clusters of four blocks and more, rows that fit a warp's registers, sets that fit beside one another).
// Which block copies a position's row follows from the position alone: groups of neighbours go round over the copying blocks.
// So a copying block need not be told what to fetch.  It puts the table's cached ids into a set of its own
// (bits by hash), and an id of its positions that is not in there, nor in those of the earlier tokens, is missed for certain,
// whatever the tokens before it take away: its row is asked for at once, and is on its way (2 us, over the host link) while
// Stage One still finds out which slot it goes to.  The slot arrives by st.async in a place that again follows from the
// position, counted by an mbarrier per token.  Misses that the block could not know of (an id that seems to be in a set, or
// that loses its slot to an earlier token of the call) it finds in the list of its misses that comes with the slots.
//
// Rows in the order of the misses.  Stage One deals the misses out, the k-th to block k % copying or in shares of neighbours, and
// sends {id, slot}.  Clusters of two and three blocks share rows with other tables' blocks (see the kernel), which takes rows
// from the end of a table's misses: so their own blocks have to take them from the front.  Rows of 1552 bytes and more: one table
// 15.5 us, with misses listed by position but not asked for early 16.0; 4096 bytes 25.4, 25.9.
#include "avsg_kernels.cuh"
#include "follow_stage_one.cuh"
#include "stage_one_common.cuh"

namespace avsg {
namespace {

constexpr uint32_t STEP_SPIN_LIMIT = 1u << 18;            // tries; the hardware suspends the warp for 4 us in each: 1 s
#ifndef AVSG_STEP_GIVE_UP                                 // (a test builds the library with waits that run out)
#define AVSG_STEP_GIVE_UP STEP_SPIN_LIMIT
#endif

// Rows that blocks of other tables may take (see avsg_step_kernel): from how many misses of a token on, how many of a
// table's rows stay for its own blocks (other blocks' caches of translations do not know the table: with 256 left 64 unequal
// requests take 326 us, with 128 330, without any sharing 324), how many warps of the call take some at most (of 144 rows
// under way the link is full; more only copy the last rows twice).
constexpr uint32_t SHARED_FROM = 512, SHARED_LEFT = 256, SHARED_WARPS = 144, SHARED_CLUSTER = 4;

// Shared memory of a call's blocks, in bytes from the start (every part on a 16-byte boundary), and what else follows from
// the sizes.  Rows that are asked for early: a token's positions are counted by groups of 1 << log_group neighbours: group
// n_q * groups, token after token, belongs to copying block group % copying, whose (group / copying)-th it is; the block counts
// its own positions through.
struct StepLayout {
    uint32_t log_group, groups;          // groups of a token
    uint32_t local;                      // positions that a copying block has room for
    uint32_t by_copying, by_groups;      // n / copying == n * by_copying >> 18 for every group and position; the same for groups
    uint32_t per_lane, per_token;        // words of 32 local positions to a lane; entries of a token in a block's list, at most
    uint32_t log_heads, nil;             // chains of the index; its closing node
    uint32_t heads;                      // chains of a packed index
    uint32_t log_seen, log_asked;        // words of the copying blocks' sets: cached ids; ids of an earlier token, each
    uint32_t node, link, fresh, head, life, bits, tot, ndead, cnt, sum, votes, miss, pos, dead, ids;    // first block
    uint32_t seen, asked, slots, id, mask, rest, list, their_ids;              // copying blocks
    uint32_t total;
};
// Tables above this take a packed index, and 16 slots a thread.  What bounds these is still the chain of passes on one SM, which
// grows little with the slots: of two tokens of K = 2048 the second pass of the index, 0.9 us.  Over a cluster of its own (one
// kernel for each stage) Stage One pays a barrier of the cluster a token instead, and Stage Two a launch and the hand-over through
// memory: 16384 slots, in two kernels / in one, us per call: two tokens of K = 2048, 1, 4, 8, 16, 24 tables 21.4 / 12.7, 32.3 / 20.9, 44.7 /
// 33.6, 72.9 / 62.9, 98.9 / 88.4; four tokens 33.1 / 18.9, 49.8 / 31.0, 72.1 / 53.3, 115.7 / 98.5, 160.5 / 143.3; three of K = 3000, one
// table 33.4 / 20.4; from and to host memory, four tokens, 1, 16 tables 52.5 / 23.9, 142 / 108 (ids and outputs went by copies).  With ids from
// the host the first block keeps these too, where rows are asked for early, and the chains are fewer (K = 2048, four tokens 3632, not 11 824,
// for 22 528 nodes); three tokens of 4096 and five of 2000 are not asked for early then.  Those calls, 1, 8, 33 tables: 47.3, 85.8, 228 / 22.7, 58.9,
// 209; 50.0, 99.8, 297 / 29.3, 64.8, 272; 51.2, 97.0, 269 / 26.4, 69.9, 247.
constexpr uint32_t WIDE_SLOTS = 8192;
// ask: rows are asked for early.  False if there is no room (without asking early there always is, up to WIDE_SLOTS).
bool step_layout(StepLayout& o, uint32_t S, uint32_t K, uint32_t n_q, uint32_t nt, uint32_t copying, bool host_ids, bool ask)
{
    // At least 32 groups a token, so that seven blocks have about the same to do: 9 tables with K = 256 30.8 us with groups of
    // 32 positions, 27.5 with rows handed out in turn.  Larger ones are loaded in longer pieces.  Misses in a run of positions go
    // to few blocks, which does not take back what asking early gives: K = 2048, two tokens, 16, 64, 256 neighbours missed of
    // each, dealt out in turn / by groups: one table 9.9 / 9.6, 10.9 / 10.5, 15.9 / 14.2 us; eight 11.8 / 10.3, 22.1 / 20.3, 64.2 /
    // 61.8; 32 22.4 / 21.0, 63.3 / 63.1, 228.0 / 227.1.
    o.log_group = 5u;
    while (o.log_group && K >> o.log_group < 32u) --o.log_group;
    o.groups = (K + (1u << o.log_group) - 1u) >> o.log_group;
    o.local = ask ? (((n_q * o.groups + copying - 1u) / copying << o.log_group) + 31u) & ~31u : 0u;
    o.by_copying = (1u << 18) / copying + 1u;
    o.by_groups = (1u << 18) / o.groups + 1u;
    o.per_lane = (o.local / 32u + 31u) / 32u;
    o.per_token = ask ? (o.groups + copying - 1u) / copying << o.log_group : 1u + (K + copying - 1u) / copying;
    o.nil = S + (n_q - 1u) * K;
    o.log_heads = 1u;
    while ((1u << o.log_heads) < 2u * S) ++o.log_heads;
    o.heads = 1u << o.log_heads;
    o.log_seen = o.log_heads;                              // 64 bits an id
    o.log_asked = 2u;
    while ((1u << o.log_asked) < 2u * K) ++o.log_asked;
    const bool packed = S > WIDE_SLOTS;
    const uint32_t least_seen = o.log_seen - 2u;           // 16 bits an id
    const uint32_t ids = ask && host_ids ? align16(n_q * K * 4u) : 0u, room = (228u << 10) / (1024u / nt) - 2560u;
    for (;;) {
        uint32_t a = 0;
        o.node = a;    a += align16((o.nil + 1u) * (packed ? 4u : 8u));            // nodes of the index; packed: their ids
        o.link = a;    a += packed ? align16((o.nil + 1u) * 2u) : 0u;
        o.fresh = a;   a += packed ? align16((n_q - 1u) * K * 2u) : 0u;
        o.head = a;    a += 4u * o.heads;
        o.life = a;    a += align16(S);                    // lifetime per slot, one signed byte
        o.bits = a;    a += align16(packed ? 2u * nt : nt);                        // one bit per slot, set where it is dead (lifetime < 0)
        o.tot = a;     a += 2u * 32u * 4u;                 // warps' miss totals, by parity
        o.ndead = a;   a += 2u * 32u * 4u;                 // warps' dead slots, by parity
        o.cnt = a;     a += 2u * 2u * 32u * 4u;            // warps' counts of the decay search, by parity
        o.sum = a;     a += 16u;                           // valid ids of the call
        o.votes = a;   a += ask ? align16((K + 31u) / 32u * 4u) : 0u;      // the token's misses, a bit per position
        o.miss = a;    a += align16(K * 4u);               // misses in position order: ids,
        o.pos = a;     a += align16(K * 2u);               //   positions
        o.dead = a;    a += align16(K * 2u);               // dead slots in slot order
        o.ids = a;     a += ids;                           // received: the ids of a call with host buffers
        const uint32_t first = a;
        a = 0;
        o.seen = a;    a += ask ? 4u << o.log_seen : 0u;
        o.asked = a;   a += ask ? (n_q - 1u) * 4u << o.log_asked : 0u;
        o.slots = a;   a += o.local * 4u;                  // received: what has become of a position
        o.id = a;      a += o.local * 4u;                  // its id
        o.mask = a;    a += align16(o.local / 32u * 4u);   // positions whose rows are asked for early
        o.rest = a;    a += align16(o.local / 32u * 4u);   //   but not by the warp that has found them
        o.list = a;    a += align16(n_q * o.per_token * 8u);   // received: a token's misses in the block's positions {place, slot}; or
                                                           //   a head {rows, first shared} and the rows that it copies {id, slot}
        o.their_ids = a; a += ids;                         // received: the ids of a call with host buffers
        o.total = first > a ? first : a;
        if (o.total <= room) return true;
        if (packed) {
            // Both parts give way by themselves: the chains get what is left, down to one for eight slots, the sets half the bits each.
            if (first > room) {
                if (first - room > 4u * o.heads || o.heads - (first - room) / 4u < S / 8u + 4u) return false;
                o.heads = (o.heads - (first - room) / 4u - 1u) & ~3u;
            } else if (o.log_seen > least_seen) {
                --o.log_seen;
            } else if (o.log_asked > 2u && (2u << o.log_asked) > K) {
                --o.log_asked;
            } else {
                return false;
            }
            continue;
        }
        if (ask && a > room) return false;
        if ((1u << o.log_heads) <= S) return !ask;
        --o.log_heads;                                     // longer chains where the rest needs the room
        o.heads /= 2u;
    }
}
constexpr uint32_t NO_ITEM = 0xFFFFFFFFu;
constexpr uint32_t NOT_MISSED = 0xFFFFFFFFu, NO_SLOT = 0xFFFFu;        // of a position; else its slot
static_assert((NOT_MISSED & 0xFFFFu) == NO_SLOT, "a position that is not missed has no slot to store to");

__device__ __forceinline__ bool wait_for(uint32_t mbar, uint32_t limit)
{
    uint32_t spin = 0;
    while (spin < limit && !mbar_done(mbar)) ++spin;
    return __all_sync(0xffffffffu, spin < limit);
}

// Programmatic dependent launch: this grid may have been started while the previous kernel of the stream was still running; nothing
// that the device writes is read before that kernel has completed.  Only then may the next grid start under this one: let go at
// the start, two and three grids wait behind one another, and each hears late that its turn has come (one table, K = 2048, one and
// two tokens 7.78, 11.12 us, now 7.45, 10.72; S = K = 2048 / 4, two tokens 7.94, 7.61; S = 256 5.55, 5.26; two tables 13.3, 13.0).
// A call with ids in host memory lets it go at the start: what that grid does before its wait is to fetch its ids, a round trip of
// the link (K = 2048, two tokens, one, two, three tables 15.4, 18.1, 21.4 us let go behind the wait, 14.5, 17.3, 20.7 at the start).
// The next grid comes when all blocks have let it go, so behind the wait only the copying blocks say so, and the first block of a
// cluster at its start: behind its wait the question costs calls too that let nobody start (host ids, S = 512, K = 65, three tokens, 7, 13
// tables 16.8, 20.1 us with it, 16.3, 19.4 without; S = 2048, K = 229, four tokens 24.6, 35.4 and 24.3, 34.7).  Nor does a branch stand
// where ids on their way from the host are in registers, which it waits for (S = 1024, K = 1000, 5, 13 tables 23.7, 44.2 us with one,
// 22.3, 40.4 without).
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// What the copying blocks are told.  Where they ask for rows early: `token`, that block `to` has n misses in its positions; `miss`,
// to the block that position i belongs to, the slot, where the position's place is and in the next entry of its list.  Where
// they don't, the rows to copy, in the order of the misses: in turn, or (share) `share` neighbours to a block; `head`, how many of n
// they are, and the first one's number among those that are shared (-1: none are); `row`, the k-th.
struct Tell {
    const StepLayout& lay;
    uint32_t copying, smem, mbar, sent;                  // of the first block's own: the same places as in the others

    __device__ __forceinline__ void token(uint32_t g, uint32_t to, uint32_t n) const
    {
        const uint32_t bar = map_rank(mbar + 8u * g, to + 1u);
        send_async(map_rank(sent + 4u * g, to + 1u), n, bar);
        arrive_expect(bar, 12u * n + 4u);
    }
    // own: the misses of the token that the blocks have been told of
    __device__ __forceinline__ void miss(uint32_t g, uint32_t i, uint32_t j, uint32_t* own) const
    {
        const uint32_t group = g * lay.groups + (i >> lay.log_group), at = group * lay.by_copying >> 18, to = group - at * copying;
        const uint32_t n = (at << lay.log_group) + (i & ((1u << lay.log_group) - 1u)), bar = map_rank(mbar + 8u * g, to + 1u);
        send_async(map_rank(smem + lay.slots + 4u * n, to + 1u), j, bar);
        const uint32_t e = atomicAdd(own + to, 1u);
        send_async(map_rank(smem + lay.list + 8u * (g * lay.per_token + e), to + 1u), (int32_t)n, (int32_t)j, bar);
    }
    __device__ __forceinline__ void head(uint32_t g, uint32_t to, uint32_t n, uint32_t share, int32_t first) const
    {
        const uint32_t rows = share == 0 ? (n + copying - 1u - to) * lay.by_copying >> 18
                              : to * share >= n ? 0u : n - to * share < share ? n - to * share : share;
        const uint32_t bar = map_rank(mbar + 8u * g, to + 1u);
        send_async(map_rank(smem + lay.list + 8u * g * lay.per_token, to + 1u), (int32_t)rows, first, bar);
        arrive_expect(bar, 8u * (rows + 1u));
    }
    __device__ __forceinline__ void row(uint32_t g, uint32_t k, uint32_t share, int32_t x, int32_t j) const
    {
        const uint32_t q = share ? k / share : k * lay.by_copying >> 18, r = k - q * (share ? share : copying);
        const uint32_t to = share ? q : r, at = share ? r : q;
        send_async(map_rank(smem + lay.list + 8u * (g * lay.per_token + 1u + at), to + 1u), x, j, map_rank(mbar + 8u * g, to + 1u));
    }
};

// A call with lifetimes above L on entry: the copying blocks hear of all tokens when the last one is placed, and only of rows that
// their slots still wait for.  list: {id, slot | position << 13 | token << 26}.  (Inline: a function call in the kernel brings every
// call's row loads late; 8 new requests 265 us and not 257.)
template <bool ASK>
__device__ __forceinline__ void tell_at_last(const Tell tell, uint32_t n_q, uint32_t K, int2* list, uint32_t count, const uint2* s_node, uint32_t* s_own)
{
    constexpr uint32_t MASK = (1u << LIST_SLOT_BITS) - 1u;
    static_assert(STEP_MAX_TOKENS <= 1u << (32u - 2u * LIST_SLOT_BITS), "a token does not fit an entry");
    drop_lost_rows(list, count, s_node);
    for (uint32_t g = 0; g < n_q; ++g) {
        if constexpr (ASK) {
            if (threadIdx.x < STEP_FEW_CLUSTER) s_own[threadIdx.x] = 0;
            __syncthreads();
            for (uint32_t e = threadIdx.x; e < count; e += blockDim.x) {
                const int2 v = list[e];
                const uint32_t what = (uint32_t)v.y;
                if (v.x >= 0 && what >> (2u * LIST_SLOT_BITS) == g) tell.miss(g, what >> LIST_SLOT_BITS & MASK, what & MASK, s_own);
            }
            __syncthreads();
            if (threadIdx.x < tell.copying) tell.token(g, threadIdx.x, s_own[threadIdx.x]);
            __syncthreads();
        } else {                                         // (K entries at a time, whatever token they are of)
            const uint32_t from = g * K, n = count <= from ? 0u : count - from < K ? count - from : K;
            if (g == 0) __syncthreads();                 // (lost rows are marked)
            if (threadIdx.x < tell.copying) tell.head(g, threadIdx.x, n, 0u, -1);
            for (uint32_t k = threadIdx.x; k < n; k += blockDim.x) tell.row(g, k, 0u, list[from + k].x, (int32_t)((uint32_t)list[from + k].y & MASK));
        }
    }
}

// The first block of a cluster: Stage One.  SPT slots per thread (a power of two): S <= SPT * blockDim.x.  IPT: the most
// ids a thread has of a token (K <= S, so SPT is always enough).  a_mbar: the copying blocks' mbarriers, one per token.
// The passes are those of avsg_stage_one_kernel, which says what they are and why.  ASK: rows are asked for early.  SHARE: rows of a
// table with very many misses may be copied by other tables' blocks.  ARRIVING: the output of that name is written as well: a hit
// whose node is not its slot's own is on a slot that an earlier token of the call has reserved, which its node says (an instance of
// its own: in a pass at the end, or as a question in every call, it costs all others more than it gives these).
template <int SPT, int IPT, bool ASK, bool SHARE, bool ARRIVING, int CAP>
__device__ __forceinline__ void place_tokens(const S1ParamsT<CAP>& p, const StepLayout& lay, const uint32_t ti, const uint32_t copying,
                                             unsigned char* smem, const uint32_t a_mbar, const uint32_t a_sent, uint32_t* s_own)
{
    constexpr int NV = (SPT + 3) / 4;                    // 4-slot vectors of ids / words of lifetimes per thread
    constexpr bool PACKED = SPT > 8;                     // (such tables are a context's: no lifetimes above L)
    constexpr uint32_t BITS = PACKED ? 16u : 8u;         // a thread's bits
    constexpr uint32_t FRESH = 1u << 15, MARK = ARRIVING ? FRESH : 0u;           // above every slot: at those that this call reserves
    const uint32_t S = p.S, K = p.K, L = p.L, NIL = lay.nil;
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u, warp = tid >> 5, nw = nt >> 5;
    const uint32_t below = (1u << lane) - 1u;            // the lanes before this one

    uint2*    s_node = reinterpret_cast<uint2*>(smem + lay.node);
    uint32_t* s_head = reinterpret_cast<uint32_t*>(smem + lay.head);
    int8_t*   s_life = reinterpret_cast<int8_t*>(smem + lay.life);
    auto*     s_bits = reinterpret_cast<typename SlotBits<SPT>::type*>(smem + lay.bits);     // a thread's slots: set where dead
    const PackedIndex ix = {reinterpret_cast<int32_t*>(smem + lay.node), reinterpret_cast<uint16_t*>(smem + lay.link),
                            reinterpret_cast<uint16_t*>(smem + lay.fresh), s_head, lay.heads, NIL, S};
    uint32_t* s_tot  = reinterpret_cast<uint32_t*>(smem + lay.tot);
    uint32_t* s_ndead = reinterpret_cast<uint32_t*>(smem + lay.ndead);
    uint32_t* s_cnt  = reinterpret_cast<uint32_t*>(smem + lay.cnt);
    uint32_t* s_sum  = reinterpret_cast<uint32_t*>(smem + lay.sum);
    uint32_t* s_votes = reinterpret_cast<uint32_t*>(smem + lay.votes);
    int32_t*  s_miss = reinterpret_cast<int32_t*>(smem + lay.miss);
    uint16_t* s_pos  = reinterpret_cast<uint16_t*>(smem + lay.pos);
    uint16_t* s_dead = reinterpret_cast<uint16_t*>(smem + lay.dead);
    const int32_t* s_ids = reinterpret_cast<const int32_t*>(smem + lay.ids);

    // slot j is no longer dead (the count follows the bit, so that an id that comes twice is counted once)
    auto revive = [&](uint32_t j, uint32_t par) {
        const uint32_t owner = j / SPT, in_word = 32u / BITS, bit = 1u << (owner % in_word * BITS + j % SPT);
        if (atomicAnd(reinterpret_cast<uint32_t*>(s_bits) + owner / in_word, ~bit) & bit)
            atomicSub(&s_ndead[par + owner / 32u], 1u);
    };
    const uint32_t ipt = (K + nt - 1) / nt;              // ids per thread
    const uint32_t i0 = warp * ipt * 32u + lane;         // position of the thread's k-th id: i0 + 32 k, below i1
    const uint32_t i1 = (warp + 1u) * ipt * 32u < K ? (warp + 1u) * ipt * 32u : K;
    int32_t xs[IPT];
    auto load_token = [&](uint32_t g) {
        const int32_t* ids = p.indices + ((size_t)ti * p.n_q + g) * K;
#pragma unroll
        for (int k = 0; k < IPT; ++k)
            xs[k] = i0 + 32u * k >= i1 ? -1 : !p.host_ids ? __ldcg(ids + i0 + 32u * k)
                    : ASK ? s_ids[g * K + i0 + 32u * k] : __ldcv(ids + i0 + 32u * k);
    };
    // the clearing comes before the wait: under the previous kernel's tail
    const uint32_t table = p.table_id[ti], id_limit = p.id_limit[ti];
    int32_t N = p.verified_len[ti];
    for (uint32_t i = tid; i < (PACKED ? lay.heads : 1u << lay.log_heads) / 4; i += nt) reinterpret_cast<uint4*>(s_head)[i] = make_uint4(NIL, NIL, NIL, NIL);
    if constexpr (PACKED) {
        if (tid == 0) { ix.id[NIL] = -2; ix.link[NIL] = (uint16_t)NIL; }
    } else {
        if (tid == 0) s_node[NIL] = make_uint2(0xFFFFFFFEu, NIL);      // an id that nobody looks for
    }
    if (tid == 0) s_sum[0] = 0;
    if (ASK && tid < 2u * STEP_FEW_CLUSTER) s_own[tid] = 0;
    // Ids in host memory are there when the call is made, and nothing on the device writes them: a call that queues behind another
    // fetches its first ones while that one's rows travel (32 tables: 5 us of link time and a round trip).
    if (!ASK && p.host_ids) load_token(0);

    wait_for_previous();

    const uint32_t j0 = tid * SPT;                       // first of the thread's slots
    const bool own = j0 < S;
    int32_t* g_tok = p.tok + (size_t)table * S;
    int8_t*  g_life = p.life + (size_t)table * S;
    int4 t4[NV];
    uint32_t w[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (tid + q * nt < S / 4) t4[q] = __ldcg(reinterpret_cast<const int4*>(g_tok) + tid + q * nt);
    life_words<SPT, true>(g_life + j0, own, w);
    if (!p.host_ids) load_token(0);
    if (p.verified_len_dev) N = __ldg(p.verified_len_dev + ti);
    cluster_wait();                                      // (the copying blocks' mbarriers are ready)
    __syncthreads();                                     // the index is empty

    // ---- ids to shared memory and into the index; global pre-decay of the lifetimes (Alg. 1 Pass 1) ----
    bool stale_ids = false;                              // ids that are no longer verified (the caller took tokens back)
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (tid + q * nt < S / 4) stale_ids = stale_ids || t4[q].x >= N || t4[q].y >= N || t4[q].z >= N || t4[q].w >= N;
    if constexpr (PACKED) index_slots(t4, ix);
    else index_slots(t4, s_node, s_head, S, lay.log_heads, NIL);
    uint32_t high = 0;                                   // lifetimes above L (only a caller's own state can have them)
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        if (own) high |= __vcmpgts4(w[q], L * 0x01010101u) & (SPT == 2 ? 0xFFFFu : 0xFFFFFFFFu);
        w[q] = decay4(w[q], 1);
    }
    store_lifetimes<SPT>(s_life, s_bits, s_ndead, own, w);
    if (ASK && p.host_ids) {
        cluster_sync();                                  // (the copying blocks have sent the ids)
        load_token(0);
    }
    const bool unusual = __syncthreads_or(high != 0) && !PACKED;

    uint32_t list_off = 0, sum_miss = 0, sum_decay = 0, valid = 0;
    uint32_t shared = 0;                                 // SHARE: rows that other blocks may take (bit 31: there will be some)
    int2* list = p.miss_list + (size_t)ti * p.list_stride;
    const Tell tell = {lay, copying, smem_u32(smem), a_mbar, a_sent};

    for (uint32_t g = 0; g < p.n_q; ++g) {
        const bool last = g + 1 == p.n_q;
        const uint32_t par = 32u * (g & 1u);
        const size_t row = ((size_t)ti * p.n_q + g) * K;
        int32_t* O = p.slots + row;
        uint8_t* Hm = p.hit ? p.hit + row : nullptr;
        uint8_t* A = ARRIVING ? p.arriving + row : nullptr;

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
        if (bad) atomicOr(p.status, ST_BAD_ID);                        // not fetched: reported and taken as padding
        if constexpr (PACKED) find_slots(xs, ix, p.status, slot);
        else find_slots(xs, s_node, s_head, lay.log_heads, NIL, p.status, slot);
        uint32_t fresh = 0;                              // hits on slots that this call has reserved
        if constexpr (ARRIVING) {
#pragma unroll
            for (int k = 0; k < IPT; ++k)
                if (slot[k] >= (int32_t)FRESH) { slot[k] -= (int32_t)FRESH; fresh |= 1u << k; }
        }
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
            rank[k] = wmiss + __popc(votes & below);                   // within the warp, in position order
            wmiss += __popc(votes);
            if (ASK && lane == 0 && i0 + 32u * k < i1) s_votes[warp * ipt + k] = votes;
            missing |= miss ? 1u << k : 0u;
            if (slot[k] >= 0) s_life[slot[k]] = (int8_t)L;
            if (store) O[i0 + 32u * k] = slot[k];
            if (store && Hm) Hm[i0 + 32u * k] = slot[k] >= 0;
            if (ARRIVING && store) A[i0 + 32u * k] = fresh >> k & 1u;
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
        __syncthreads();

        // ---- CollectDead and the misses, each in order; the prefix over the warps: lane l looks at warp l ----
        uint32_t t = lane < nw ? s_ndead[par + lane] | s_tot[par + lane] << 16 : 0u;
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u);
        const uint32_t all = __reduce_add_sync(0xffffffffu, t);
        const uint32_t n_g = all >> 16;
        uint32_t dtotal = all & 0xFFFFu, dead_before = before & 0xFFFFu, d = 0;
        sum_miss += n_g;
        if (tid == 0 && p.miss_count) p.miss_count[(size_t)ti * p.n_q + g] = (int32_t)n_g;
        const bool share_it = SHARE && n_g > SHARED_FROM && !unusual;
        if (share_it && !shared) {
            shared = SHARED_COMING;
            if (tid == 0) {                              // (in place before the table's own blocks hear of the rows)
                p.shared[ti].taken = p.shared[ti].begun = 0;
                __threadfence();
                *reinterpret_cast<volatile uint32_t*>(&p.shared[ti].rows) = SHARED_COMING;
                __threadfence();
            }
        }
        if (missing) {
#pragma unroll
            for (int k = 0; k < IPT; ++k) {
                if (missing & (1u << k)) {
                    s_miss[(before >> 16) + rank[k]] = xs[k];
                    s_pos[(before >> 16) + rank[k]] = (uint16_t)(i0 + 32u * k);
                }
            }
        }
        if (!last) load_token(g + 1);                                      // arrives while this token's misses are placed
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
        if (ASK && tid < STEP_FEW_CLUSTER) s_own[(~g & 1u) * STEP_FEW_CLUSTER + tid] = 0;         // for the next token
        const uint32_t n_take = n_g < dtotal ? n_g : dtotal;
        if (dead_before < n_take) {                      // some of the first n_g dead slots are this warp's
            uint32_t bits = s_bits[tid], r, unused;
            warp_rank<SPT>(__popc(bits), below, r, unused);
            for (r += dead_before; bits && r < n_take; bits &= bits - 1u, ++r) s_dead[r] = (uint16_t)(j0 + __ffs((int)bits) - 1);
            s_bits[tid] = (typename SlotBits<SPT>::type)bits;          // what is handed out is dead no more
        }
        uint32_t left = __shfl_sync(0xffffffffu, t & 0xFFFFu, (int)warp);          // the warp's dead slots for the next token
        if (dead_before < n_take) left = left > n_take - dead_before ? left - (n_take - dead_before) : 0u;
        if (lane == 0) s_ndead[32u - par + warp] = left;
        __syncthreads();

        // a copying block's rows, where none are asked for early: in turn where few tables have eight blocks each, and where other
        // blocks may take some (so that what is left is at the end), else a share in position order
        const uint32_t share = CAP == STEP_FEW_TABLES || share_it ? 0u : (n_take + copying - 1u) / copying;
        if constexpr (ASK) {
            // What a copying block gets of this token: counted by a warp for each (the first warps install); in small blocks, which have
            // down to four warps, by four lanes for each (S = 256, K = 64, two tokens: 7.5 us with a warp, 7.0).  Not both in one
            // kernel: small calls feel its length (one table of S = 1024, K = 256: 6.3 us, 6.5 with both).
            const uint32_t group0 = g * lay.groups, in_group = (1u << lay.log_group) - 1u;
            auto count = [&](uint32_t to, uint32_t in, uint32_t lanes) -> uint32_t {
                // (its first group is the first one that is `to` modulo copying)
                uint32_t group = (group0 * lay.by_copying >> 18) * copying + to, n = 0;
                if (group < group0) group += copying;
                for (uint32_t q = group - group0 + in * copying; n_g && q < lay.groups; q += lanes * copying) {
                    const uint32_t i = q << lay.log_group;
                    n += __popc(s_votes[i / 32u] >> i % 32u & ~(~1u << in_group));
                }
                return n;
            };
            if constexpr (SPT > 2) {
                for (uint32_t to = nw - 1u - warp; to < copying && !unusual; to += nw) {
                    const uint32_t n = __reduce_add_sync(0xffffffffu, count(to, lane, 32u));
                    if (lane == 0) tell.token(g, to, n);
                }
            } else if (warp == nw - 1u && !unusual) {
                uint32_t n = lane / 4u < copying ? count(lane / 4u, lane & 3u, 4u) : 0u;
                n += __shfl_xor_sync(0xffffffffu, n, 1);
                n += __shfl_xor_sync(0xffffffffu, n, 2);
                if ((lane & 3u) == 0 && lane / 4u < copying) tell.token(g, lane / 4u, n);
            }
        } else if (tid < copying && !unusual) {
            tell.head(g, tid, n_take, share, share_it ? (int32_t)((shared & ~SHARED_COMING) + tid) : -1);
        }

        // ---- install: the k-th miss in position order takes the k-th dead slot ----
        for (uint32_t k = tid; k < n_g; k += nt) {
            const uint32_t i = s_pos[k];
            const int32_t x = s_miss[k];
            const int32_t j = k < n_take ? s_dead[k] : -1;
            if (unusual) {
                if (k < n_take) list[list_off + k] = make_int2(x, (int32_t)((uint32_t)j | i << LIST_SLOT_BITS | g << (2u * LIST_SLOT_BITS)));
            } else if constexpr (ASK) {
                tell.miss(g, i, (uint32_t)j & 0xFFFFu, s_own + (g & 1u) * STEP_FEW_CLUSTER);
            } else if (k < n_take) {
                tell.row(g, k, share, x, j);
            }
            if (k < n_take) {
                if constexpr (PACKED) ix.id[j] = x;
                else s_node[j].x = (uint32_t)x;
                s_life[j] = (int8_t)L;
                if (share_it) list[(shared & ~SHARED_COMING) + k] = make_int2(x, j);
                g_tok[j] = x >= N ? -1 : x;                            // speculative ids are forgotten (end of Alg. 4)
                if (!last) {
                    const uint32_t n = S + list_off + k;
                    if constexpr (PACKED) {
                        ix.id[n] = x;
                        ix.slot[n - S] = (uint16_t)((uint32_t)j + MARK);
                        ix.link[n] = (uint16_t)atomicExch(ix.chain(x), n);
                    } else {
                        s_node[n] = make_uint2((uint32_t)x, ((uint32_t)j + MARK) << 16 | atomicExch(&s_head[hash_id(x, lay.log_heads)], n));
                    }
                }
            }
            O[i] = j;
            if (Hm) Hm[i] = 0;
            if (ARRIVING) A[i] = j >= 0;
        }
        list_off += n_take;
        if (share_it) shared += n_take;
        sum_decay += d;
        __syncthreads();
        announce_token(p, ti, g, n_take);
    }
    if (unusual) tell_at_last<ASK>(tell, p.n_q, K, list, list_off, s_node, s_own);
    if (SHARE && shared && tid == 0) {
        __threadfence();
        *reinterpret_cast<volatile uint32_t*>(&p.shared[ti].rows) = shared == SHARED_COMING ? 0u : shared ^ (SHARED_COMING | SHARED_OPEN);
    }

    // ---- write back: lifetimes; resident ids that are no longer verified become empty (Alg. 4) ----
    life_words<SPT>(s_life + j0, own, w);
    life_words_store<SPT>(g_life + j0, own, w);
    if (stale_ids) {
        for (uint32_t q = 0; q < NV; ++q)
            for (uint32_t j = 4u * (tid + q * nt); j < 4u * (tid + q * nt) + 4u && j < S; ++j)
                if ((PACKED ? ix.id[j] : (int32_t)s_node[j].x) >= N) g_tok[j] = -1;
    }
    if (tid == 0) {
        TableStats* st = p.stats + table;                // (reductions: nothing waits for the old values)
        atomicAdd(&st->steps, 1ull);
        atomicAdd(&st->tokens, (unsigned long long)p.n_q);
        atomicAdd(&st->hits, (unsigned long long)(s_sum[0] - sum_miss));
        atomicAdd(&st->misses, (unsigned long long)sum_miss);
        atomicAdd(&st->rows, (unsigned long long)list_off);
        atomicAdd(&st->extra_decays, (unsigned long long)sum_decay);
    }
}

// The positions of a copying block (block `rank` of its cluster) in the call's first n groups.
__device__ __forceinline__ uint32_t positions_of(const StepLayout& lay, uint32_t rank, uint32_t n)
{
    return n >= rank ? (((n - rank) * lay.by_copying >> 18) + 1u) << lay.log_group : 0u;
}
// The token and the position in it (K or more: none) of a block's n-th.
struct Place { uint32_t g, i; };
__device__ __forceinline__ Place place(const StepLayout& lay, uint32_t rank, uint32_t copying, uint32_t n)
{
    const uint32_t group = rank - 1u + copying * (n >> lay.log_group), g = group * lay.by_groups >> 18;
    return {g, (group - g * lay.groups << lay.log_group) + (n & ~(~0u << lay.log_group))};
}

// A set of ids: three bits, by hash, of a word, by hash.  An id that is in it is found; of those that are not, 0.1 % are found
// too at 64 bits an id (1.6 % with one bit: a small call then often waits for the row that it has asked for late).
__device__ __forceinline__ uint32_t set_bits(int32_t x)
{
    const uint32_t h = (uint32_t)x * 0x85EBCA6Bu;
    return __funnelshift_l(0u, 1u, h >> 27) | __funnelshift_l(0u, 1u, h >> 22) | __funnelshift_l(0u, 1u, h >> 17);
}
__device__ __forceinline__ void set_add(uint32_t* set, uint32_t log_words, int32_t x)
{
    atomicOr(set + hash_id(x, log_words), set_bits(x));
}
__device__ __forceinline__ bool set_has(const uint32_t* set, uint32_t log_words, int32_t x)
{
    return (~set[hash_id(x, log_words)] & set_bits(x)) == 0;
}

// A row that a copying block owes: the position in the block's own count, the token, the id.
struct Item { uint32_t n, g, x; };

// A copying block finds out which of its positions are missed for certain: their ids are in no slot and in no earlier token
// of the call.  What it does not find so (an id that seems to be in a set; a resident one that loses its slot to an earlier
// token) is news from the first block.  The first of the first token that a warp finds is its own to ask for, and returned; the others
// are left in lay.rest, in position order, token after token (for the other warps behind a barrier).
// What takes the time is instruction issue and bank conflicts for 32 warps.  From the call's start, 32 tables of 8192 slots,
// K = 2048, two tokens, three copying blocks: ids and cached ids are loaded after 2.9 us, the sets are there after 3.9, the first
// rows are asked for after 4.7, where rows that wait for their slots are asked for after 6.5.  Other ways to know: a chained index
// like Stage One's 5.9 us; the block's positions in a chained index, and the cached ids looked up in that, 7.1 to 8.
template <int SPT, int IPT, int CAP>
__device__ __forceinline__ Item match(const S1ParamsT<CAP>& p, const StepLayout& lay, const uint32_t ti, const uint32_t rank,
                                      const uint32_t copying, unsigned char* smem)
{
    constexpr int NV = (SPT + 3) / 4, OWN = 4;           // of its positions a warp takes OWN times 32 at a time
    const uint32_t S = p.S, K = p.K, id_limit = p.id_limit[ti];
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u, warp = tid >> 5, W = nt >> 5;
    uint32_t* s_seen = reinterpret_cast<uint32_t*>(smem + lay.seen);
    uint32_t* s_asked = reinterpret_cast<uint32_t*>(smem + lay.asked);
    int32_t*  s_id   = reinterpret_cast<int32_t*>(smem + lay.id);
    uint32_t* s_mask = reinterpret_cast<uint32_t*>(smem + lay.mask);
    uint32_t* s_rest = reinterpret_cast<uint32_t*>(smem + lay.rest);
    int32_t*  s_ids  = reinterpret_cast<int32_t*>(smem + lay.their_ids);
    const uint32_t mine = positions_of(lay, rank, p.n_q * lay.groups), asked_words = 1u << lay.log_asked;
    const int32_t* g_ids = p.indices + (size_t)ti * p.n_q * K;

    auto id_at = [&](uint32_t i) -> int32_t { return p.host_ids ? s_ids[i] : __ldcg(g_ids + i); };

    for (uint32_t i = tid; i < (lay.slots - lay.seen) / 16u; i += nt) reinterpret_cast<uint4*>(s_seen)[i] = make_uint4(0, 0, 0, 0);
    if (p.host_ids) {
        // Ids in host memory are there when the call is made, and nothing on the device writes them: a call that queues
        // behind another fetches its first ones while that one's rows travel.  The copying blocks share the reading, and
        // send what they have read to all blocks.
        const uint32_t all = p.n_q * K, step = copying * nt;
        int32_t x[OWN];
        for (uint32_t from = (rank - 1u) * nt + tid, first = 1;; from += OWN * step) {
#pragma unroll
            for (int m = 0; m < OWN; ++m) x[m] = from + m * step < all ? __ldcv(g_ids + from + m * step) : -1;
            if (first) {
                wait_for_previous();
                cluster_wait();
                first = 0;
            }
#pragma unroll
            for (int m = 0; m < OWN; ++m) {
                const uint32_t i = from + m * step;
                if (i >= all) break;
                for (uint32_t r = 0; r <= copying; ++r)
                    stc_u32(map_rank(smem_u32(smem) + (r ? lay.their_ids : lay.ids) + 4u * i, r), (uint32_t)x[m]);
            }
            if (from - tid + OWN * step >= all) break;
        }
        cluster_sync();
    } else {
        wait_for_previous();
        if (p.early) let_next_start();
    }

    // ---- every global load is issued first: cached ids, the first token's, the block's own ids ----
    // Nothing orders the reads of cached ids before the first block's stores to them.  An id of this call that is read too early
    // only keeps its rows from being asked for early.  One that is gone already (its slot was reserved, or it is no longer verified)
    // makes a position look missed that an earlier token's lookup or the position's own has found: then a row is read in vain, and
    // dropped, because the position stays NOT_MISSED.  So sets decide what is asked for, and what has been received what is stored.
    int4 t4[NV];
    int32_t xo[OWN], xe[IPT];
    uint32_t xg[OWN];                                    // the tokens of xo[]
    const int4* g_tok = reinterpret_cast<const int4*>(p.tok + (size_t)p.table_id[ti] * S);
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (tid + q * nt < S / 4) t4[q] = __ldcg(g_tok + tid + q * nt);
    auto load_own = [&](uint32_t from) {
#pragma unroll
        for (int m = 0; m < OWN; ++m) {
            const uint32_t word = from + warp + W * m, n = word * 32u + lane;
            if (word * 32u >= mine) break;               // (most blocks have one or two words a warp: what none has costs nothing)
            xo[m] = -1;
            const Place q = place(lay, rank, copying, n);
            xg[m] = q.g;
            if (n < mine && q.i < K) xo[m] = id_at(q.g * K + q.i);
        }
    };
    auto load_earlier = [&](uint32_t g) {
#pragma unroll
        for (int k = 0; k < IPT; ++k)
            if (tid + k * nt < K) xe[k] = id_at(g * K + tid + k * nt);
    };
    if (p.n_q > 1u) load_earlier(0);
    load_own(0);
    if (!p.host_ids) cluster_wait();                     // (under the loads)
    cluster_arrive_relaxed();                            // (what this block sends is sent)
    __syncthreads();                                 // the sets are empty
#pragma unroll
    for (int q = 0; q < NV; ++q)
        if (tid + q * nt < S / 4) {                  // (not those of empty slots: a word that all add to takes 4 us)
            if (t4[q].x >= 0) set_add(s_seen, lay.log_seen, t4[q].x);
            if (t4[q].y >= 0) set_add(s_seen, lay.log_seen, t4[q].y);
            if (t4[q].z >= 0) set_add(s_seen, lay.log_seen, t4[q].z);
            if (t4[q].w >= 0) set_add(s_seen, lay.log_seen, t4[q].w);
        }
    for (uint32_t g = 0; g + 1u < p.n_q; ++g) {
#pragma unroll
        for (int k = 0; k < IPT; ++k)
            if (tid + k * nt < K && xe[k] >= 0) set_add(s_asked + g * asked_words, lay.log_asked, xe[k]);
        if (g + 2u < p.n_q) load_earlier(g + 1u);
    }
    __syncthreads();
    Item item = {NO_ITEM, 0u, 0u};
    const uint32_t first_token = positions_of(lay, rank, lay.groups);
    for (uint32_t from = 0; from * 32u < mine; from += OWN * W) {
        if (from) load_own(from);
#pragma unroll
        for (int m = 0; m < OWN; ++m) {
            const uint32_t word = from + warp + W * m, n = word * 32u + lane;
            if (word * 32u >= mine) break;
            const int32_t x = xo[m];
            bool certain = (uint32_t)x < id_limit && !set_has(s_seen, lay.log_seen, x);
            for (uint32_t e = 0; e < xg[m] && certain; ++e) certain = !set_has(s_asked + e * asked_words, lay.log_asked, x);
            const uint32_t votes = __ballot_sync(0xffffffffu, certain);
            s_id[n] = x;
            uint32_t rest = votes;
            const uint32_t l = __ffs((int)votes) - 1u;
            // (a row of a later token is left: the queue has the tokens in order, and who holds one copies nothing until it is placed)
            if (votes && item.n == NO_ITEM && word * 32u + l < first_token) {
                item = {word * 32u + l, 0u, (uint32_t)__shfl_sync(0xffffffffu, x, (int)l)};
                rest &= rest - 1u;
            }
            if (lane == 0) { s_mask[word] = votes; s_rest[word] = rest; }
        }
    }
    return item;
}

__device__ __forceinline__ SharedRows read_shared(const SharedRows* at)
{
    SharedRows s;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(s.rows), "=r"(s.pad), "=r"(s.taken), "=r"(s.begun) : "l"(at) : "memory");
    return s;
}

// A warp that is through with its own table's rows copies rows that other tables share.
template <int CAP>
__device__ __forceinline__ void take_shared_rows(const S1ParamsT<CAP>& p, const uint32_t ti, const uint32_t group)
{
    const uint32_t lane = threadIdx.x & 31u, cpr = p.row_bytes >> 4;
    // all tables at a time: one after the other they had held up the end of a call with many
    SharedRows now = {0u, 0u, 0u, 0u};
    if (group + lane < p.n_launch && group + lane != ti) now = read_shared(p.shared + group + lane);
    const bool some = (now.rows & SHARED_COMING) ||
                      ((now.rows & SHARED_OPEN) && now.taken + now.begun + SHARED_LEFT < (now.rows & ~SHARED_OPEN));
    for (uint32_t which = __ballot_sync(0xffffffffu, some); which; which &= which - 1u) {
        const uint32_t t = group + __ffs((int)which) - 1u;
        SharedRows s = read_shared(p.shared + t);
        for (uint32_t spin = 0; (s.rows & SHARED_COMING) && spin < OVERLAP_SPIN_LIMIT; ++spin) {     // (that Stage One runs, and waits for nobody)
            __nanosleep(64);
            s = read_shared(p.shared + t);
        }
        __threadfence();
        const uint32_t rows = __shfl_sync(0xffffffffu, s.rows, 0) ^ SHARED_OPEN;
        if (rows >= SHARED_OPEN) continue;                             // closed meanwhile
        const uint64_t src = p.kv_base[t], stride = p.kv_stride[t];
        const uint64_t dst = reinterpret_cast<uint64_t>(p.buffer + (size_t)p.table_id[t] * p.S * p.row_bytes);
        const int2* list = p.miss_list + (size_t)t * p.list_stride;
        for (;;) {
            uint32_t at = 0xFFFFFFFFu;
            if (lane == 0 && s.taken + s.begun + SHARED_LEFT < rows) at = atomicAdd(&p.shared[t].taken, 1u);
            at = __shfl_sync(0xffffffffu, at, 0);
            if (at >= rows) break;
            const int2 e = __ldcg(list + (rows - 1u - at));            // what is taken is copied
            s = read_shared(p.shared + t);                             // (comes with the row)
            if (e.x < 0 || e.y < 0 || (uint32_t)e.y >= p.S) {
                if (lane == 0) atomicOr(p.status, ST_BAD_SLOT);
                continue;
            }
            copy_row(src + (uint64_t)(uint32_t)e.x * stride, dst + (uint64_t)(uint32_t)e.y * p.row_bytes, cpr, lane);
        }
    }
}

// A call in one kernel: a cluster of two to eight blocks per table, in either mode.  What it saves is a launch (1.8 us of host
// time, which bounds the smallest calls), the way from the end of one grid to the start of the next, and the hand-over
// through global memory with its fences.  A copying block keeps 20 KB of rows on the way, a row per warp, so that
// seven can fill the link with one table's rows (2 us round trip x 47 GB/s) and the other sizes with what runs beside it.
// Measured, in two kernels (Stage Two overlapped where that is faster) / in one whose rows are asked for when their slots are
// known, us per call:
//   K = 256, S = 1024, one table 8.4 / 5.8;  K = 2048, S = 8192, two tokens, one table 17.2 / 12.2, from a graph 19.8 / 18.3;
//   the same with 4, 8, 16, 32, 48, 64 tables 26.2 / 22.4, 39.0 / 35.6, 65.9 / 63.6, 119.9 / 116.8, 174.0 / 173.6, 228.3 / 226.8;
//   the same from 11 GB of host memory with 8, 16, 32, 48, 64 tables 51 / 46, 88 / 84, 173 / 155, 242 / 229, 315 / 296.
// Asked for at once, before / now: one table 12.9 / 11.5, 8 tables with K = 1000 and 1152-byte rows 36.9 / 34.9, 32 tables 120.5 /
// 117.6, 16 from 11 GB 85.7 / 83.3, 8 new requests 260.4 / 257.1; 20 tables of S = 2048, K = 512 36.7 / 36.3.
// The line of 11 GB is what the end of a call is for.  Where a table's pages are spread over much host memory, translating
// their addresses limits the rows, and a cluster, which lies in one GPC, finds its table's translations there if the
// table was there in the call before.  So calls of more than a few tables let the next grid start only when their
// blocks exit: its clusters then find the same SMs free, in the same order.  Started early they take whatever is free at
// that time: eight tables 60 us and not 46, 16 113 and not 84 (step_early() says which calls gain by it).
// The warps of a block take its rows from a counter, in position order, so that neighbours in host memory go together.
// (Asked for early, such clusters leave 64 unequal requests at 330 us and not 333, but rows taken by others are then spread over
// all positions: one cold table of 64, the others with hits only, 67 us with 656-byte rows and not 62, 138 with 1552 and not 100.)
// SHARE (two and three blocks).  A cluster alone cannot fill the link with one table's rows where it has few copying blocks (an
// SM gets 20 of them a us, the link carries 72), so a new request among steady ones would be left behind: 64 tables, one of
// them cold, 332 us against 277 in two kernels, whose rows are cut evenly over all SMs (Eq. 6).  So a table that misses more
// than SHARED_FROM ids in a token writes these misses to its list in global memory too, and says so.  Its own blocks copy them
// from the front; a few warps of other tables that are through take single rows from the back, counted in SharedRows::taken,
// until few are left; the own blocks stop where the others have begun.  Both may copy a row in the middle, to the same effect.
// Every row is copied: what the own blocks leave out is counted in `taken`, and what is counted there is copied by who counted it.
// Nobody waits, but for a Stage One that has announced rows and runs.  One cold table of 45, 64: 229, 332 us without, 215, 283
// with it, 211, 277 in two kernels; the others with hits only 70, 124, 50, 57, 46, 46; all steady 169, 239.5, 170, 240.5, 172, 241.
// With four blocks it costs every call more (16 tables 64.7 us, 65.5 with it) than it gives one with a new request (16, 32
// tables, one cold: 115, 172 without, 113, 170 with it, 110, 167 in two kernels).  With all rows of such a table claimed one by
// one, its own blocks' too, the cold calls were quicker still (45 tables 214), but a call where most tables had many misses
// lost 5 to 20 %: the requests for claims and list entries wait behind the rows'.  Several rows of a warp at once bring an SM
// from 20 rows a us to 28 at most.
template <int SPT, int IPT, int CAP, bool ASK, bool SHARE, bool ARRIVING>
__global__ void __launch_bounds__(1024, 1) avsg_step_kernel(const __grid_constant__ S1ParamsT<CAP> p, const __grid_constant__ StepLayout lay)
{
    static_assert(!ASK || !SHARE, "rows that are shared are copied in the order of the misses");
    constexpr bool FEW = CAP == STEP_FEW_TABLES;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_mbar[STEP_MAX_TOKENS], s_meet[ASK || FEW ? 1 : STEP_MAX_TOKENS];
    __shared__ uint32_t s_sent[ASK ? STEP_MAX_TOKENS : 1];             // received: a token's misses in the block's positions
    __shared__ uint32_t s_own[2 * STEP_FEW_CLUSTER];                   // first block: of those, how many it has sent, by parity of the token
    __shared__ uint32_t s_next;                                        // of the rows to be asked for, the first that no warp has taken
    __shared__ volatile uint32_t s_mine;                               // rows that are shared: the first that others have taken
    const uint32_t rank = cluster_rank(), cluster = !ASK && FEW ? STEP_FEW_CLUSTER : cluster_size(), copying = cluster - 1u;
    const uint32_t ti = blockIdx.x / cluster, lane = threadIdx.x & 31u, W = blockDim.x >> 5, warp = threadIdx.x >> 5;
    uint32_t* s_slots = reinterpret_cast<uint32_t*>(smem + lay.slots);
    if (p.early && (p.host_ids || rank == 0)) let_next_start();
    if (SHARE && threadIdx.x == 0) s_mine = 0xFFFFFFFFu;
    if (rank != 0) {
        if (threadIdx.x < p.n_q) {
            mbar_init(smem_u32(s_mbar + threadIdx.x), 1u);
            if (!ASK && !FEW) mbar_init(smem_u32(s_meet + threadIdx.x), W);
        }
        if constexpr (ASK) {
            if (threadIdx.x == 0) s_next = 0;
            for (uint32_t i = threadIdx.x; i < lay.local; i += blockDim.x) s_slots[i] = NOT_MISSED;
            for (uint32_t i = threadIdx.x; i < lay.local / 32u; i += blockDim.x) reinterpret_cast<uint32_t*>(smem + lay.rest)[i] = 0;
        }
    }
    __syncthreads();
    cluster_arrive();
    if (rank == 0) {
        place_tokens<SPT, IPT, ASK, SHARE, ARRIVING>(p, lay, ti, copying, smem, smem_u32(s_mbar), smem_u32(s_sent), s_own);
        __syncwarp();
        // Everything is sent.  Written, too, where other blocks read it; else nobody has to wait until the memory system says so (the
        // blocks of one table's call stood 0.6 us behind their last rows: K = 2048, two tokens 10.35, now 10.19; S = 2048 7.48, 7.33).
        if (SHARE || p.out.n_slots) cluster_arrive();
        else cluster_arrive_relaxed();
        return;
    }
    const uint32_t cpr = p.row_bytes >> 4;
    const uint64_t src = p.kv_base[ti], stride = p.kv_stride[ti];
    const uint64_t dst = reinterpret_cast<uint64_t>(p.buffer + (size_t)p.table_id[ti] * p.S * p.row_bytes);
    bool there = true;                                                 // nothing was waited for in vain
    uint32_t turn = warp;                                              // SHARE: warps in the order in which they are through
    if constexpr (ASK) {
        Row row;
        Item item = match<SPT, IPT>(p, lay, ti, rank, copying, smem);
        const int32_t* s_id = reinterpret_cast<const int32_t*>(smem + lay.id);
        const uint32_t* s_mask = reinterpret_cast<const uint32_t*>(smem + lay.mask);
        const uint32_t* s_rest = reinterpret_cast<const uint32_t*>(smem + lay.rest);
        const int2* s_list = reinterpret_cast<const int2*>(smem + lay.list);
        auto slot_of = [&](uint32_t what) -> uint32_t {                // what a position has received; NO_SLOT: there were not enough
            const uint32_t j = what & 0xFFFFu;
            if (j < p.S) return j;
            if (j != NO_SLOT && lane == 0) atomicOr(p.status, ST_BAD_SLOT);
            return NO_SLOT;
        };
        uint32_t upto = 0;                                             // rows that no warp has found first: those of a few
                                                                       // neighbouring words, a lane, and those before them
        auto next = [&] {                                              // the next of these is the warp's
            uint32_t k = 0;
            if (lane == 0) k = atomicAdd(&s_next, 1u);
            k = __shfl_sync(0xffffffffu, k, 0);
            item.n = NO_ITEM;
            const uint32_t behind = __ballot_sync(0xffffffffu, upto > k);
            if (behind == 0) return;
            const uint32_t l = __ffs((int)behind) - 1u;
            if (l) k -= __shfl_sync(0xffffffffu, upto, (int)l - 1);
            uint32_t a = l * lay.per_lane, m = s_rest[a];
            for (; k >= __popc(m); m = s_rest[++a]) k -= __popc(m);
            item.n = a * 32u + __ffs((int)__ballot_sync(0xffffffffu, (m >> lane & 1u) && __popc(m & ((1u << lane) - 1u)) == k)) - 1u;
            item.g = place(lay, rank, copying, item.n).g;
            item.x = (uint32_t)s_id[item.n];
        };
        uint32_t told = 0;                                             // tokens that the block has heard of
        for (bool first = true;; first = false) {
            // the row is on its way before its slot is known (one place in the code, so that no copy from register to register waits for it)
            load_row(row, src + (uint64_t)item.x * stride, item.n != NO_ITEM ? cpr : 0u, lane);
            if (first) {
                __syncthreads();                                       // every warp has looked at its positions
                for (uint32_t a = lane * lay.per_lane; a < lay.local / 32u && a < (lane + 1u) * lay.per_lane; ++a) upto += __popc(s_rest[a]);
                upto = warp_incl_scan(upto, lane);
                if (item.n == NO_ITEM) {
                    next();
                    if (item.n != NO_ITEM) continue;
                }
            }
            for (; told < p.n_q && (item.n == NO_ITEM || told <= item.g); ++told) {
                there = wait_for(smem_u32(s_mbar + told), AVSG_STEP_GIVE_UP);          // (Stage One's loops are bounded, far below this)
                if (!there) break;
                // the token's misses that are not asked for early, in turn
                for (uint32_t e = W - 1u - warp; e < s_sent[told]; e += W) {
                    const int2 what = s_list[told * lay.per_token + e];
                    const uint32_t n = (uint32_t)what.x;
                    if (s_mask[n / 32u] >> n % 32u & 1u) continue;
                    const uint32_t j = slot_of((uint32_t)what.y);
                    if (j != NO_SLOT) copy_row(src + (uint64_t)(uint32_t)s_id[n] * stride, dst + (uint64_t)j * p.row_bytes, cpr, lane);
                }
            }
            if (!there || item.n == NO_ITEM) break;
            const uint32_t j = slot_of(s_slots[item.n]);
            if (j != NO_SLOT) store_row(row, dst + (uint64_t)j * p.row_bytes, cpr, lane);
            next();
        }
    } else {
        wait_for_previous();
        if (p.early && !p.host_ids) let_next_start();
        cluster_wait();
        cluster_arrive();
        uint32_t from = 0;                                             // the warp that is next
        for (uint32_t g = 0; g < p.n_q; ++g) {
            const int2* got = reinterpret_cast<const int2*>(smem + lay.list) + g * lay.per_token;
            there = wait_for(smem_u32(s_mbar + g), AVSG_STEP_GIVE_UP);
            if (!there) break;
            const uint32_t count = (uint32_t)got[0].x;
            const int32_t at = got[0].y;                               // of the first row among those that are shared; -1
            SharedRows s = {SHARED_COMING, 0u, 0u, 0u};
            for (uint32_t k = warp >= from ? warp - from : warp + W - from; k < count; k += W) {
                if (SHARE && at >= 0) {
                    if (warp == 0) {                                   // for all warps: requests wait behind the rows' where the link is full
                        if (!(s.rows & SHARED_COMING)) s_mine = (s.rows & ~SHARED_OPEN) > s.taken ? (s.rows & ~SHARED_OPEN) - s.taken : 0u;
                        s = read_shared(p.shared + ti);                // (comes with the row)
                        if (lane == 0) atomicAdd(&p.shared[ti].begun, W);
                    }
                    if (at + k * copying >= s_mine) break;             // others have the rest
                }
                const int2 e = got[1u + k];
                if (e.x < 0) continue;                                 // (its slot has gone to another id)
                if (e.y < 0 || (uint32_t)e.y >= p.S) {
                    if (lane == 0) atomicOr(p.status, ST_BAD_SLOT);
                    continue;
                }
                copy_row(src + (uint64_t)(uint32_t)e.x * stride, dst + (uint64_t)e.y * p.row_bytes, cpr, lane);
            }
            if (FEW || count < W || (SHARE && g + 1u == p.n_q)) {
                from = (from + count) % W;
            } else if (g + 1u < p.n_q) {                               // the warps meet
                from = 0;
                if (lane == 0) mbar_arrive(smem_u32(s_meet + g));
                there = wait_for(smem_u32(s_meet + g), AVSG_STEP_GIVE_UP);
                if (!there) break;
            }
        }
        turn = warp >= from ? warp - from : warp + W - from;
    }
    // Warps that take other tables' rows: those that had the fewest of the last token, a few of each block
    uint32_t others = 0;                                               // what 32 of the tables share, one a lane
    const uint32_t group = (ti + turn) % ((p.n_launch + 31u) / 32u) * 32u;
    const bool takes = SHARE && turn * (p.n_launch - 1u) * copying < SHARED_WARPS * ((p.n_launch + 31u) / 32u);
    if (takes && group + lane < p.n_launch) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(others) : "l"(&p.shared[group + lane].rows) : "memory");
    // Stage One does not know who has given up, and nothing may be sent to a block that is gone: every block stays until
    // Stage One is through, and one that gave up until what was sent has arrived.
    cluster_wait();
    if (!there) {
        if (lane == 0) atomicOr(p.status, ST_WAIT_TIMEOUT);
        for (uint32_t g = 0; g < p.n_q && wait_for(smem_u32(s_mbar + g), STEP_SPIN_LIMIT); ++g) {}
    }
    if (p.out.n_slots) put_outputs_of(p.out, ti, p.n_q * p.K, p.n_q, warp * copying + rank - 1u, W * copying, lane);
    if constexpr (SHARE) {
        // Closed for who has not begun yet, and so closed between calls (Stage One is through and writes it no more).
        if (threadIdx.x == 0) atomicAnd(&p.shared[ti].rows, SHARED_OPEN - 1u);
        if (takes && __any_sync(0xffffffffu, (others & (SHARED_COMING | SHARED_OPEN)) != 0)) take_shared_rows(p, ti, group);
    }
}

}  // namespace

// At least 16 warps a block where the table has the slots for it: they copy.
uint32_t step_threads(uint32_t S, uint32_t K)
{
    const uint32_t t = stage_one_threads(S, K), most = S / 2 < 512u ? S / 2 : 512u;
    return t > most ? t : most;
}

namespace {

template <int CAP, bool ASK, bool SHARE = false, bool ARRIVING = false>
const void* step_kernel(uint32_t spt, uint32_t ipt)
{
    switch (spt) {
        case 16: return ipt <= 2 ? reinterpret_cast<const void*>(avsg_step_kernel<16, 2, CAP, ASK, SHARE, ARRIVING>)
                      : ipt <= 4 ? reinterpret_cast<const void*>(avsg_step_kernel<16, 4, CAP, ASK, SHARE, ARRIVING>)
                                 : reinterpret_cast<const void*>(avsg_step_kernel<16, 8, CAP, ASK, SHARE, ARRIVING>);
        case 8:  return ipt <= 2 ? reinterpret_cast<const void*>(avsg_step_kernel<8, 2, CAP, ASK, SHARE, ARRIVING>)
                      : ipt <= 4 ? reinterpret_cast<const void*>(avsg_step_kernel<8, 4, CAP, ASK, SHARE, ARRIVING>)
                                 : reinterpret_cast<const void*>(avsg_step_kernel<8, 8, CAP, ASK, SHARE, ARRIVING>);
        case 4:  return ipt <= 2 ? reinterpret_cast<const void*>(avsg_step_kernel<4, 2, CAP, ASK, SHARE, ARRIVING>)
                                 : reinterpret_cast<const void*>(avsg_step_kernel<4, 4, CAP, ASK, SHARE, ARRIVING>);
        default: return reinterpret_cast<const void*>(avsg_step_kernel<2, 2, CAP, ASK, SHARE, ARRIVING>);
    }
}

void step_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* attr, uint32_t n_tables, uint32_t cluster, uint32_t threads, size_t smem)
{
    cfg.gridDim = dim3(n_tables * cluster);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}
}  // namespace

// Loads this file's kernels and raises their limit of dynamic shared memory to the device's (see stage_one_prepare() on why
// that is not left to their first launch).
cudaError_t step_prepare(size_t max_smem)
{
    for (uint32_t spt : {2u, 4u, 8u, 16u})
        for (uint32_t ipt = 2u; ipt <= spt && ipt <= 8u; ipt *= 2u)    // (K <= S, and STEP_MAX_IDS)
            for (const void* k : {step_kernel<STEP_FEW_TABLES, true>(spt, ipt), step_kernel<STEP_FEW_TABLES, false>(spt, ipt), step_kernel<STEP_MAX_TABLES, true>(spt, ipt),
                                  step_kernel<STEP_MAX_TABLES, false>(spt, ipt), step_kernel<STEP_MAX_TABLES, false, true>(spt, ipt),
                                  step_kernel<STEP_FEW_TABLES, true, false, true>(spt, ipt), step_kernel<STEP_MAX_TABLES, true, false, true>(spt, ipt)}) {
                cudaFuncAttributes fa;
                cudaError_t e = cudaFuncGetAttributes(&fa, k);
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(max_smem - fa.sharedSizeBytes));
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

// Above WIDE_SLOTS: where the index has room (n_q and K decide), and not calls of few tokens with three and two blocks a table, whose
// rows two kernels cut evenly over all SMs: K = 2048, two kernels / one, us: 36, 50, 74 tables, one token 83.9 / 83.0, 109.8 / 112.0, 154.9 /
// 156.7; K = 1024, two tokens, 40, 64 tables 99.9 / 94.9, 149.0 / 147.3, but 64 cold ones 1103 / 1114; K = 2048, three tokens, 40, 50,
// 74 tables 200 / 190, 243 / 238, 350 / 345, 60 cold ones 810 / 810; four tokens, 40, 64 tables 248 / 234, 381 / 371.  (All with device ids.
// With host buffers two kernels also pay for copies and events; where the line would lie for these has not been measured.)
bool step_serves(uint32_t S, uint32_t K, uint32_t n_q, uint32_t cluster, uint32_t row_bytes, bool arriving)
{
    StepLayout lay;
    if (arriving && (cluster < SHARED_CLUSTER || row_bytes > 16u * ROW_CHUNKS || !step_layout(lay, S, K, n_q, step_threads(S, K), cluster - 1u, false, true)))
        return false;
    return S <= WIDE_SLOTS || (S <= STEP_MAX_SLOTS && K <= STEP_MAX_IDS && n_q + cluster >= 5u &&
                               step_layout(lay, S, K, n_q, step_threads(S, K), cluster - 1u, false, false));
}

StepClusters step_clusters(size_t max_smem)
{
    StepClusters s;
    for (uint32_t cl : {2u, 3u, 4u, STEP_FEW_CLUSTER}) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[2];
        int fit = 0;
        step_config(cfg, attr, 1, cl, 1024, max_smem - 2048);      // (the largest; statically it has 1 KB)
        if (cudaOccupancyMaxActiveClusters(&fit, step_kernel<STEP_MAX_TABLES, true>(8, 2), &cfg) != cudaSuccess) { cudaGetLastError(); fit = 0; }
        s.fit[cl] = (uint32_t)fit;
    }
    return s;
}

template <int CAP>
cudaError_t launch_step(const S1ParamsT<CAP>& p, uint32_t cluster, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    const uint32_t nt = step_threads(p.S, p.K);
    const bool share = CAP == STEP_MAX_TABLES && cluster < SHARED_CLUSTER;
    StepLayout lay;
    const bool ask = !share && p.row_bytes <= 16u * ROW_CHUNKS && step_layout(lay, p.S, p.K, p.n_q, nt, cluster - 1u, p.host_ids != 0, true);
    if (!ask) step_layout(lay, p.S, p.K, p.n_q, nt, cluster - 1u, p.host_ids != 0, false);
    step_config(cfg, attr, p.n_launch, cluster, nt, lay.total);
    cfg.stream = stream;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    void* args[] = {const_cast<S1ParamsT<CAP>*>(&p), &lay};
    const uint32_t spt = p.S / nt, ipt = (p.K + nt - 1) / nt;
    const void* kernel = ask && p.arriving ? step_kernel<CAP, true, false, true>(spt, ipt) : ask ? step_kernel<CAP, true>(spt, ipt) : step_kernel<CAP, false>(spt, ipt);
    if constexpr (CAP == STEP_MAX_TABLES)
        if (share) kernel = step_kernel<CAP, false, true>(spt, ipt);
    return cudaLaunchKernelExC(&cfg, kernel, args);
}
template cudaError_t launch_step(const StepParams& p, uint32_t cluster, cudaStream_t stream);
template cudaError_t launch_step(const StepParamsFew& p, uint32_t cluster, cudaStream_t stream);

}  // namespace avsg
