// Internal declarations shared by the kernels and the C-ABI host code.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace avsg {

// Device status word: kernels OR one of these in when a bounded loop runs out
// or an index leaves its range; nothing ever traps.
enum : uint32_t {
    ST_PROBE_EXHAUSTED = 1u << 0,   // hash probe visited every bucket
    ST_NO_DEAD_SLOTS   = 1u << 1,   // fewer reclaimable slots than misses (Eq. 7 violated)
    ST_BAD_SLOT        = 1u << 2,   // slot / position index out of range
    ST_BAD_SEGMENT     = 1u << 3,   // transfer kernel could not resolve a miss
    ST_BAD_ID          = 1u << 4,   // an id beyond the table's host rows or the direct index (treated as padding)
    ST_WAIT_TIMEOUT    = 1u << 5,   // overlapped Stage Two: a bounded wait for Stage One ran out
};

// One segment of the step's miss list = the misses of one table, in token
// order then position order (Alg. 4 appends every token's misses to the step's transfer list).
struct SegDesc {
    uint64_t src_base;    // host KV base of the table (device-visible address)
    uint64_t src_stride;  // bytes between host rows
    uint64_t dst_base;    // device buffer base of the table
    uint32_t count;       // entries in the segment
    uint32_t pad;
};

// Wall-clock span of a grid for avsg_set_timing: every block reports its start and end (globaltimer, ns).
__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Inclusive prefix sum over the lanes of a warp.
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= (uint32_t)o) v += n;
    }
    return v;
}

// Exclusive prefix sum over the block in thread order (the order-preserving compactions of Stage One, the miss
// prefix sums of Stage Two); s_w holds 33 words of shared memory.  Every thread of the block calls it.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* s_w, uint32_t& total)
{
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const uint32_t incl = warp_incl_scan(v, lane);
    if (lane == 31) s_w[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < nwarps ? s_w[lane] : 0u;
        uint32_t wi = warp_incl_scan(w, lane);
        s_w[lane] = wi - w;
        if (lane == 31) s_w[32] = wi;
    }
    __syncthreads();
    total = s_w[32];
    return incl - v + s_w[warp];
}

struct TableStats {
    unsigned long long steps, tokens, hits, misses, rows, extra_decays;
};

constexpr int S1_MAX_TABLES = 128;   // tables per Stage One launch with the small argument block (3.3 KB)
constexpr int S1_BIG_TABLES = 1024;  // ... with the large one (25 KB; kernel arguments may take up to 32 764 bytes)
constexpr int MAX_IPT = 8;           // ids per thread
constexpr int MAX_SPT = 8;           // slots per thread
constexpr int XFER_MAX_SEG = 2048;   // segments per Stage Two launch (prefix sums live in shared memory)

// Calls with host buffers: Stage Two writes the call's outputs from the library's device buffers (256-byte aligned) into
// the caller's mapped host memory, which the GPU's side of the link that the gather leaves free carries.
struct HostOut {
    const int32_t* slots = nullptr;  int32_t* host_slots = nullptr;  uint32_t n_slots = 0;
    const uint8_t* hit = nullptr;    uint8_t* host_hit = nullptr;    uint32_t n_hit = 0;           // none: 0
    const int32_t* count = nullptr;  int32_t* host_count = nullptr;  uint32_t n_count = 0;
};

constexpr int OVERLAP_MAX_TOKENS = 8;

// Calls in one kernel: a thread-block cluster per table, one block for Stage One and the others for Stage Two.
constexpr int STEP_MAX_TABLES = 74, STEP_FEW_TABLES = 8;      // sizes of the argument block
constexpr uint32_t STEP_FEW_CLUSTER = 8;
constexpr uint32_t STEP_EARLY_TABLES = 3;            // see step_early()
constexpr uint64_t STEP_EARLY_BYTES = 2ull << 30;
constexpr uint32_t STEP_MAX_TOKENS = 64;
constexpr uint32_t STEP_MAX_SLOTS = 16384, STEP_MAX_IDS = 8192;      // of a table; of a token, where a table has more than 8192
// What a table that misses far more than its cluster's blocks can have under way shares with the other blocks of the call:
// see avsg_step_kernel.
struct __align__(16) SharedRows {
    uint32_t rows;      // how many there are, with SHARED_OPEN while others may begin to take some; SHARED_COMING until that is known
    uint32_t pad;
    uint32_t taken;     // by others, from the last one backwards
    uint32_t begun;     // by the table's own blocks, about
};
constexpr uint32_t SHARED_COMING = 1u << 31, SHARED_OPEN = 1u << 30;

// The per-call host arrays travel as kernel arguments, CAP tables' worth of them: a call needs no staging copy.
template <int CAP>
struct S1ParamsT {
    int32_t*       tok;          // [num_tables][S]
    int8_t*        life;         // [num_tables][S]
    uint8_t*       buffer;       // [num_tables][S * row_bytes]
    TableStats*    stats;        // [num_tables]
    int2*          miss_list;    // [segments][list_stride]  (x, slot)
    SegDesc*       seg;          // [segments]
    uint32_t*      status;       // mapped host word
    const int32_t* indices;      // [n][n_q][K]
    int32_t*       slots;        // [n][n_q][K]
    uint8_t*       hit;          // [n][n_q][K] or null
    int32_t*       miss_count;   // [n][n_q] or null
    uint8_t*       arriving = nullptr;          // a call in one kernel: [n][n_q][K] or null
    uint32_t S, logH, row_bytes, K, n_q, L;
    uint32_t first;              // index within the call of this launch's first table
    uint32_t n_launch;           // tables of this launch (the grid may have fewer blocks: a block then serves several)
    uint32_t list_stride;        // entries per segment of miss_list
    uint32_t* qword;             // paper-literal mode: packed metadata words [num_tables][S], else null
    uint32_t probe_retries, hash_a1, hash_a2;   // paper-literal mode: R, a1, a2
    unsigned long long* t_range = nullptr;      // timing on: [0] earliest block start, [1] latest block end (ns)
    // overlapped Stage Two (null otherwise): flags[ti * n_q + g], for token g of the ti-th table of the call: every block
    // of the table adds ANNOUNCED + the misses it has placed; zero until then (see take_flags_down())
    uint32_t* flags = nullptr;
    // calls with host buffers in that mode (null otherwise): the table that places the call's last token last
    // writes the call's sequence number to *done_seq, which the output download waits for
    unsigned long long* done_seq = nullptr;
    uint32_t*           done_ctr = nullptr;     // arrivals after the call's last token; wraps to zero at `expect`
    unsigned long long  host_seq = 0;
    uint32_t            expect = 0;             // Stage One blocks that place tables of the call
    HostOut             out;                    // a call in one kernel: what its Stage Two writes to the host
    SharedRows*         shared = nullptr;       // a call in one kernel: [STEP_MAX_TABLES], neither coming nor open between calls
    uint32_t            early = 1;              // the next grid may start under this one (with flags it has to)
    uint32_t            host_ids = 0;           // indices is mapped host memory that holds the ids when the call is made
    const int32_t* verified_len_dev = nullptr;  // [n] of the call: read instead of verified_len[] when set
    uint32_t table_id[CAP];
    int32_t  verified_len[CAP];
    uint32_t id_limit[CAP];      // ids >= this are not looked up or fetched (host rows of the table; direct index size)
    uint64_t kv_base[CAP];
    uint64_t kv_stride[CAP];
};
using S1Params = S1ParamsT<S1_MAX_TABLES>;
using S1ParamsBig = S1ParamsT<S1_BIG_TABLES>;
static_assert(sizeof(S1ParamsBig) <= 32764, "kernel argument block too large");

struct XferParams {
    const SegDesc* seg;
    const int2*    miss_list;
    uint32_t*      status;
    uint32_t n_seg, list_stride, row_bytes, request_level, S;
    HostOut out;
    // timing on: [0] earliest block start, [1] latest block end, [2] earliest start of a block's copy loop,
    // [3] earliest arrival of a block's first row, [4] earliest end of a block that copied something (ns)
    unsigned long long* t_range = nullptr;
};

constexpr uint32_t S1_ROUND_BLOCKS = 32;             // Stage One blocks of a call that is served in rounds
constexpr int OVERLAP_MAX_TABLES = S1_BIG_TABLES;   // one Stage One launch
constexpr uint32_t ANNOUNCED = 1u << 16;            // in a hand-over flag: one block's announcement (a count needs 16 bits)
constexpr uint32_t OVERLAP_SPIN_LIMIT = 1u << 18;   // polls before the wait gives up; a poll is an L2 round trip plus a 64 ns sleep, ~0.8 us measured: ~0.2 s

// Stage Two that is resident while Stage One runs and starts on misses as they are announced (see the kernel).
// The tables' bases come as kernel arguments, CAP tables' worth.
template <int CAP>
struct XferOverlapParamsT {
    const int2*    miss_list;
    uint32_t*      status;
    const uint32_t* flags;       // [n][n_q] written by Stage One (see S1ParamsT)
    uint32_t announcers;         // Stage One blocks per table
    uint8_t*       buffer;       // [num_tables][S * row_bytes]
    uint32_t n, n_q, list_stride, row_bytes, S;
    uint32_t round_size;         // tables per round (n: one round)
    HostOut out;
    unsigned long long* t_range = nullptr;
    uint32_t table_id[CAP];
    uint64_t kv_base[CAP];
    uint64_t kv_stride[CAP];
};
using XferOverlapParams = XferOverlapParamsT<S1_MAX_TABLES>;
using XferOverlapParamsBig = XferOverlapParamsT<S1_BIG_TABLES>;

struct PosParams {               // comparator S2: equal top-K position partition
    const SegDesc* seg;          // per table: host base, stride, buffer base
    const int32_t* indices;      // [n][n_q*K]
    const int32_t* slots;        // [n][n_q*K] (written by Stage One)
    const uint8_t* hit;          // [n][n_q*K] (written by Stage One)
    uint32_t*      status;
    uint32_t n, per_table, row_bytes, S;     // per_table = n_q * K positions
};

struct AllKParams {
    const int32_t* indices;      // [n][n_q*K]
    int32_t*       slots;
    uint8_t*       hit;
    int32_t*       miss_count;
    int2*          miss_list;
    SegDesc*       seg;
    TableStats*    stats;
    uint8_t*       buffer;
    uint32_t*      status;
    uint32_t S, row_bytes, K, n_q, first, list_stride;
    uint32_t table_id[S1_MAX_TABLES];
    uint32_t id_limit[S1_MAX_TABLES];
    uint64_t kv_base[S1_MAX_TABLES];
    uint64_t kv_stride[S1_MAX_TABLES];
};

struct ResetParams {             // stream-ordered reset of some tables: empty, dead, counters and rows zeroed
    int32_t* tok; int8_t* life; uint8_t* buffer; TableStats* stats;
    uint32_t* qword;             // paper-literal mode, else null
    uint32_t S, row_bytes;
    uint32_t table_id[S1_MAX_TABLES];
};
constexpr uint32_t RESET_THREADS = 256;
cudaError_t launch_reset_tables(const ResetParams& p, uint32_t n_tables, uint32_t sm_count, cudaStream_t stream);

size_t stage_one_smem_bytes(uint32_t S, uint32_t K, uint32_t n_q);
size_t stage_one_paper_smem_bytes(uint32_t S, uint32_t K, uint32_t L);
uint32_t stage_one_threads(uint32_t S, uint32_t K);
cudaError_t stage_one_prepare(size_t max_smem);
// both stages of a call of up to STEP_MAX_TABLES tables in one kernel
using StepParams = S1ParamsT<STEP_MAX_TABLES>;
using StepParamsFew = S1ParamsT<STEP_FEW_TABLES>;
struct StepClusters {
    uint32_t fit[STEP_FEW_CLUSTER + 1] = {};           // clusters of each size that the device holds at once (B200: 15 of eight
                                                       // blocks, 33 of four, 45 of three, 74 of two)
    // Blocks per table for a call of n tables with blocks of `threads`; 0: two kernels.  All clusters of a call have to be
    // on the device at once; of smaller blocks an SM holds as many as make 1024 threads.
    // Above four blocks a cluster gains little (16 tables with 3, 4, 6 blocks 67.1, 66.1, 64.9 us; 12 with 3, 4, 8 52.2,
    // 51.3, 51.0; 8 with 4, 8 36.3, 35.8; 4 with 4, 8 23.8, 22.6) and takes SMs from what runs beside the call, so
    // only few tables get eight.  Two blocks are what is left above 45 tables: 64 tables 227 us, in two kernels 228.
    uint32_t of(uint32_t n, uint32_t threads) const
    {
        if (n > (uint32_t)STEP_MAX_TABLES) return 0;
        const uint32_t whole = (n * threads + 1023u) / 1024u;          // tables, in blocks of 1024 threads
        if (whole <= (uint32_t)STEP_FEW_TABLES && whole <= fit[STEP_FEW_CLUSTER]) return STEP_FEW_CLUSTER;
        for (uint32_t cl = 4; cl >= 2; --cl)
            if (whole <= fit[cl]) return cl;
        return 0;
    }
};
cudaError_t step_prepare(size_t max_smem);
// Whether the first block of a cluster has room for such a table (with up to 8192 slots it always has); with the `arriving`
// output: whether rows are asked for early.
bool step_serves(uint32_t S, uint32_t K, uint32_t n_q, uint32_t cluster, uint32_t row_bytes, bool arriving);
StepClusters step_clusters(size_t max_smem);            // after step_prepare
// Whether the blocks of a call in one kernel take no more than half of what the SMs hold of them.  Blocks of 1024 threads then leave half
// of the SMs to other grids; smaller ones, of which an SM holds several, may stand on all SMs and leave half of each.
inline bool step_leaves_half(uint32_t n, uint32_t threads, uint32_t cluster, uint32_t sm_count)
{
    return (uint64_t)n * cluster * threads <= (uint64_t)sm_count / 2u * 1024u;
}
// Whether a call that says when Stage One is done (reach: host bytes that its ids can reach) is better off with a kernel for each stage
// though it would leave half of the SMs.  Its consumer may run on another stream while the next calls queue.  The clusters then take
// the SMs that the consumer has left, and not those whose caches know their tables; where much has to be translated that costs more
// than the one kernel saves.  A call and a stand-in that reads all its rows on another stream (148 blocks, with 120 KB of shared memory /
// with none), four contexts in turn, a kernel for each stage -> one kernel: 12 tables, K = 2048, two tokens, 2.1 GB 79 -> 73 / 91 -> 79 us, 4.1
// GB 86 -> 99 / 96 -> 80, 8.3 GB 95 -> 128 / 111 -> 91; 14 tables, 9.6 GB 106 -> 123 / 129 -> 126; 18 tables, 3.1 GB 118 -> 102 / 122 -> 107; four
// tokens, 16 tables, 2.8 GB 183 -> 167 / 190 -> 181, 11 GB 244 -> 276 / 253 -> 288 (another box: 12 tables, 8.3 GB 94 -> 103 / 105 -> 87, 14 111 ->
// 116 / 126 -> 114).  And 18 tables without a consumer 101 -> 92 from 3.1, 104 -> 127 from 6.2 GB.  What is given up for that: with a
// consumer on the same stream 12 tables, 8.3 GB 104 -> 86.  With fewer ids or up to eight tables none of it is lost: 16 tables, K = 1000,
// 11 GB 51 -> 40 / 55 -> 40; 8 tables, 5.5 GB 69 -> 59 / 66 -> 58.
constexpr uint32_t STEP_FAR_IDS = 2048;                  // of a table
constexpr uint64_t STEP_FAR_BYTES = 3ull << 30;
inline bool step_reaches_far(uint32_t n, uint32_t table_ids, uint64_t reach)
{
    return n > (uint32_t)STEP_FEW_TABLES && table_ids > STEP_FAR_IDS && reach > STEP_FAR_BYTES;
}
// Whether the grid behind a call in one kernel may start under it (see the kernel).  Up to three tables; and up to eight, or as many
// as leave half of the SMs free with clusters of four, that reach little host memory (id_limit: rows a table's ids can
// reach).  Early / late, calls of K = 2048: one table 13.2 / 13.4
// us (0.08 GB) and 13.7 / 13.9 (0.6 GB); two 17.1 / 17.1, 18.0 / 18.0 (1.3 GB); three 21.4 / 21.3, 23.3 / 23.7 (1.9 GB); four 25.8 /
// 25.8 (0.3 GB), 27.8 / 27.3 (1.3 GB), 28.9 / 28.2 (2.6 GB); six 34.4 / 34.4 (0.5 GB), 36.7 / 36.0 (1.9 GB), 39.1 / 37.2 (3.8 GB); eight 42.8 /
// 42.8 (0.6 GB), 44.2 / 44.3 (1.3 GB), 45.2 / 44.9 (1.9 GB), 46.5 / 45.3 (2.6 GB), 58.3 / 46.7 (5.1 GB); five tables with K = 139 9.3 / 9.7.
// 12, 18 tables of K = 1000 27.0 / 27.6, 37.4 / 38.0 (0.1 and 0.2 GB), 31.4 / 32.0, 44.2 / 44.9 (0.5, 0.8 GB), 33.3 / 33.8, 49.8 / 47.6 (2.1, 3.1 GB); of
// K = 2048 37.6 / 38.1, 54.0 / 54.5, 60.0 / 60.4 and 52.9 / 53.4, 77.6 / 77.9, 89.9 / 87.4; 28 of S = 1024 13.9 / 14.1, 14.3 / 14.5, 15.2 / 15.2; but 12
// in clusters of eight of small blocks 9.5 / 9.3 (S = 1024), 20.1 / 20.1 (2048), 18.9 / 18.9 (4096; 1.8 GB 20.0 / 19.8).
// (Beside 100 GEMMs on another stream 100 calls of 9, 12, 16, 18 tables are through after 12.1, 12.8, 13.1, 13.5 ms so and 11.6, 12.4, 13.0, 14.0 late;
// beside 20 after 4.6, 5.2, 6.2, 6.8 and 5.4, 6.4, 7.4, 7.7.)
// Where the blocks leave no room nothing is gained (32 tables 113.0 / 112.9), and ids in host memory that are fetched under a call's rows slow these
// down (39 tables, K = 3430: 215 / 124).
template <int CAP>
bool step_early(const S1ParamsT<CAP>& p, uint32_t threads, uint32_t cluster, uint32_t sm_count)
{
    if (p.n_launch <= STEP_EARLY_TABLES) return true;
    if (p.host_ids || (p.n_launch > (uint32_t)STEP_FEW_TABLES && (cluster == STEP_FEW_CLUSTER || !step_leaves_half(p.n_launch, threads, cluster, sm_count))))
        return false;
    uint64_t bytes = 0;
    for (uint32_t i = 0; i < p.n_launch; ++i) bytes += p.id_limit[i] * p.kv_stride[i];
    return bytes <= STEP_EARLY_BYTES;
}
uint32_t step_threads(uint32_t S, uint32_t K);
// State that Stage One can read in pieces of 16 (ids) and 8 bytes (lifetimes).  A context's is; a caller's own may begin at
// any id and any lifetime (S is a multiple of 32, so that what holds for the first table holds for all).  Such a call takes
// two kernels, whose Stage One reads element by element: a test of the alignment inside the kernels made every call slower
// (one table 12.1 us, with it 12.6).
inline bool state_is_aligned(const int32_t* tok, const int8_t* life)
{
    return reinterpret_cast<uint64_t>(tok) % 16u == 0 && reinterpret_cast<uint64_t>(life) % 8u == 0;
}
// StepParamsFew: up to STEP_FEW_TABLES tables of STEP_FEW_CLUSTER blocks
template <int CAP> cudaError_t launch_step(const S1ParamsT<CAP>& p, uint32_t cluster, cudaStream_t stream);
// n_blocks thread blocks serve the p.n_launch tables of the launch (one block per table unless the call runs in rounds);
// state that is not aligned: with the small argument block only
cudaError_t launch_stage_one(const S1Params& p, uint32_t n_blocks, cudaStream_t stream);
cudaError_t launch_stage_one(const S1ParamsBig& p, uint32_t n_blocks, cudaStream_t stream);   // hash / direct index only
// Stage One with one table per thread-block cluster of C blocks (C = 2, 4 or 8; hash / direct index only)
size_t stage_one_cluster_smem_bytes(uint32_t S, uint32_t K, uint32_t n_q, uint32_t C);
cudaError_t stage_one_cluster_prepare(size_t max_smem);
int stage_one_cluster_max_active(uint32_t S, uint32_t K, uint32_t n_q, uint32_t C);   // after ..._prepare
cudaError_t launch_stage_one_cluster(const S1Params& p, uint32_t n_tables, uint32_t C, cudaStream_t stream);
cudaError_t launch_stage_one_cluster(const S1ParamsBig& p, uint32_t n_tables, uint32_t C, cudaStream_t stream);
cudaError_t launch_all_k_prepare(const AllKParams& p, uint32_t n_tables, cudaStream_t stream);
cudaError_t launch_transfer(const XferParams& p, uint32_t blocks, uint32_t threads, cudaStream_t stream);
cudaError_t launch_transfer_overlap(const XferOverlapParams& p, uint32_t blocks, uint32_t threads, cudaStream_t stream);
cudaError_t launch_transfer_overlap(const XferOverlapParamsBig& p, uint32_t blocks, uint32_t threads, cudaStream_t stream);
cudaError_t launch_transfer_positions(const PosParams& p, uint32_t blocks, uint32_t threads, cudaStream_t stream);

// Optional output of a call (latency hiding, Sec. 6 with Sec. 3.6): which positions' rows come with THIS call's
// Stage Two.  Calls in one kernel write it there (an instance of that kernel, see place_tokens()).  For the others it is a
// kernel of its own between Stage One and Stage Two, so that the Stage One kernels carry no code for
// an output few calls ask for (inside them it cost every call 1.7 us).  It also makes the call's "Stage One is
// done" announcement when the caller asked for both.
struct ArrivingParams {
    const SegDesc* seg;              // per table of the call: count = entries of its miss list
    const int2*    miss_list;        // [n][list_stride] (id, slot)
    const int32_t* slots;            // [n][per_table]
    uint8_t*       arriving;         // [n][per_table] out
    unsigned long long* done_seq;    // or null
    uint32_t*      done_ctr;         // wraps to zero at the grid size
    unsigned long long value;
    uint32_t n, per_table, S, list_stride;
    // overlapped Stage Two: Stage One's hand-over flags (see S1ParamsT), else null
    const uint32_t* flags;
    uint32_t announcers;             // Stage One blocks per table
    uint32_t n_q;
    uint32_t* status;
};
cudaError_t launch_arriving(const ArrivingParams& p, uint32_t blocks, cudaStream_t stream);
cudaError_t arriving_prepare();
cudaError_t transfer_prepare();

}  // namespace avsg
