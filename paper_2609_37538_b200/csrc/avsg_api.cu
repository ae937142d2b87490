// C ABI of the AVSG decode-step operator (see include/avsg.h): argument
// checking, device state, kernel launches.  No step of the operator runs on
// the host; there is no CPU fallback.
#include <new>
#include <string.h>
#include <vector>

#include <cuda.h>          // types of the one driver entry point fetched at run time (nothing links libcuda)

#include "avsg.h"
#include "avsg_kernels.cuh"
#include "host_buffers.h"

using namespace avsg;

namespace {
constexpr size_t HOST_ODD_IDS = 16384;             // see step_impl()
constexpr uint32_t XFER_THREADS = 256;             // per block of a transfer grid, unless the caller sets a geometry
constexpr size_t FLAG_BYTES = ((size_t)OVERLAP_MAX_TABLES * OVERLAP_MAX_TOKENS + 1) * sizeof(uint32_t);
}

struct avsg_ctx {
    avsg_config cfg;
    uint32_t logS = 0, logH = 0;
    uint32_t s1_cluster = 1;           // blocks that share one table in Stage One (1 = the single-block kernel)
    bool one_kernel = false;           // both stages in one kernel, where a call allows it
    uint32_t host_status = 0;          // status bits raised on the host side (sticky like the device word)
    uint32_t list_stride = 0;          // entries per miss-list segment
    int sm_count = 0;
    uint32_t xfer_blocks = 0, xfer_threads = XFER_THREADS;
    bool timing = false, events_recorded = false;

    int32_t* d_tok = nullptr;
    int8_t* d_life = nullptr;
    uint8_t* d_buffer = nullptr;
    TableStats* d_stats = nullptr;
    StepClusters step_clusters;                    // calls in one kernel
    bool geometry_set = false;                     // another geometry than the default one
    SharedRows* d_shared = nullptr;                // calls in one kernel [STEP_MAX_TABLES]
    uint32_t* d_flags = nullptr;                   // hand-over flags per (table of the call, token)
                                                   //   [OVERLAP_MAX_TABLES x TOKENS], and one that is never raised
    unsigned long long* d_sync = nullptr;          //   [2] sequence number of the last host-buffer call,
                                                   //   [3] arrivals after a host-buffer call's last token
    S1ParamsBig* big_args = nullptr;               // host: the large argument blocks, built in place per call
    XferOverlapParamsBig* big_xfer_args = nullptr;
    unsigned long long* d_trange = nullptr;        // [8] time marks of the last timed call, then [8] their initial values
    unsigned long long* d_trange_init = nullptr;
    int2* d_list = nullptr;
    SegDesc* d_seg = nullptr;
    uint32_t* d_status = nullptr;
    uint32_t* d_q = nullptr;           // paper-literal mode: packed words, or null
    uint32_t* d_q_snap = nullptr;
    int32_t* d_tok_snap = nullptr;
    int8_t* d_life_snap = nullptr;
    // staging of avsg_step_host
    int32_t* d_idx_stage = nullptr;
    int32_t* d_slots_stage = nullptr;
    uint8_t* d_hit_stage = nullptr;
    int32_t* d_mc_stage = nullptr;
    // copy-engine comparator (pinned host copies of the miss list)
    SegDesc* h_seg = nullptr;
    int2* h_list = nullptr;

    std::vector<uint64_t> kv_host, kv_dev;     // last validated host KV base per table
    std::vector<uint32_t> seen;                // distinctness check of table ids
    uint32_t epoch = 0;
    std::vector<const void*> call_kv_host;     // host pointers of the current call (copy-engine mode)
    std::vector<uint64_t> call_kv_dev;         // their device-visible addresses, resolved before anything is launched
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    // avsg_step_host: the outputs go back on a side stream while Stage Two runs
    cudaStream_t side = nullptr;
    // cuStreamWaitValue64, when driver and device offer it: in the overlapped mode the output download of a call
    // with host buffers waits for the sequence number Stage One writes once all its outputs exist, instead of for
    // an event between the two grids (which would run them one after the other)
    CUresult (*wait_value64)(CUstream, CUdeviceptr, cuuint64_t, unsigned int) = nullptr;
    unsigned long long host_seq = 0;               // calls with host buffers issued in that mode so far
    cudaEvent_t ev_outputs_ready = nullptr, ev_outputs_copied = nullptr, ev_ids_ready = nullptr;
    uint64_t last_rows = 0;
};

namespace {

struct DeviceGuard {
    int prev = -1;
    bool ok = true, other = false;
    explicit DeviceGuard(int dev)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
        other = prev != dev;
        if (other && cudaSetDevice(dev) != cudaSuccess) ok = false;
    }
    ~DeviceGuard() { if (other) cudaSetDevice(prev); }
};

#define CU(call) do { if ((call) != cudaSuccess) return AVSG_ECUDA; } while (0)

bool is_pow2(uint32_t v) { return v && !(v & (v - 1)); }
uint32_t ilog2(uint32_t v) { uint32_t l = 0; while ((1u << l) < v) ++l; return l; }

void free_all(avsg_ctx* c)
{
    cudaFree(c->d_tok); cudaFree(c->d_life); cudaFree(c->d_buffer); cudaFree(c->d_stats); cudaFree(c->d_trange);
    cudaFree(c->d_shared); cudaFree(c->d_flags); cudaFree(c->d_sync);
    delete c->big_args;
    delete c->big_xfer_args;
    cudaFree(c->d_list); cudaFree(c->d_seg); cudaFree(c->d_status); cudaFree(c->d_q); cudaFree(c->d_q_snap);
    cudaFree(c->d_tok_snap); cudaFree(c->d_life_snap);
    cudaFree(c->d_idx_stage); cudaFree(c->d_slots_stage); cudaFree(c->d_hit_stage); cudaFree(c->d_mc_stage);
    if (c->h_seg) cudaFreeHost(c->h_seg);
    if (c->h_list) cudaFreeHost(c->h_list);
    for (auto& e : c->ev) if (e) cudaEventDestroy(e);
    if (c->ev_outputs_ready) cudaEventDestroy(c->ev_outputs_ready);
    if (c->ev_outputs_copied) cudaEventDestroy(c->ev_outputs_copied);
    if (c->ev_ids_ready) cudaEventDestroy(c->ev_ids_ready);
    if (c->side) cudaStreamDestroy(c->side);
}

int init_tables(avsg_ctx* c, uint32_t first, uint32_t n)
{
    const size_t S = c->cfg.buffer_slots;
    CU(cudaMemset(c->d_tok + first * S, 0xFF, n * S * sizeof(int32_t)));        // id -1: empty
    CU(cudaMemset(c->d_life + first * S, 0xFF, n * S));                         // lifetime -1: dead
    CU(cudaMemset(c->d_buffer + first * S * c->cfg.row_bytes, 0, n * S * c->cfg.row_bytes));
    CU(cudaMemset(c->d_stats + first, 0, n * sizeof(TableStats)));
    if (c->d_q) {                                           // lifetime -1, mapping invalid: 0xFF800000
        std::vector<uint32_t> init(n * S, 0xFF800000u);
        CU(cudaMemcpy(c->d_q + first * S, init.data(), init.size() * sizeof(uint32_t), cudaMemcpyHostToDevice));
    }
    return AVSG_OK;
}

// Device-visible address of a host KV base (pinned + mapped host memory, or device memory).
int resolve_kv(avsg_ctx* c, uint32_t table, const void* host_ptr, uint64_t* dev)
{
    const uint64_t h = reinterpret_cast<uint64_t>(host_ptr);
    if (c->kv_host[table] == h && c->kv_dev[table]) { *dev = c->kv_dev[table]; return AVSG_OK; }
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, host_ptr) != cudaSuccess) { cudaGetLastError(); return AVSG_EINVAL; }
    if (at.type == cudaMemoryTypeUnregistered || at.devicePointer == nullptr) return AVSG_EINVAL;
    c->kv_host[table] = h;
    c->kv_dev[table] = reinterpret_cast<uint64_t>(at.devicePointer);
    *dev = c->kv_dev[table];
    return AVSG_OK;
}

int check_args(avsg_ctx* c, const avsg_step_args* a)
{
    if (!c || !a) return AVSG_EINVAL;
    if (a->n == 0 || a->n > c->cfg.num_tables || a->n > (uint32_t)XFER_MAX_SEG) return AVSG_EINVAL;
    if (!a->table_ids || !a->indices || !a->kv_base || !(a->verified_len || a->verified_len_dev) || !a->slots)
        return AVSG_EINVAL;
    if (a->n_tokens == 0 || a->n_tokens > c->cfg.max_tokens || a->topk == 0 || a->topk > c->cfg.max_topk)
        return AVSG_EINVAL;
    if ((uint64_t)a->n_tokens * a->topk > c->cfg.buffer_slots) return AVSG_ECAPACITY;      // Eq. 7
    if (++c->epoch == 0) { std::fill(c->seen.begin(), c->seen.end(), 0u); c->epoch = 1; }
    for (uint32_t i = 0; i < a->n; ++i) {
        const uint32_t t = a->table_ids[i];
        if (t >= c->cfg.num_tables || c->seen[t] == c->epoch) return AVSG_EINVAL;
        c->seen[t] = c->epoch;
        if (a->row_stride && (a->row_stride[i] % 16 || a->row_stride[i] < c->cfg.row_bytes)) return AVSG_EINVAL;
        if (!a->kv_base[i] || (reinterpret_cast<uint64_t>(a->kv_base[i]) & 15u)) return AVSG_EINVAL;
        if (a->kv_rows && a->kv_rows[i] > 0x80000000u) return AVSG_EINVAL;
    }
    return AVSG_OK;
}

// Comparator: the miss list goes back to the host, then one asynchronous copy per run of
// consecutive (host row, slot) pairs is queued on the copy engine.
int copy_engine_transfer(avsg_ctx* c, const avsg_step_args* a, cudaStream_t stream)
{
    const uint32_t n = a->n;
    CU(cudaMemcpyAsync(c->h_seg, c->d_seg, n * sizeof(SegDesc), cudaMemcpyDeviceToHost, stream));
    CU(cudaStreamSynchronize(stream));
    uint32_t max_count = 0;
    for (uint32_t i = 0; i < n; ++i) max_count = c->h_seg[i].count > max_count ? c->h_seg[i].count : max_count;
    if (max_count == 0) return AVSG_OK;
    if (max_count > c->list_stride) return AVSG_EDEVICE_STATUS;
    const size_t pitch = (size_t)c->list_stride * sizeof(int2);
    CU(cudaMemcpy2DAsync(c->h_list, pitch, c->d_list, pitch, (size_t)max_count * sizeof(int2), n,
                         cudaMemcpyDeviceToHost, stream));
    CU(cudaStreamSynchronize(stream));
    const uint64_t rb = c->cfg.row_bytes;
    for (uint32_t i = 0; i < n; ++i) {
        const SegDesc& sd = c->h_seg[i];
        const int2* e = c->h_list + (size_t)i * c->list_stride;
        const uint8_t* src_base = static_cast<const uint8_t*>(c->call_kv_host[i]);
        uint32_t k = 0;
        while (k < sd.count) {
            if (e[k].x < 0 || e[k].y < 0 || (uint32_t)e[k].y >= c->cfg.buffer_slots) { ++k; continue; }
            uint32_t run = 1;
            if (sd.src_stride == rb)
                while (k + run < sd.count && e[k + run].x == e[k].x + (int32_t)run && e[k + run].y == e[k].y + (int32_t)run) ++run;
            CU(cudaMemcpyAsync(reinterpret_cast<void*>(sd.dst_base + (uint64_t)e[k].y * rb),
                               src_base + (uint64_t)e[k].x * sd.src_stride, run * rb, cudaMemcpyDefault, stream));
            k += run;
        }
    }
    return AVSG_OK;
}

// The transfer kernel's arguments but for the tables' own.
template <typename X>
void overlap_params(avsg_ctx* c, X& x, uint32_t n, uint32_t n_q, uint32_t round_size)
{
    x.miss_list = c->d_list; x.status = c->d_status; x.buffer = c->d_buffer;
    x.flags = c->d_flags; x.announcers = c->s1_cluster;
    x.n = n; x.n_q = n_q; x.list_stride = c->list_stride; x.row_bytes = c->cfg.row_bytes; x.S = c->cfg.buffer_slots;
    x.round_size = round_size; x.t_range = nullptr;
}

int step_impl(avsg_ctx* c, const avsg_step_args* a, cudaStream_t stream, bool host_io)
{
    int rc = check_args(c, a);
    if (rc != AVSG_OK) return rc;
    if ((a->stage_one_done || a->arriving) && (host_io || c->cfg.transfer_mode == AVSG_XFER_ALL_K ||
                                               (reinterpret_cast<uint64_t>(a->stage_one_done) & 7u)))
        return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;

    const uint32_t n = a->n, K = a->topk, n_q = a->n_tokens;
    const size_t n_ids = (size_t)n * n_q * K;
    const int32_t* indices = a->indices;
    int32_t* slots = a->slots;
    uint8_t* hit = a->hit;
    int32_t* miss_count = a->miss_count;
    // Host buffers.  Page-locked ones are used by the kernels themselves: Stage One reads the ids in place and Stage Two
    // writes the outputs back, so that the calls of a stream follow one another as launches do, without an event between
    // them (measured with 32 tables: see put_outputs()).  Pageable ones, the paper-literal kernel and the comparators
    // go through copies on a side stream, and so do tables of several Stage One blocks, each of which would read all ids
    // from the host (in two kernels, S = 16384 with 38, 50, 64 tables 168, 210, 263 us by copies, 219, 285, 372 in place; S = 32768, four
    // tokens, 16 tables 146 and 306; only one to four tables were quicker in place).  So do calls of more than
    // HOST_ODD_IDS ids whose tokens do not all begin on 32-byte boundaries, which the link moves in parts of its units, while
    // a copy costs its event.  In place, begun 0, 32 and 4 bytes behind a line / by copies: 32 tables with K = 264 (four
    // tokens) 51, 44, - / 71; 520 (two) 44, 34, 60 / 62; 2048 (two) 139, 130, 222 / 153; 100 tables, one token, K = 168 31, 30,
    // 61 / 51; 328 41, 34, 84 / 58; six tables, K = 1000, four tokens 37, 34, 69 / 57; 16384 ids: eight tables, two tokens 26,
    // 21, 42 / 45; 32 tables, one token 22, 18, 32 / 41.  And ids that do not begin on a word's boundary, which the copies take.
    HostOut out;
    bool host_ids = false;
    // One kernel for both stages, where the tables' clusters fit the device (see avsg_step_kernel for what it saves).  Its
    // blocks take whole SMs.  So a caller who wants the hits before the rows are there (stage_one_done) gets it from calls that
    // leave half of the SMs to the kernel that starts on the hits (or are small: STEP_EARLY_TABLES), unless they reach far
    // (step_reaches_far()), and that kernel may start at once.  K = 2048, two tokens, 64 Ki positions, with both early outputs, three
    // kernels / one, 3, 8, 18 tables: calls alone 32.7 / 20.7, 58.7 / 46.0, 109.1 / 95.9 us; each with a stand-in for a consumer (see
    // step_reaches_far()) behind it on the stream, which starts with the call, 42.8 / 31.2, 76.9 / 57.0, 138.2 / 120.1; with one on
    // another stream while the next calls queue 40.9 / 32.6, 71.8 / 59.9, 125.3 / 109.5; if the next call waits for that one too 51.3 / 45.3,
    // 85.3 / 69.1, 141.9 / 117.9.  What loses is this last way with a consumer that would fill the SMs besides (no shared memory): the
    // one kernel's word comes later than a Stage One grid's, and half of the SMs are taken (K = 2048, one token, 12, 14, 16, 18 tables 60.7,
    // 62.4, 62.3, 66.7 / 58.8, 64.4, 68.2, 71.4; small blocks, S = 1024, K = 256, 18, 31, 37 tables 41.3, 42.5, 42.1 / 36.9, 43.2, 45.9).
    // If the kernel behind such a call came only at its end, calls without a consumer would keep their SMs from one to the next (8
    // tables, 5.5 GB 63.6 us, then 45.4, in three kernels 58.6), but a consumer on the same stream could not start (57.1, 66.4, 72.7).
    //
    // id_limit_of: ids at or beyond this are never looked up or fetched: the table's host rows when the caller states them,
    // and the size of the direct index
    auto id_limit_of = [&](uint32_t i) -> uint32_t {
        uint32_t lim = a->kv_rows ? a->kv_rows[i] : 0x80000000u;
        if (c->cfg.index_mode == AVSG_INDEX_DIRECT && c->cfg.max_context < lim) lim = c->cfg.max_context;
        return lim;
    };
    auto stride_of = [&](uint32_t i) -> uint64_t { return a->row_stride ? a->row_stride[i] : c->cfg.row_bytes; };
    auto reach = [&] {
        uint64_t bytes = 0;
        for (uint32_t i = 0; i < n; ++i) bytes += id_limit_of(i) * stride_of(i);
        return bytes;
    };
    const bool sm_copies = c->cfg.transfer_mode == AVSG_XFER_SM_BALANCED || c->cfg.transfer_mode == AVSG_XFER_SM_OVERLAP;
    uint32_t cluster = 0;
    if (sm_copies && c->one_kernel && n_q <= STEP_MAX_TOKENS && !c->timing && !c->geometry_set) {
        cluster = c->step_clusters.of(n, step_threads(c->cfg.buffer_slots, K));
        if (cluster && !step_serves(c->cfg.buffer_slots, K, n_q, cluster, c->cfg.row_bytes, a->arriving != nullptr)) cluster = 0;
        if (cluster && a->stage_one_done && n > STEP_EARLY_TABLES &&
            (!step_leaves_half(n, step_threads(c->cfg.buffer_slots, K), cluster, (uint32_t)c->sm_count) || step_reaches_far(n, n_q * K, reach())))
            cluster = 0;
    }
    const bool in_place = (K % 8u == 0 && reinterpret_cast<uint64_t>(a->indices) % 32u == 0) || n_ids <= HOST_ODD_IDS;
    if (host_io && c->cfg.index_mode != AVSG_INDEX_PAPER && (c->s1_cluster == 1 || cluster) && in_place && sm_copies) {
        const int32_t* ids = reinterpret_cast<uint64_t>(a->indices) % 4u == 0 ? mapped(a->indices, n_ids) : nullptr;
        out.host_slots = mapped(a->slots, n_ids);
        out.host_hit = a->hit ? mapped(a->hit, n_ids) : nullptr;
        out.host_count = a->miss_count ? mapped(a->miss_count, (size_t)n * n_q) : nullptr;
        if (ids && out.host_slots && !a->hit == !out.host_hit && !a->miss_count == !out.host_count) {
            host_ids = true;
            host_io = false;
            indices = ids;
            out.slots = slots = c->d_slots_stage; out.n_slots = (uint32_t)n_ids;
            out.hit = hit = a->hit ? c->d_hit_stage : nullptr; out.n_hit = a->hit ? (uint32_t)n_ids : 0u;
            out.count = miss_count = a->miss_count ? c->d_mc_stage : nullptr; out.n_count = a->miss_count ? n * n_q : 0u;
        }
    }
    if (host_io) {
        // The ids go up on the side stream, where they queue behind the previous call's output download (and
        // therefore behind its Stage One, the last reader of the staging buffer) but not behind its Stage Two:
        // when calls are issued back to back the upload hides under the previous call's gather.
        CU(cudaMemcpyAsync(c->d_idx_stage, a->indices, n_ids * sizeof(int32_t), cudaMemcpyHostToDevice, c->side));
        CU(cudaEventRecord(c->ev_ids_ready, c->side));
        CU(cudaStreamWaitEvent(stream, c->ev_ids_ready, 0));
        indices = c->d_idx_stage;
        slots = c->d_slots_stage;
        hit = a->hit ? c->d_hit_stage : nullptr;
        miss_count = a->miss_count ? c->d_mc_stage : nullptr;
    }
    uint32_t mode = c->cfg.transfer_mode;
    // tables per Stage One launch: the small argument block when it is enough (and for the kernels that only have
    // that one), else the large one
    const uint32_t chunk = (n <= (uint32_t)S1_MAX_TABLES || mode == AVSG_XFER_ALL_K || c->cfg.index_mode == AVSG_INDEX_PAPER)
                               ? (uint32_t)S1_MAX_TABLES : (uint32_t)S1_BIG_TABLES;
    // With a Stage One block per table on most of the SMs, the blocks of a transfer kernel behind it crowd onto the rest: a
    // balanced call of that many tables is served like an overlapped one, in rounds (below).  128 tables with 2.8, 5.5, 11
    // GB of host memory 414, 575, 743 us behind Stage One, 393, 426, 443 in rounds; 80 tables 251 and 250; from and to
    // host memory 80, 96, 128 tables 316, 375, 537 and 305, 365, 487.
    if (mode == AVSG_XFER_SM_BALANCED && n > (uint32_t)c->sm_count / 2 && c->s1_cluster == 1 && c->cfg.index_mode != AVSG_INDEX_PAPER &&
        !host_io && !c->timing && !c->geometry_set)
        mode = AVSG_XFER_SM_OVERLAP;
    if (mode == AVSG_XFER_SM_OVERLAP && (n > chunk || n_q > (uint32_t)OVERLAP_MAX_TOKENS))
        mode = AVSG_XFER_SM_BALANCED;                  // the overlapped kernel pairs with ONE Stage One launch
    // The overlapped transfer grid shares the GPU with the Stage One grid it waits for.  When Stage One's blocks
    // take more than half of the SMs, many transfer blocks only find room once Stage One is over and their fixed
    // shares (Eq. 6) finish late: measured, a 96- or 128-table call with one Stage One block per table is 3-6 %
    // slower overlapped than not (64: 2 % faster).
    // Such calls keep Stage One on S1_ROUND_BLOCKS SMs: its blocks serve the tables round by round and the transfer
    // grid, resident on the other SMs, copies round r's misses while round r + 1 is matched (single-block hash /
    // direct kernels; the cluster and paper-literal kernels run Stage Two after Stage One instead).
    uint32_t round_size = n;
    if (mode == AVSG_XFER_SM_OVERLAP && (uint64_t)n * c->s1_cluster > (uint64_t)c->sm_count / 2) {
        if (c->s1_cluster == 1 && c->cfg.index_mode != AVSG_INDEX_PAPER)
            round_size = S1_ROUND_BLOCKS;
        else
            mode = AVSG_XFER_SM_BALANCED;
    }
    // host buffers in the overlapped mode: no event between the two grids, the download waits for a sequence number
    const bool overlap = mode == AVSG_XFER_SM_OVERLAP;
    const bool wait_on_sequence = host_io && overlap && c->wait_value64 != nullptr;
    // the position-level comparator reads the hit mask: use the library's own buffer if the caller wants none
    if (mode == AVSG_XFER_POSITION_LEVEL && !hit) hit = c->d_hit_stage;
    if (c->timing) {
        // grid spans: [0] Stage One first start, [1] its last end, [2], [3] the same for Stage Two
        CU(cudaMemcpyAsync(c->d_trange, c->d_trange_init, 8 * sizeof(unsigned long long), cudaMemcpyDeviceToDevice, stream));
        CU(cudaEventRecord(c->ev[0], stream));
    }

    c->call_kv_host.assign(a->kv_base, a->kv_base + n);
    // every host KV base is resolved (and refused, if the GPU cannot read it) before the first launch of the call:
    // a call either starts completely or not at all
    c->call_kv_dev.resize(n);
    for (uint32_t i = 0; i < n; ++i)
        if ((rc = resolve_kv(c, a->table_ids[i], a->kv_base[i], &c->call_kv_dev[i])) != AVSG_OK) return rc;
    // Stage One's arguments for tables [first, first + cnt) of the call, and its launch with the small or the large block
    auto fill = [&](auto& p, uint32_t first, uint32_t cnt) {
        p.tok = c->d_tok; p.life = c->d_life; p.buffer = c->d_buffer; p.stats = c->d_stats;
        p.miss_list = c->d_list; p.seg = c->d_seg; p.status = c->d_status;
        p.indices = indices; p.slots = slots; p.hit = hit; p.miss_count = miss_count;
        p.host_ids = host_ids;
        p.S = c->cfg.buffer_slots; p.logH = c->logH; p.row_bytes = c->cfg.row_bytes;
        p.K = K; p.n_q = n_q; p.L = (uint32_t)c->cfg.max_lifetime;
        p.first = first; p.list_stride = c->list_stride;
        p.n_launch = cnt;
        // A transfer grid that is placed while Stage One holds nearly all SMs crowds onto the others: it has to wait then
        // (S = 16384, two blocks a table, not overlapped, 64 and 72 tables: 334, 311 us and 233, 259 where it waits; with 50
        // tables 186 and 185).
        p.early = cnt * c->s1_cluster <= (uint32_t)c->sm_count * 3u / 4u;
        p.qword = c->d_q; p.probe_retries = c->cfg.probe_retries; p.hash_a1 = c->cfg.hash_a1; p.hash_a2 = c->cfg.hash_a2;
        p.t_range = c->timing ? c->d_trange : nullptr;
        p.verified_len_dev = a->verified_len_dev;
        // (every field is assigned: the large block is re-used from call to call)
        p.flags = overlap ? c->d_flags : nullptr;
        // the caller's word: written by Stage One itself, or by the `arriving` kernel behind it when that output
        // is asked for too (the word then also covers it)
        p.done_seq = wait_on_sequence ? c->d_sync + 2
                                      : (a->arriving ? nullptr : reinterpret_cast<unsigned long long*>(a->stage_one_done));
        p.done_ctr = reinterpret_cast<uint32_t*>(c->d_sync + 3);
        p.host_seq = wait_on_sequence ? c->host_seq + 1 : a->stage_one_done_value;
        p.expect = n * c->s1_cluster;
        for (uint32_t i = 0; i < cnt; ++i) {
            p.table_id[i] = a->table_ids[first + i];
            p.verified_len[i] = a->verified_len ? a->verified_len[first + i] : 0;
            p.id_limit[i] = id_limit_of(first + i);
            p.kv_base[i] = c->call_kv_dev[first + i];
            p.kv_stride[i] = stride_of(first + i);
        }
    };
    auto stage_one = [&](auto& p, uint32_t first, uint32_t cnt) -> int {
        fill(p, first, cnt);
        if (c->s1_cluster > 1) CU(launch_stage_one_cluster(p, cnt, c->s1_cluster, stream));
        else CU(launch_stage_one(p, cnt < round_size ? cnt : round_size, stream));
        return AVSG_OK;
    };
    if (cluster && !host_io) {
        auto step = [&](auto&& p) -> int {
            fill(p, 0, n);
            p.flags = nullptr; p.expect = n; p.out = out; p.shared = c->d_shared; p.arriving = a->arriving;
            p.done_seq = reinterpret_cast<unsigned long long*>(a->stage_one_done);
            p.early = a->stage_one_done || step_early(p, step_threads(p.S, K), cluster, (uint32_t)c->sm_count);
            CU(launch_step(p, cluster, stream));
            return AVSG_OK;
        };
        return cluster == STEP_FEW_CLUSTER && n <= (uint32_t)STEP_FEW_TABLES ? step(StepParamsFew()) : step(StepParams());
    }
    for (uint32_t first = 0; first < n; first += chunk) {
        const uint32_t cnt = n - first < chunk ? n - first : chunk;
        if (mode == AVSG_XFER_ALL_K) {
            AllKParams p;
            p.indices = indices; p.slots = slots; p.hit = hit; p.miss_count = miss_count;
            p.miss_list = c->d_list; p.seg = c->d_seg; p.stats = c->d_stats; p.buffer = c->d_buffer;
            p.status = c->d_status;
            p.S = c->cfg.buffer_slots; p.row_bytes = c->cfg.row_bytes; p.K = K; p.n_q = n_q;
            p.first = first; p.list_stride = c->list_stride;
            for (uint32_t i = 0; i < cnt; ++i) {
                p.table_id[i] = a->table_ids[first + i];
                p.id_limit[i] = id_limit_of(first + i);
                p.kv_base[i] = c->call_kv_dev[first + i];
                p.kv_stride[i] = stride_of(first + i);
            }
            CU(launch_all_k_prepare(p, cnt, stream));
        } else if (chunk == (uint32_t)S1_MAX_TABLES) {
            S1Params p;
            if ((rc = stage_one(p, first, cnt)) != AVSG_OK) return rc;
        } else {
            if ((rc = stage_one(*c->big_args, first, cnt)) != AVSG_OK) return rc;
        }
    }
    if (a->arriving) {
        ArrivingParams q;
        q.seg = c->d_seg; q.miss_list = c->d_list; q.slots = slots; q.arriving = a->arriving;
        q.done_seq = reinterpret_cast<unsigned long long*>(a->stage_one_done);
        q.done_ctr = reinterpret_cast<uint32_t*>(c->d_sync + 3);
        q.value = a->stage_one_done_value;
        q.n = n; q.per_table = n_q * K; q.S = c->cfg.buffer_slots; q.list_stride = c->list_stride;
        q.flags = overlap ? c->d_flags : nullptr;
        q.announcers = c->s1_cluster; q.n_q = n_q; q.status = c->d_status;
        CU(launch_arriving(q, (uint32_t)c->sm_count, stream));
    }
    // (no event between the two grids in overlap mode: it would serialise them; ev[1] is recorded with ev[2])
    if (c->timing && mode != AVSG_XFER_SM_OVERLAP) CU(cudaEventRecord(c->ev[1], stream));

    // The slot table, hit mask and miss counts are final once Stage One has run.  They travel device -> host on a
    // side stream while Stage Two pulls rows host -> device: the two directions of the link overlap.
    auto download_outputs = [&]() -> int {
        CU(cudaMemcpyAsync(a->slots, c->d_slots_stage, n_ids * sizeof(int32_t), cudaMemcpyDeviceToHost, c->side));
        if (a->hit) CU(cudaMemcpyAsync(a->hit, c->d_hit_stage, n_ids, cudaMemcpyDeviceToHost, c->side));
        if (a->miss_count)
            CU(cudaMemcpyAsync(a->miss_count, c->d_mc_stage, (size_t)n * n_q * sizeof(int32_t), cudaMemcpyDeviceToHost, c->side));
        CU(cudaEventRecord(c->ev_outputs_copied, c->side));
        return AVSG_OK;
    };
    if (host_io && !wait_on_sequence) {
        CU(cudaEventRecord(c->ev_outputs_ready, stream));
        CU(cudaStreamWaitEvent(c->side, c->ev_outputs_ready, 0));
        if ((rc = download_outputs()) != AVSG_OK) return rc;
    }

    if (mode == AVSG_XFER_COPY_ENGINE) {
        if ((rc = copy_engine_transfer(c, a, stream)) != AVSG_OK) return rc;
    } else if (mode == AVSG_XFER_POSITION_LEVEL) {
        PosParams q;
        q.seg = c->d_seg; q.indices = indices; q.slots = slots; q.hit = hit; q.status = c->d_status;
        q.n = n; q.per_table = n_q * K; q.row_bytes = c->cfg.row_bytes; q.S = c->cfg.buffer_slots;
        CU(launch_transfer_positions(q, c->xfer_blocks ? c->xfer_blocks : (uint32_t)c->sm_count, c->xfer_threads, stream));
    } else if (overlap) {
        auto launch = [&](auto& x) -> cudaError_t {
            overlap_params(c, x, n, n_q, round_size);
            x.out = out;
            x.t_range = c->timing ? c->d_trange + 2 : nullptr;
            for (uint32_t i = 0; i < n; ++i) {
                x.table_id[i] = a->table_ids[i];
                x.kv_base[i] = c->call_kv_dev[i];
                x.kv_stride[i] = stride_of(i);
            }
            return launch_transfer_overlap(x, c->xfer_blocks ? c->xfer_blocks : (uint32_t)c->sm_count, c->xfer_threads, stream);
        };
        cudaError_t e;
        if (n <= (uint32_t)S1_MAX_TABLES) {
            XferOverlapParams x;
            e = launch(x);
        } else {
            e = launch(*c->big_xfer_args);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();                  // this call reserved slots whose rows were never copied
            c->host_status |= AVSG_STATUS_LAUNCH_FAILED;
            return AVSG_ECUDA;
        }
        if (wait_on_sequence) {
            c->host_seq += 1;
            if (c->wait_value64(c->side, reinterpret_cast<CUdeviceptr>(c->d_sync + 2), c->host_seq,
                                CU_STREAM_WAIT_VALUE_GEQ) != CUDA_SUCCESS)
                return AVSG_ECUDA;
            if ((rc = download_outputs()) != AVSG_OK) return rc;
        }
    } else {
        XferParams x;
        x.seg = c->d_seg; x.miss_list = c->d_list; x.status = c->d_status;
        x.n_seg = n; x.list_stride = c->list_stride; x.row_bytes = c->cfg.row_bytes;
        x.request_level = mode == AVSG_XFER_REQUEST_LEVEL; x.S = c->cfg.buffer_slots;
        x.out = out;
        x.t_range = c->timing ? c->d_trange + 2 : nullptr;
        const uint32_t blocks = x.request_level ? n : (c->xfer_blocks ? c->xfer_blocks : (uint32_t)c->sm_count);
        if (launch_transfer(x, blocks, c->xfer_threads, stream) != cudaSuccess) {
            cudaGetLastError();
            c->host_status |= AVSG_STATUS_LAUNCH_FAILED;
            return AVSG_ECUDA;
        }
    }
    if (c->timing) {
        if (mode == AVSG_XFER_SM_OVERLAP) CU(cudaEventRecord(c->ev[1], stream));
        CU(cudaEventRecord(c->ev[2], stream));
        c->events_recorded = true;
    }

    if (host_io) CU(cudaStreamWaitEvent(stream, c->ev_outputs_copied, 0));     // the call ends when the outputs are home
    return AVSG_OK;
}

int read_status(avsg_ctx* c, uint32_t* word)
{
    uint32_t st = 0;
    CU(cudaMemcpy(&st, c->d_status, sizeof(st), cudaMemcpyDeviceToHost));
    st |= c->host_status;
    if (word) *word = st;
    return st ? AVSG_EDEVICE_STATUS : AVSG_OK;
}

}  // namespace

extern "C" {

int avsg_create(const avsg_config* cfg, avsg_ctx** out)
{
    if (!cfg || !out) return AVSG_EINVAL;
    if (cfg->num_tables == 0 || !is_pow2(cfg->buffer_slots) || cfg->buffer_slots < 32) return AVSG_EINVAL;
    if (cfg->buffer_slots > 32768) return AVSG_EUNSUPPORTED;
    if (cfg->stage_one_cluster > 8 || (cfg->stage_one_cluster & (cfg->stage_one_cluster - 1))) return AVSG_EINVAL;
    if (cfg->max_topk > 32768) return AVSG_EUNSUPPORTED;
    if (cfg->row_bytes == 0 || cfg->row_bytes % 16) return AVSG_EINVAL;
    if (cfg->max_topk == 0 || cfg->max_tokens == 0) return AVSG_EINVAL;
    if (cfg->max_lifetime < 1 || cfg->max_lifetime > 126) return AVSG_EINVAL;
    if (cfg->transfer_mode > AVSG_XFER_SM_OVERLAP || cfg->index_mode > AVSG_INDEX_PAPER) return AVSG_EINVAL;
    if (cfg->index_mode == AVSG_INDEX_DIRECT && cfg->max_context == 0) return AVSG_EINVAL;
    if ((uint64_t)cfg->max_topk * cfg->max_tokens > cfg->buffer_slots) return AVSG_ECAPACITY;   // Eq. 7
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || cfg->device < 0 || cfg->device >= ndev) return AVSG_ECUDA;
    DeviceGuard guard(cfg->device);
    if (!guard.ok) return AVSG_ECUDA;

    avsg_ctx* c = new (std::nothrow) avsg_ctx();
    if (!c) return AVSG_ENOMEM;
    c->cfg = *cfg;
    if (c->cfg.probe_retries == 0) c->cfg.probe_retries = 3;
    if (c->cfg.hash_a1 == 0) c->cfg.hash_a1 = 1000003u;
    if (c->cfg.hash_a2 == 0) c->cfg.hash_a2 = 998244353u;
    c->logS = ilog2(cfg->buffer_slots);
    c->logH = c->logS + 1;
    c->list_stride = cfg->max_topk * cfg->max_tokens;
    const size_t T = cfg->num_tables, S = cfg->buffer_slots;
    c->kv_host.assign(T, 0); c->kv_dev.assign(T, 0); c->seen.assign(T, 0);

    int max_smem = 0;
    cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, cfg->device);
    cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, cfg->device);
    // Blocks per table in Stage One: what the configuration asks for, else the single-block kernel while the table
    // fits one SM's shared memory and the smallest cluster that holds it above that.
    {
        const uint32_t S = cfg->buffer_slots, K = cfg->max_topk, L = (uint32_t)cfg->max_lifetime;
        auto fits = [&](uint32_t C) -> bool {
            if (cfg->index_mode == AVSG_INDEX_PAPER)
                return C == 1 && S <= 8192 && stage_one_paper_smem_bytes(S, K, L) <= (size_t)max_smem;
            if (C == 1) return S <= 8192 && stage_one_smem_bytes(S, K, cfg->max_tokens) <= (size_t)max_smem;
            return S / C >= 32 && S / C <= 8192 && stage_one_cluster_smem_bytes(S, K, cfg->max_tokens, C) <= (size_t)max_smem;
        };
        uint32_t C = cfg->stage_one_cluster;
        if (C == 0)
            for (C = 1; C <= 8 && !fits(C); C *= 2) {}
        if (C > 8 || !fits(C)) { delete c; return AVSG_EUNSUPPORTED; }
        c->s1_cluster = C;
        c->one_kernel = cfg->index_mode != AVSG_INDEX_PAPER && (C == 1 || (cfg->stage_one_cluster == 0 && S <= STEP_MAX_SLOTS));
    }
    // always raise the kernels' dynamic shared-memory limit to the device maximum: the attribute is
    // per function, so a context with a small table must not lower it under a context with a large one
    if (stage_one_prepare((size_t)max_smem) != cudaSuccess || step_prepare((size_t)max_smem) != cudaSuccess || stage_one_cluster_prepare((size_t)max_smem) != cudaSuccess ||
        transfer_prepare() != cudaSuccess || arriving_prepare() != cudaSuccess) {
        delete c; return AVSG_ECUDA;
    }
    c->step_clusters = step_clusters((size_t)max_smem);
    // a cluster shape that fits on paper may still find no home on the device (blocks of one cluster share a GPC)
    if (c->s1_cluster > 1 &&
        stage_one_cluster_max_active(cfg->buffer_slots, cfg->max_topk, cfg->max_tokens, c->s1_cluster) < 1) {
        delete c; return AVSG_EUNSUPPORTED;
    }

    const size_t n_ids = T * c->list_stride;
    bool ok = true;
    ok = ok && cudaMalloc(&c->d_tok, T * S * sizeof(int32_t)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_life, T * S) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_buffer, T * S * cfg->row_bytes) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_stats, T * sizeof(TableStats)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_trange, 16 * sizeof(unsigned long long)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_shared, STEP_MAX_TABLES * sizeof(SharedRows)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_flags, FLAG_BYTES) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_sync, 8 * sizeof(unsigned long long)) == cudaSuccess;
    c->big_args = new (std::nothrow) S1ParamsBig();
    c->big_xfer_args = new (std::nothrow) XferOverlapParamsBig();
    ok = ok && c->big_args != nullptr && c->big_xfer_args != nullptr;
    ok = ok && cudaMalloc(&c->d_list, n_ids * sizeof(int2)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_seg, T * sizeof(SegDesc)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_status, 256) == cudaSuccess;
    if (cfg->index_mode == AVSG_INDEX_PAPER) {
        ok = ok && cudaMalloc(&c->d_q, T * S * sizeof(uint32_t)) == cudaSuccess;
        ok = ok && cudaMalloc(&c->d_q_snap, T * S * sizeof(uint32_t)) == cudaSuccess;
    }
    ok = ok && cudaMalloc(&c->d_tok_snap, T * S * sizeof(int32_t)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_life_snap, T * S) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_idx_stage, n_ids * sizeof(int32_t)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_slots_stage, n_ids * sizeof(int32_t)) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_hit_stage, n_ids) == cudaSuccess;
    ok = ok && cudaMalloc(&c->d_mc_stage, T * cfg->max_tokens * sizeof(int32_t)) == cudaSuccess;
    ok = ok && cudaHostAlloc(&c->h_seg, T * sizeof(SegDesc), cudaHostAllocDefault) == cudaSuccess;
    ok = ok && cudaHostAlloc(&c->h_list, n_ids * sizeof(int2), cudaHostAllocDefault) == cudaSuccess;
    for (auto& e : c->ev) ok = ok && cudaEventCreate(&e) == cudaSuccess;
    ok = ok && cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking) == cudaSuccess;
    {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
        int can64 = 0;
        // attribute 122 of the driver's numbering (the runtime's enum does not name it): 64-bit stream memory operations
        if (cudaGetDriverEntryPoint("cuStreamWaitValue64", &fn, cudaEnableDefault, &found) == cudaSuccess &&
            found == cudaDriverEntryPointSuccess &&
            cudaDeviceGetAttribute(&can64, static_cast<cudaDeviceAttr>(CU_DEVICE_ATTRIBUTE_CAN_USE_64_BIT_STREAM_MEM_OPS),
                                   cfg->device) == cudaSuccess && can64)
            c->wait_value64 = reinterpret_cast<CUresult (*)(CUstream, CUdeviceptr, cuuint64_t, unsigned int)>(fn);
        else
            cudaGetLastError();
    }
    ok = ok && cudaEventCreateWithFlags(&c->ev_outputs_ready, cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->ev_outputs_copied, cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->ev_ids_ready, cudaEventDisableTiming) == cudaSuccess;
    if (!ok) { cudaGetLastError(); free_all(c); delete c; return AVSG_ENOMEM; }
    {
        // [0] Stage One first start, [1] its last end; Stage Two: [2] first start, [3] last end, [4] first copy loop,
        // [5] first row in, [6] first block done; minima start at "never", maxima at 0
        const unsigned long long never = ~0ull;
        const unsigned long long init[16] = {never, 0, never, 0, never, never, never, 0, never, 0, never, 0, never, never, never, 0};
        c->d_trange_init = c->d_trange + 8;
        if (cudaMemcpy(c->d_trange, init, sizeof(init), cudaMemcpyHostToDevice) != cudaSuccess ||
            cudaMemset(c->d_shared, 0, STEP_MAX_TABLES * sizeof(SharedRows)) != cudaSuccess ||
            cudaMemset(c->d_flags, 0, FLAG_BYTES) != cudaSuccess ||
            cudaMemset(c->d_sync, 0, 8 * sizeof(unsigned long long)) != cudaSuccess) {
            free_all(c); delete c; return AVSG_ECUDA;
        }
    }
    if (cudaMemset(c->d_status, 0, 256) != cudaSuccess || cudaMemset(c->d_seg, 0, T * sizeof(SegDesc)) != cudaSuccess ||
        init_tables(c, 0, (uint32_t)T) != AVSG_OK || cudaDeviceSynchronize() != cudaSuccess) {
        free_all(c); delete c; return AVSG_ECUDA;
    }
    *out = c;
    return AVSG_OK;
}

int avsg_destroy(avsg_ctx* c)
{
    if (!c) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    cudaDeviceSynchronize();
    free_all(c);
    delete c;
    return AVSG_OK;
}

int avsg_reset(avsg_ctx* c, const uint32_t* table_ids, uint32_t n)
{
    if (!c || (!table_ids && n)) return AVSG_EINVAL;
    for (uint32_t i = 0; i < n; ++i) if (table_ids[i] >= c->cfg.num_tables) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    for (uint32_t i = 0; i < n; ++i) {
        int rc = init_tables(c, table_ids[i], 1);
        if (rc != AVSG_OK) return rc;
        c->kv_host[table_ids[i]] = 0; c->kv_dev[table_ids[i]] = 0;
    }
    CU(cudaDeviceSynchronize());
    return AVSG_OK;
}

int avsg_reset_async(avsg_ctx* c, const uint32_t* table_ids, uint32_t n, void* cuda_stream)
{
    if (!c || (!table_ids && n)) return AVSG_EINVAL;
    for (uint32_t i = 0; i < n; ++i) if (table_ids[i] >= c->cfg.num_tables) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    for (uint32_t first = 0; first < n; first += S1_MAX_TABLES) {
        const uint32_t cnt = n - first < (uint32_t)S1_MAX_TABLES ? n - first : (uint32_t)S1_MAX_TABLES;
        ResetParams p;
        p.tok = c->d_tok; p.life = c->d_life; p.buffer = c->d_buffer; p.stats = c->d_stats; p.qword = c->d_q;
        p.S = c->cfg.buffer_slots; p.row_bytes = c->cfg.row_bytes;
        for (uint32_t i = 0; i < cnt; ++i) {
            p.table_id[i] = table_ids[first + i];
            c->kv_host[p.table_id[i]] = 0; c->kv_dev[p.table_id[i]] = 0;      // the next request brings its own host KV
        }
        CU(launch_reset_tables(p, cnt, (uint32_t)c->sm_count, static_cast<cudaStream_t>(cuda_stream)));
    }
    return AVSG_OK;
}

int avsg_step(avsg_ctx* c, const avsg_step_args* a, void* stream)
{
    return step_impl(c, a, static_cast<cudaStream_t>(stream), false);
}

int avsg_step_host(avsg_ctx* c, const avsg_step_args* a, void* stream)
{
    return step_impl(c, a, static_cast<cudaStream_t>(stream), true);
}

int avsg_buffer(avsg_ctx* c, uint32_t table_id, void** d_rows)
{
    if (!c || !d_rows || table_id >= c->cfg.num_tables) return AVSG_EINVAL;
    *d_rows = c->d_buffer + (size_t)table_id * c->cfg.buffer_slots * c->cfg.row_bytes;
    return AVSG_OK;
}

int avsg_stats(avsg_ctx* c, avsg_stats_t* out)
{
    if (!c || !out) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    std::vector<TableStats> h(c->cfg.num_tables);
    CU(cudaMemcpy(h.data(), c->d_stats, h.size() * sizeof(TableStats), cudaMemcpyDeviceToHost));
    memset(out, 0, sizeof(*out));
    for (const TableStats& t : h) {
        out->steps += t.steps; out->tokens += t.tokens; out->hits += t.hits; out->misses += t.misses;
        out->rows_copied += t.rows; out->extra_decays += t.extra_decays;
    }
    out->bytes_copied = out->rows_copied * c->cfg.row_bytes;
    if (c->timing && c->events_recorded) {
        float a = 0.f, b = 0.f;
        if (cudaEventElapsedTime(&a, c->ev[0], c->ev[1]) == cudaSuccess) out->last_stage_one_us = a * 1000.f;
        if (cudaEventElapsedTime(&b, c->ev[1], c->ev[2]) == cudaSuccess) out->last_transfer_us = b * 1000.f;
        cudaGetLastError();
        unsigned long long r[8];
        CU(cudaMemcpy(r, c->d_trange, sizeof(r), cudaMemcpyDeviceToHost));
        if (r[1] > r[0]) out->last_stage_one_kernel_us = (float)(r[1] - r[0]) * 1e-3f;
        if (r[3] > r[2]) out->last_transfer_kernel_us = (float)(r[3] - r[2]) * 1e-3f;
        if (r[3] > r[2] && r[1] > r[0] && r[2] >= r[0]) out->last_transfer_start_us = (float)(r[2] - r[0]) * 1e-3f;
        const unsigned long long never = ~0ull;
        if (r[1] > r[0] && r[3] > r[2]) {                 // the other marks, all measured from Stage One's first start
            if (r[4] != never && r[4] >= r[0]) out->last_copy_start_us = (float)(r[4] - r[0]) * 1e-3f;
            if (r[5] != never && r[5] >= r[0]) out->last_first_row_us = (float)(r[5] - r[0]) * 1e-3f;
            if (r[6] != never && r[6] >= r[0]) out->last_first_block_done_us = (float)(r[6] - r[0]) * 1e-3f;
            if (r[3] >= r[0]) out->last_call_kernel_us = (float)((r[3] > r[1] ? r[3] : r[1]) - r[0]) * 1e-3f;
        }
    }
    out->last_rows = out->rows_copied - c->last_rows;
    c->last_rows = out->rows_copied;
    return read_status(c, nullptr);
}

int avsg_table_stats(avsg_ctx* c, uint32_t table_id, avsg_stats_t* out)
{
    if (!c || !out || table_id >= c->cfg.num_tables) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    TableStats t;
    CU(cudaMemcpy(&t, c->d_stats + table_id, sizeof(t), cudaMemcpyDeviceToHost));
    memset(out, 0, sizeof(*out));
    out->steps = t.steps; out->tokens = t.tokens; out->hits = t.hits; out->misses = t.misses;
    out->rows_copied = t.rows; out->extra_decays = t.extra_decays;
    out->bytes_copied = out->rows_copied * c->cfg.row_bytes;
    return read_status(c, nullptr);
}

int avsg_sync_status(avsg_ctx* c, uint32_t* status_word)
{
    if (!c) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    return read_status(c, status_word);
}

int avsg_clear_status(avsg_ctx* c)
{
    if (!c) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    CU(cudaMemset(c->d_status, 0, sizeof(uint32_t)));
    // (every call takes its hand-over flags down itself; the arrival counter wraps to zero by itself, and a
    // table closes the rows that it shares, unless a grid was lost half way)
    CU(cudaMemset(c->d_sync + 3, 0, sizeof(unsigned long long)));
    CU(cudaMemset(c->d_shared, 0, STEP_MAX_TABLES * sizeof(SharedRows)));
    c->host_status = 0;
    return AVSG_OK;
}

int avsg_probe_wait_limit(avsg_ctx* c, void* cuda_stream)
{
    if (!c) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    XferOverlapParams x;
    overlap_params(c, x, 1, 1, 1);
    x.table_id[0] = 0; x.kv_base[0] = 0; x.kv_stride[0] = 0;
    x.flags = c->d_flags + (size_t)OVERLAP_MAX_TABLES * OVERLAP_MAX_TOKENS;      // never raised: the wait must run out
    CU(launch_transfer_overlap(x, c->xfer_blocks ? c->xfer_blocks : (uint32_t)c->sm_count, c->xfer_threads,
                               static_cast<cudaStream_t>(cuda_stream)));
    return AVSG_OK;
}

int avsg_export_state(avsg_ctx* c, uint32_t table_id, int32_t* tok, int8_t* life)
{
    if (!c || !tok || !life || table_id >= c->cfg.num_tables) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    const size_t S = c->cfg.buffer_slots;
    CU(cudaDeviceSynchronize());
    CU(cudaMemcpy(tok, c->d_tok + table_id * S, S * sizeof(int32_t), cudaMemcpyDeviceToHost));
    CU(cudaMemcpy(life, c->d_life + table_id * S, S, cudaMemcpyDeviceToHost));
    return read_status(c, nullptr);
}

int avsg_import_state(avsg_ctx* c, uint32_t table_id, const int32_t* tok, const int8_t* life)
{
    if (!c || !tok || !life || table_id >= c->cfg.num_tables) return AVSG_EINVAL;
    const size_t S = c->cfg.buffer_slots;
    for (size_t j = 0; j < S; ++j)
        if (life[j] < -1 || life[j] > c->cfg.max_lifetime || tok[j] < -1) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    CU(cudaMemcpy(c->d_tok + table_id * S, tok, S * sizeof(int32_t), cudaMemcpyHostToDevice));
    CU(cudaMemcpy(c->d_life + table_id * S, life, S, cudaMemcpyHostToDevice));
    if (c->d_q) {                                           // ids and lifetimes kept, every mapping invalid
        std::vector<uint32_t> q(S);
        for (size_t j = 0; j < S; ++j) q[j] = ((uint32_t)(uint8_t)life[j] << 24) | 0x00800000u;
        CU(cudaMemcpy(c->d_q + table_id * S, q.data(), S * sizeof(uint32_t), cudaMemcpyHostToDevice));
    }
    return AVSG_OK;
}

int avsg_export_hash_state(avsg_ctx* c, uint32_t table_id, int32_t* cc, uint32_t* q)
{
    if (!c || !cc || !q || table_id >= c->cfg.num_tables || !c->d_q) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    const size_t S = c->cfg.buffer_slots;
    CU(cudaDeviceSynchronize());
    CU(cudaMemcpy(cc, c->d_tok + table_id * S, S * sizeof(int32_t), cudaMemcpyDeviceToHost));
    CU(cudaMemcpy(q, c->d_q + table_id * S, S * sizeof(uint32_t), cudaMemcpyDeviceToHost));
    return read_status(c, nullptr);
}

int avsg_import_hash_state(avsg_ctx* c, uint32_t table_id, const int32_t* cc, const uint32_t* q)
{
    if (!c || !cc || !q || table_id >= c->cfg.num_tables || !c->d_q) return AVSG_EINVAL;
    const size_t S = c->cfg.buffer_slots;
    std::vector<int8_t> life(S);
    for (size_t j = 0; j < S; ++j) {
        life[j] = (int8_t)(q[j] >> 24);
        if (life[j] < -1 || life[j] > c->cfg.max_lifetime || cc[j] < -1) return AVSG_EINVAL;
    }
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    CU(cudaDeviceSynchronize());
    CU(cudaMemcpy(c->d_tok + table_id * S, cc, S * sizeof(int32_t), cudaMemcpyHostToDevice));
    CU(cudaMemcpy(c->d_q + table_id * S, q, S * sizeof(uint32_t), cudaMemcpyHostToDevice));
    CU(cudaMemcpy(c->d_life + table_id * S, life.data(), S, cudaMemcpyHostToDevice));
    return AVSG_OK;
}

int avsg_save_state(avsg_ctx* c, void* stream)
{
    if (!c) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    const size_t n = (size_t)c->cfg.num_tables * c->cfg.buffer_slots;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CU(cudaMemcpyAsync(c->d_tok_snap, c->d_tok, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    CU(cudaMemcpyAsync(c->d_life_snap, c->d_life, n, cudaMemcpyDeviceToDevice, s));
    if (c->d_q) CU(cudaMemcpyAsync(c->d_q_snap, c->d_q, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    return AVSG_OK;
}

int avsg_restore_state(avsg_ctx* c, void* stream)
{
    if (!c) return AVSG_EINVAL;
    DeviceGuard guard(c->cfg.device);
    if (!guard.ok) return AVSG_ECUDA;
    const size_t n = (size_t)c->cfg.num_tables * c->cfg.buffer_slots;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    CU(cudaMemcpyAsync(c->d_tok, c->d_tok_snap, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    CU(cudaMemcpyAsync(c->d_life, c->d_life_snap, n, cudaMemcpyDeviceToDevice, s));
    if (c->d_q) CU(cudaMemcpyAsync(c->d_q, c->d_q_snap, n * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
    return AVSG_OK;
}

int avsg_set_transfer_mode(avsg_ctx* c, uint32_t mode)
{
    if (!c || mode > AVSG_XFER_SM_OVERLAP) return AVSG_EINVAL;
    c->cfg.transfer_mode = mode;
    return AVSG_OK;
}

int avsg_set_timing(avsg_ctx* c, int enable)
{
    if (!c) return AVSG_EINVAL;
    c->timing = enable != 0;
    c->events_recorded = false;
    return AVSG_OK;
}

int avsg_set_transfer_geometry(avsg_ctx* c, uint32_t blocks, uint32_t threads)
{
    if (!c || threads < 32 || threads > 1024 || threads % 32 || blocks > 65535) return AVSG_EINVAL;
    c->xfer_blocks = blocks;
    c->xfer_threads = threads;
    c->geometry_set = blocks != 0 || threads != XFER_THREADS;
    return AVSG_OK;
}

const char* avsg_strerror(int code)
{
    switch (code) {
        case AVSG_OK: return "ok";
        case AVSG_EINVAL: return "invalid argument";
        case AVSG_ENOMEM: return "out of memory";
        case AVSG_ECUDA: return "CUDA runtime error";
        case AVSG_ECAPACITY: return "buffer_slots < n_tokens * topk (capacity bound violated)";
        case AVSG_EDEVICE_STATUS: return "a kernel reported a problem in the device status word";
        case AVSG_EUNSUPPORTED: return "shape not supported by this build";
        default: return "unknown error";
    }
}

}  // extern "C"
