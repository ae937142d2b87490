"""The operator's work in a decode loop: what a serving program has the library do, over the range it is used in.

A pass is one decode iteration of one layer: one call for all requests of the batch, through the entry point that the
case names.  The selections follow a cyclic trace per request, so that passes can be repeated without end at a steady
hit rate; a trace is long enough that a row comes round again only after it has left the buffer.  Sizes are those of
the five configurations of avsg_traces (top-K 256 and 2048 of 8 Ki to 1 Mi context, 1024 and 8192 slots, 656-byte rows,
1 or 2 tokens per iteration, 1 to 64 requests) and of the tests and sweeps around them (1152-byte rows, 16384 slots,
4 tokens, 128 tables in one call, K = 1000).

Keys of a case: entry (step: device tensors, the decode loop's call; graph: the same call captured and replayed;
host: ids and outputs in pinned host memory; noalloc: caller-owned state), tables, topk, slots, tokens, row_bytes,
context (ctx_min below it: log-uniform over the requests), overlap (mean share of a selection that stays from one
token to the next; spread 0: Beta-distributed around it, else uniform per request within overlap +- spread), near
(share of the positions drawn from the `window` most recent ids), index, overlapped (Stage Two while Stage One runs),
shuffled (ids in the order of their scores rather than of their positions), cold (every pass serves requests that are
new to their tables), early (the outputs that let a consumer start on the resident rows).
"""
import math

import numpy as np
import torch

import paper_2609_37538_b200 as avsg

HOST_KV_LIMIT = 11_100_000_000       # host KV bytes of one case: what the largest configurations hold
POOL_CHUNK = 2112 << 20              # the process's pool of host KV grows by this much
MAX_LIFETIME = 16


def _case(name, **kw):
    c = dict(entry="step", tables=1, topk=2048, slots=8192, tokens=2, row_bytes=656, context=131072, ctx_min=0,
             overlap=0.9, spread=0.0, near=0.5, window=4096, index="hash", overlapped=False, shuffled=False, cold=False,
             early=False)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configuration: one short request without token prediction; all latency and launches
        _case("one_short_request", topk=256, slots=1024, tokens=1, context=8192, near=0.0, window=0),
        # one interactive request with token prediction, with the settings avsg_create has by default
        _case("one_request"),
        # the same request in an engine that replays its decode step from a CUDA graph
        _case("one_request_graph", entry="graph", index="direct", overlapped=True),
        # a small batch of an engine that owns all device memory: K not a power of two, ids in score order, bf16 rows
        _case("batch8_noalloc", entry="noalloc", tables=8, topk=1000, slots=4096, tokens=1, row_bytes=1152, context=65536,
              overlap=0.8, shuffled=True),
        # one layer of the batch-32 configuration that the benchmark runs
        _case("batch32", tables=32, index="direct", overlapped=True),
        # the same with the default settings and with ids in score order
        _case("batch32_defaults", tables=32, shuffled=True),
        # the same from and to host memory: a scheduler on the host picks the ids and reads the slot tables
        _case("batch32_host", entry="host", tables=32, index="direct", overlapped=True),
        # long contexts: 16 requests of 1 Mi positions, a fifth of the selection in a small often used range
        _case("long_context16", tables=16, context=1 << 20, near=0.2, window=512, index="direct", overlapped=True),
        # many unequal requests: contexts from 4 Ki to 512 Ki, selections that stay by 50 to 99 %
        _case("unequal64", tables=64, tokens=1, ctx_min=4096, context=524288, overlap=0.745, spread=0.245, near=0.0, window=0,
              index="direct"),
        # requests that come into the batch: after prefill every selected row has to be fetched
        _case("new_requests8", tables=8, cold=True),
        # three predicted tokens need a pool that no single SM holds; attention starts on the resident rows
        _case("four_tokens_pool16k", tables=16, tokens=4, slots=16384, index="direct", overlapped=True, early=True),
        # all layers' tables of a large batch in one call
        _case("one_call128", tables=128, context=32768, index="direct", overlapped=True),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(work(c)["bytes"] for c in listed())
    while True:
        entry = rng.choice(["step", "step", "step", "graph", "host", "noalloc"])
        tokens = rng.choice([1, 1, 2, 2, 2, 3, 4])
        topk = _log_uniform(rng, 64, 4096) if rng.random() < 0.5 else rng.choice([256, 512, 1024, 2048, 2048])
        tables = _log_uniform(rng, 1, 32 if entry == "noalloc" else 128)
        slots = max(256, 1 << (tokens * topk - 1).bit_length()) << rng.choice([0, 1, 1, 2, 2])
        row_bytes = rng.choice([656, 656, 1152, 512, 1024])
        context = _log_uniform(rng, 4096, 1 << 20)
        near = rng.choice([0.0, 0.2, 0.5])
        c = _case(None, entry=entry, tables=tables, topk=topk, slots=slots, tokens=tokens, row_bytes=row_bytes,
                  context=context, ctx_min=rng.choice([0, 0, 4096]), overlap=round(rng.uniform(0.6, 0.97), 3), near=near,
                  window=4096 if near == 0.5 else 512 if near else 0, index=rng.choice(["hash", "direct"]),
                  overlapped=rng.random() < 0.5, shuffled=rng.random() < 0.5, cold=rng.random() < 0.1,
                  early=rng.random() < 0.2)
        if entry == "noalloc":
            c.update(index="hash", overlapped=False, cold=False, early=False)
        elif entry != "step":
            c.update(early=False)
        if entry == "graph":
            c.update(cold=False)
        if (context < c["ctx_min"] or 2 * max(topk, c["window"]) > (c["ctx_min"] or context)
                or slots > (8192 if entry == "noalloc" else 32768)
                or entry == "noalloc" and tables * tokens * topk > avsg.NOALLOC_MAX_IDS
                or tables * tokens * topk > 600_000 or tables * context * row_bytes > HOST_KV_LIMIT
                or work(c)["bytes"] > most):
            continue
        return c


def _expected_misses(c):
    """Rows that a pass has to fetch: selections that changed and went to a position that is not in the buffer (most of
    the near ones are; the traces show within a fifth of this, batch8_noalloc a third more)."""
    far = c["topk"] * (1.0 - c["near"])
    changed = far * (1.0 - c["overlap"])
    if c["cold"]:
        return c["tables"] * (c["topk"] + (c["tokens"] - 1) * c["topk"] * (1.0 - c["overlap"]))
    context = c["context"] if not c["ctx_min"] else math.sqrt(c["ctx_min"] * c["context"])
    missed = changed * max(0.05, 1.0 - min(c["slots"], far * 8) / context)
    return c["tables"] * c["tokens"] * (missed + 0.3 * c["topk"] * c["near"] * (1.0 - c["overlap"]))


def work(case):
    c = case
    ids = c["tables"] * c["tokens"] * c["topk"]
    rows = _expected_misses(c) * c["row_bytes"]
    # rows: read from the host once and written to the device once; per slot an id and a lifetime, in and out;
    # per position the id in, slot and hit flag out
    return {"bytes": 2 * rows + 2 * 5 * c["tables"] * c["slots"] + 9 * ids, "flops": 0}


def tolerance(case):
    return "exact"                   # slot numbers, flags, counts and bytes: there is nothing to round


# ---- host KV: one pool per process, as a serving program keeps it; blocks of it are dealt out to the requests ----------
_pool = []


def _deal_host_kv(sizes, rng):
    """A block of the pool for each of the sizes, laid out in an order that the seed decides.  The pool holds random bytes."""
    at, k, blocks = int(rng.integers(0, 1 << 13)) * 4096, 0, [0] * len(sizes)
    for i in rng.permutation(len(sizes)):
        if at + sizes[i] > POOL_CHUNK:
            at, k = 0, k + 1
        if k == len(_pool):
            chunk = avsg.pinned_empty(POOL_CHUNK, huge_pages=True)
            gen = torch.Generator(device="cuda").manual_seed(k)
            words = torch.randint(-(1 << 62), 1 << 62, (POOL_CHUNK // 8,), dtype=torch.int64, device="cuda", generator=gen)
            torch.from_numpy(chunk.numpy()).copy_(words.view(torch.uint8))
            _pool.append(chunk)
        blocks[i] = _pool[k].data_ptr() + at
        at += -(-sizes[i] // 4096) * 4096
    return blocks


# ---- traces -------------------------------------------------------------------------------------------------------------
def _iterations(c):
    if c["cold"]:
        return 16
    new = c["tokens"] * c["topk"] * (1.0 - c["near"]) * (1.0 - c["overlap"])
    return int(min(max(24, 3 * c["slots"] / new), 192))


def _contexts(c, rng):
    if not c["ctx_min"]:
        return np.full(c["tables"], c["context"], dtype=np.int64)
    return np.exp(rng.uniform(math.log(c["ctx_min"]), math.log(c["context"]), c["tables"])).astype(np.int64)


def _trace(c, contexts, rng, gen):
    """int32 [iterations, tables, tokens, topk] on the device.  Position p of a selection draws its ids from a range of
    its own, keeps its id with the overlap's probability and takes a new one otherwise; after the last iteration the
    first one follows.  Ids are unique within a token and ascend unless `shuffled`."""
    n, K, G = c["tables"], c["topk"], c["tokens"]
    T = _iterations(c)
    R = int(round(K * c["near"]))
    U = K - R
    far = torch.from_numpy(contexts - (c["window"] if R else 0)).cuda().view(n, 1)
    ctx = torch.from_numpy(contexts).cuda().view(n, 1)
    p, q = torch.arange(U + 1, device="cuda").view(1, -1), torch.arange(R + 1, device="cuda").view(1, -1)
    edges = [far * p // U] if U else []
    lo = [e[:, :-1] for e in edges] + ([(far + (ctx - far) * q // R)[:, :-1]] if R else [])
    hi = [e[:, 1:] for e in edges] + ([(far + (ctx - far) * q // R)[:, 1:]] if R else [])
    lo, width = torch.cat(lo, 1), torch.cat(hi, 1) - torch.cat(lo, 1)
    if c["spread"]:
        keep = np.broadcast_to(rng.uniform(c["overlap"] - c["spread"], c["overlap"] + c["spread"], n), (T * G, n))
    else:
        keep = rng.beta(20 * c["overlap"], 20 * (1 - c["overlap"]), (T * G, n))
    keep = torch.from_numpy(np.ascontiguousarray(keep, dtype=np.float32)).cuda()
    out = torch.empty((T * G, n, K), dtype=torch.int32, device="cuda")
    step = torch.arange(T * G, dtype=torch.int32, device="cuda").view(-1, 1)
    for i in range(n):
        new = torch.rand((T * G, K), device="cuda", generator=gen) >= keep[:, i : i + 1]
        last = torch.where(new, step, -1).cummax(0).values
        last = torch.where(last < 0, last[-1:].clamp(min=0), last)
        draws = torch.rand((T * G, K), device="cuda", generator=gen).gather(0, last.long())
        ids = (lo[i] + (draws * width[i]).long().clamp(max=torch.clamp(width[i] - 1, min=0))).int()
        out[:, i] = torch.where(width[i] > 0, ids, -1)
        if c["shuffled"]:
            order = torch.rand((T * G, K), device="cuda", generator=gen).argsort(1)
            out[:, i] = out[:, i].gather(1, order)
    return out.view(T, G, n, K).transpose(1, 2).contiguous()


class _Rows:
    """The tables' buffers, which lie one behind the other, as one array of 8-byte words [tables, slots, words]."""

    def __init__(self, ctx, c):
        base = ctx.buffer(0).data_ptr()
        assert all(ctx.buffer(i).data_ptr() == base + i * c["slots"] * c["row_bytes"] for i in range(c["tables"]))
        self.keep = ctx
        self.__cuda_array_interface__ = {"shape": (c["tables"], c["slots"], c["row_bytes"] // 8), "typestr": "<i8",
                                         "data": (base, False), "version": 3, "strides": None}


def prepare(case, seed):
    c = dict(case)
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    n, G, K, S = c["tables"], c["tokens"], c["topk"], c["slots"]
    contexts = _contexts(c, rng)
    kv = _deal_host_kv([int(x) * c["row_bytes"] for x in contexts], rng)
    trace = _trace(c, contexts, rng, gen)
    verified = [int(x) - (G - 1) for x in contexts]       # the newest positions are speculative
    rows = [int(x) for x in contexts]
    host = c["entry"] == "host"
    s = {"case": c, "at": 0, "verified": verified, "kv": kv, "kv_rows": rows}
    where = dict(pin_memory=True) if host else dict(device="cuda")
    s["slots"] = torch.empty((n, G, K), dtype=torch.int32, **where)
    s["hit"] = torch.empty((n, G, K), dtype=torch.uint8, **where)
    s["miss_count"] = torch.empty((n, G), dtype=torch.int32, **where)
    if host:
        pinned = torch.empty(trace.shape, dtype=torch.int32, pin_memory=True)
        pinned.copy_(trace)
        trace = pinned
    s["trace"] = list(trace.unbind(0))
    if c["entry"] == "noalloc":
        s["tok"] = torch.full((n, S), -1, dtype=torch.int32, device="cuda")
        s["life"] = torch.full((n, S), -1, dtype=torch.int8, device="cuda")
        s["buffer"] = torch.zeros((n, S, c["row_bytes"]), dtype=torch.uint8, device="cuda")
        s["rows"] = s["buffer"].view(torch.int64)
        return s
    ctx = avsg.Context(num_tables=n, buffer_slots=S, row_bytes=c["row_bytes"], max_topk=K, max_tokens=G,
                       max_lifetime=MAX_LIFETIME,
                       transfer_mode=avsg.XFER_SM_OVERLAP if c["overlapped"] else avsg.XFER_SM_BALANCED,
                       index_mode=avsg.INDEX_DIRECT if c["index"] == "direct" else avsg.INDEX_HASH,
                       max_context=int(contexts.max()))
    s["ctx"] = ctx
    s["rows"] = torch.as_tensor(_Rows(ctx, c), device="cuda")
    s["tables"] = list(range(n))
    s["call"] = ctx.prepare(s["tables"], kv, G, K, kv_rows=rows)
    if c["early"]:
        s["done"] = torch.zeros(1, dtype=torch.int64, device="cuda")
        s["arriving"] = torch.empty((n, G, K), dtype=torch.uint8, device="cuda")
    if c["entry"] == "graph":
        s["ids"] = torch.empty((n, G, K), dtype=torch.int32, device="cuda")
        s["verified_dev"] = torch.tensor(verified, dtype=torch.int32, device="cuda")
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["call"].run(s["ids"], s["verified_dev"], s["slots"], s["hit"], s["miss_count"])
    return s


def run(state):
    s = state
    c = s["case"]
    ids = s["trace"][s["at"] % len(s["trace"])]
    s["at"] += 1
    out = [s["slots"], s["hit"], s["miss_count"], s["rows"]]
    if c["entry"] == "noalloc":
        avsg.step_noalloc(s["tok"], s["life"], s["buffer"], ids, s["kv"], s["verified"], max_lifetime=MAX_LIFETIME,
                          slots=s["slots"], hit=s["hit"], miss_count=s["miss_count"], kv_rows=s["kv_rows"])
        return out + [s["tok"], s["life"]]
    if c["entry"] == "graph":
        s["ids"].copy_(ids)
        s["graph"].replay()
        return out
    if c["cold"]:
        s["ctx"].reset_async(s["tables"])
    if c["early"]:
        s["call"].run(ids, s["verified"], s["slots"], s["hit"], s["miss_count"],
                      stage_one_done=(s["done"], s["at"]), arriving=s["arriving"])
        return out + [s["done"], s["arriving"]]
    s["call"].run(ids, s["verified"], s["slots"], s["hit"], s["miss_count"], host=c["entry"] == "host")
    return out
