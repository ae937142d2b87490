"""Calls with host buffers: page-locked ones that the kernels use in place, pageable and oddly placed ones, and calls that
queue behind one another with ids written just before each of them; compared with the oracle (nothing to tolerate)."""
import numpy as np
import pytest

import avsg_traces as tr
from oracle import OracleTable

pytestmark = pytest.mark.gpu


def _setup(avsg, n, n_q, K, S, rb, ctxlen, mode, T, cluster=0):
    traces = [tr.generate(tr.TraceConfig(seed=71, table=i, topk=K, n_q=n_q, n_iters=T, context=ctxlen, ctx_growth=n_q > 1,
                                         beta=(9, 1), p_recent=0.5, recent_window=512))
              for i in range(n)]
    kv = avsg.pinned_empty(ctxlen * rb)
    tr.fill_kv(kv.data_ptr(), 71, 0, ctxlen, rb)
    ctx = avsg.Context(n, S, rb, K, n_q, 16, transfer_mode=getattr(avsg, mode), stage_one_cluster=cluster)
    return traces, kv, ctx, [OracleTable(S, rb, 16) for _ in range(n)]


# outputs of 1, 2 and 3 x 16 bytes and of no multiple of 4; buffers at odd places; rounds; the two-launch balanced mode
@pytest.mark.parametrize("mode", ["XFER_SM_BALANCED", "XFER_SM_OVERLAP"])
@pytest.mark.parametrize("n,n_q,K,kind", [(1, 1, 1, "pinned"), (3, 2, 37, "pinned"), (3, 2, 37, "odd"), (2, 2, 64, "pageable"),
                                          (2, 2, 64, "pageable ids"), (76, 2, 33, "pinned"), (130, 1, 16, "odd")])
def test_kinds_of_host_buffers(mode, n, n_q, K, kind):
    import torch
    import paper_2609_37538_b200 as avsg
    T, S, rb, ctxlen = 6, 256, 48, 4000
    traces, kv, ctx, orc = _setup(avsg, n, n_q, K, S, rb, ctxlen, mode, T)
    call = ctx.prepare(list(range(n)), [kv] * n, n_q, K)
    lead = 1 if kind == "odd" else 0                     # hit flags one byte, slots and counts one word off 16 bytes
    ids_pinned, out_pinned = not kind.startswith("pageable"), kind != "pageable"
    ids = torch.empty(n * n_q * K + lead, dtype=torch.int32, pin_memory=ids_pinned)[lead:].view(n, n_q, K)
    slots = torch.empty(n * n_q * K + lead, dtype=torch.int32, pin_memory=out_pinned)[lead:].view(n, n_q, K)
    hit = torch.empty(n * n_q * K + lead, dtype=torch.uint8, pin_memory=out_pinned)[lead:].view(n, n_q, K)
    count = torch.empty(n * n_q + lead, dtype=torch.int32, pin_memory=out_pinned)[lead:].view(n, n_q)
    for t in range(T):
        X = np.stack([traces[i][0][t] for i in range(n)])
        N = [int(traces[i][1][t]) for i in range(n)]
        ids.copy_(torch.from_numpy(X))
        slots.fill_(-7); hit.fill_(9); count.fill_(-7)
        with_all = t % 3 != 2                            # every third call asks for the slots alone
        call.run(ids, N, slots, hit if with_all else None, count if with_all else None, host=True)
        torch.cuda.synchronize()
        for i in range(n):
            r = orc[i].step(X[i], N[i], kv.numpy(), rb)
            assert (slots[i].numpy() == r.O).all(), (t, i)
            if with_all:
                assert (hit[i].numpy() == r.M).all() and (count[i].numpy() == r.n).all(), (t, i)
            else:
                assert (hit[i].numpy() == 9).all() and (count[i].numpy() == -7).all(), (t, i)
    for i in range(0, n, max(1, n // 5)):
        assert (ctx.buffer(i).cpu().numpy() == orc[i].rows()).all(), i
    assert ctx.sync_status() == 0


@pytest.mark.parametrize("mode", ["XFER_SM_BALANCED", "XFER_SM_OVERLAP"])
@pytest.mark.parametrize("cluster", [0, 2])
def test_calls_that_queue_behind_one_another(mode, cluster):
    """Nothing waits between the calls; every second one has device buffers, and one has pageable ids."""
    import torch
    import paper_2609_37538_b200 as avsg
    n, n_q, K, S, rb, ctxlen, T = 5, 2, 256, 1024, 656, 20000, 24
    traces, kv, ctx, orc = _setup(avsg, n, n_q, K, S, rb, ctxlen, mode, T, cluster)
    call = ctx.prepare(list(range(n)), [kv] * n, n_q, K)
    outs, ids, dev_ids = [], [], []
    for t in range(T):
        X = torch.from_numpy(np.stack([traces[i][0][t] for i in range(n)]))
        ids.append(torch.full((n, n_q, K), -1, dtype=torch.int32) if t == 9 else
                   torch.full((n, n_q, K), -1, dtype=torch.int32, pin_memory=True))
        where = dict(pin_memory=True) if t % 2 else dict(device="cuda")
        outs.append((torch.empty((n, n_q, K), dtype=torch.int32, **where), torch.empty((n, n_q, K), dtype=torch.uint8, **where),
                     torch.empty((n, n_q), dtype=torch.int32, **where)))
        dev_ids.append(X.cuda())
    torch.cuda.synchronize()
    for t in range(T):
        N = [int(traces[i][1][t]) for i in range(n)]
        if t % 2:
            ids[t].copy_(dev_ids[t].cpu() if t % 4 == 1 else torch.from_numpy(np.stack([traces[i][0][t] for i in range(n)])))
        call.run(ids[t] if t % 2 else dev_ids[t], N, *outs[t], host=bool(t % 2))
    torch.cuda.synchronize()
    for t in range(T):
        for i in range(n):
            r = orc[i].step(traces[i][0][t], int(traces[i][1][t]), kv.numpy(), rb)
            assert (outs[t][0][i].cpu().numpy() == r.O).all() and (outs[t][1][i].cpu().numpy() == r.M).all(), (t, i)
            assert (outs[t][2][i].cpu().numpy() == r.n).all(), (t, i)
    for i in range(n):
        assert (ctx.buffer(i).cpu().numpy() == orc[i].rows()).all(), i
    assert ctx.sync_status() == 0


@pytest.mark.parametrize("mode", ["XFER_SM_BALANCED", "XFER_SM_OVERLAP"])
@pytest.mark.parametrize("n", [2, 76])
@pytest.mark.parametrize("ids_at,slots_at,hit_at,count_at", [(1, 0, 0, 0), (2, 6, 1, 2), (3, 4, 3, 1), (0, 1, 5, 3), (4, 3, 2, 0)])
def test_buffers_off_the_boundary_of_a_word(mode, n, ids_at, slots_at, hit_at, count_at):
    """Pinned buffers that begin at any byte of a message, as host-side packing may leave them."""
    import torch
    import paper_2609_37538_b200 as avsg
    T, S, rb, ctxlen, n_q, K = 4, 256, 48, 4000, 2, 32
    traces, kv, ctx, orc = _setup(avsg, n, n_q, K, S, rb, ctxlen, mode, T)
    call = ctx.prepare(list(range(n)), [kv] * n, n_q, K)

    def place(at, dtype, *shape):
        whole = torch.full((at + int(np.prod(shape)) * np.dtype(dtype).itemsize + 8,), 0x5A, dtype=torch.uint8, pin_memory=True)
        return whole, np.ndarray(shape, dtype, buffer=whole.numpy(), offset=at)

    bufs = [place(ids_at, np.int32, n, n_q, K), place(slots_at, np.int32, n, n_q, K), place(hit_at, np.uint8, n, n_q, K),
            place(count_at, np.int32, n, n_q)]
    ids, slots, hit, count = [view for _, view in bufs]
    for t in range(T):
        X = np.stack([traces[i][0][t] for i in range(n)])
        N = [int(traces[i][1][t]) for i in range(n)]
        ids[:] = X
        call.run(*[x if isinstance(x, list) else x.ctypes.data for x in (ids, N, slots, hit, count)], host=True)
        torch.cuda.synchronize()
        for i in range(n):
            r = orc[i].step(X[i], N[i], kv.numpy(), rb)
            assert (slots[i] == r.O).all() and (hit[i] == r.M).all() and (count[i] == r.n).all(), (t, i)
    for whole, view in bufs:                             # nothing beside them was written
        at = view.ctypes.data - whole.data_ptr()
        assert (whole[:at] == 0x5A).all() and (whole[at + view.nbytes :] == 0x5A).all()
    assert ctx.sync_status() == 0


def test_many_ids_off_the_link_s_units_go_by_copy():
    """Where more than 16384 ids begin decides the route."""
    import torch
    import paper_2609_37538_b200 as avsg
    n, n_q, ctxlen, rb = 12, 2, 4000, 48
    for K, offsets in ((704, (0, 1, 8, 4, 24, 7)), (700, (0, 8)), (682, (0, 1))):          # (in ids; the last has 16368)
        traces, kv, ctx, orc = _setup(avsg, n, n_q, K, 2048, rb, ctxlen, "XFER_SM_BALANCED", len(offsets))
        whole = torch.full((n * n_q * K + 32,), -1, dtype=torch.int32, pin_memory=True)
        base = -whole.data_ptr() % 64 // 4
        slots = torch.empty((n, n_q, K), dtype=torch.int32, pin_memory=True)
        for t, off in enumerate(offsets):
            ids = whole[base + off : base + off + n * n_q * K].view(n, n_q, K)
            ids.copy_(torch.from_numpy(np.stack([traces[i][0][t] for i in range(n)])))
            N = [int(traces[i][1][t]) for i in range(n)]
            with torch.autograd.profiler.profile(use_device="cuda") as seen:
                ctx.prepare(list(range(n)), [kv] * n, n_q, K).run(ids, N, slots, host=True)
                torch.cuda.synchronize()
            copies = sum("Memcpy" in e.name for e in seen.function_events)
            for i in range(n):
                assert (slots[i].numpy() == orc[i].step(traces[i][0][t], N[i], kv.numpy(), rb).O).all(), (K, t, i)
            assert (copies > 0) == (K == 700 or (K == 704 and off % 8 != 0)), (K, off, copies)
        assert ctx.sync_status() == 0
