"""Stage One at the sizes where its split of slots and ids over threads changes, with ids that
share one chain of its index, and with states only a caller's own table can have; compared with the oracle after every
call (whole numbers: nothing to tolerate)."""
import numpy as np
import pytest

import avsg_traces as tr
from oracle import OracleTable

pytestmark = pytest.mark.gpu
RB, CTX = 32, 60000


def _same_bucket_ids(S, n, bucket):
    """n ids whose multiplicative hash falls into one of the 2 S buckets."""
    x = np.arange(1 << 22, dtype=np.uint64)
    h = ((x * 2654435769) & 0xFFFFFFFF) >> np.uint64(32 - int(2 * S).bit_length() + 1)
    return x[h == bucket][:n].astype(np.int32)


# S below four warps' slots; K around S / 4 (the number of threads changes); one and two ids per thread and more;
# K = S; the smallest K; as many nodes as fit one SM (N_q K = S)
@pytest.mark.parametrize("S,K,n_q", [(32, 32, 1), (32, 1, 8), (64, 31, 2), (256, 64, 4), (256, 65, 3), (1024, 256, 2),
                                     (1024, 257, 3), (2048, 2048, 1), (4096, 1024, 4), (4096, 1025, 3), (8192, 1, 8),
                                     (8192, 2047, 4), (8192, 2049, 3), (8192, 4097, 1), (8192, 1024, 8)])
def test_splits_of_slots_and_ids(S, K, n_q):
    _steps(S, K, n_q, 0, 3)


# a cluster's blocks with fewer slots than threads, with words of positions that no block or only some warps have, with
# several passes over the positions, with more ids coming in than a block has slots; L = 1: the shortest decay search
@pytest.mark.parametrize("S,K,n_q,C,L", [(256, 256, 1, 8, 3), (256, 31, 8, 8, 1), (512, 170, 3, 4, 2), (2048, 1025, 1, 2, 126),
                                         (4096, 1024, 4, 4, 1), (16384, 2047, 8, 0, 3), (16384, 5000, 3, 4, 5),
                                         (32768, 4097, 2, 8, 30)])
def test_splits_over_a_cluster(S, K, n_q, C, L):
    _steps(S, K, n_q, C, L)


def _steps(S, K, n_q, cluster, L):
    import torch
    import paper_2609_37538_b200 as avsg
    T, n = 6, 2
    rng = np.random.default_rng([S, K, n_q])
    kv = avsg.pinned_empty(CTX * RB)
    tr.fill_kv(kv.data_ptr(), 1, 0, CTX, RB)
    ctx = avsg.Context(n, S, RB, K, n_q, L, stage_one_cluster=cluster)
    orc = [OracleTable(S, RB, L) for _ in range(n)]
    for t in range(T):
        span = min(CTX, 3 * S // 2 + K)               # a good share of the ids comes back
        X = np.stack([[rng.choice(span, K, replace=False) for _ in range(n_q)] for _ in range(n)]).astype(np.int32)
        X[:, :, K // 2] = -1                          # padding in the middle
        N = [span - 7 * t for _ in range(n)]          # shrinks: resident ids become unverified
        ctx.set_transfer_mode(avsg.XFER_SM_OVERLAP if t % 2 else avsg.XFER_SM_BALANCED)
        out = ctx.step(list(range(n)), torch.from_numpy(X).cuda(), [kv] * n, N)
        slots, hit, mc = out.slots.cpu().numpy(), out.hit.cpu().numpy(), out.miss_count.cpu().numpy()
        for i in range(n):
            r = orc[i].step(X[i], N[i], kv.numpy(), RB)
            assert (slots[i] == r.O).all() and (hit[i] == r.M).all() and (mc[i] == r.n).all(), (t, i)
            tok, life = ctx.export_state(i)
            c, l = orc[i].export_state()
            assert (tok == c).all() and (life == l).all(), (t, i)
            assert (ctx.buffer(i).cpu().numpy() == orc[i].rows()).all(), (t, i)
            ts, oc = ctx.table_stats(i), orc[i].counters()
            assert all(ts[k] == oc[k] for k in ("hits", "misses", "rows_copied", "extra_decays")), (t, i)
    assert ctx.sync_status() == 0


@pytest.mark.parametrize("S", [128, 16384])
def test_ids_of_one_chain(S):
    """Every id hashes to the same bucket: one chain holds all of them, the table's and those that come in.  (The packed index of 16384
    slots has up to 2 S chains; ids of the first one of so many are of the first one with fewer too.)"""
    import torch
    import paper_2609_37538_b200 as avsg
    K, n_q, L = 32, 4, 4
    ids = _same_bucket_ids(S, 256, 77 if S == 128 else 0)
    assert len(ids) >= 100
    rows = int(ids.max()) + 1
    kv = avsg.pinned_empty(rows * 16)
    kv.numpy()[:] = np.random.default_rng(5).integers(0, 256, rows * 16, dtype=np.uint8)
    ctx, orc = avsg.Context(1, S, 16, K, n_q, L), OracleTable(S, 16, L)
    rng = np.random.default_rng(6)
    for t in range(12):
        X = np.stack([rng.choice(ids, K, replace=False) for _ in range(n_q)])
        out = ctx.step([0], torch.from_numpy(X[None]).cuda(), [kv], [rows])
        r = orc.step(X, rows, kv.numpy(), 16)
        assert (out.slots.cpu().numpy()[0] == r.O).all() and (out.hit.cpu().numpy()[0] == r.M).all(), t
    assert (ctx.buffer(0).cpu().numpy() == orc.rows()).all() and ctx.sync_status() == 0


def test_lifetimes_above_the_maximum():
    """Caller-owned state from a longer maximum lifetime: slots reserved early in a call are reclaimed later in it, and
    an id that was reserved and lost within the call is missed again."""
    import torch
    import paper_2609_37538_b200 as avsg
    S, K, n_q, L = 64, 16, 4, 3
    kv = avsg.pinned_empty(4000 * RB)
    tr.fill_kv(kv.data_ptr(), 3, 0, 4000, RB)
    rng = np.random.default_rng(9)
    tok = np.full(S, -1, np.int32)
    life = np.full(S, -1, np.int8)
    tok[::2], life[::2] = np.arange(1000, 1000 + S // 2), 90          # half of the table outlives the call
    orc = OracleTable(S, RB, L)
    orc.import_state(tok, life)
    d = dict(device="cuda")
    tok_d, life_d = torch.from_numpy(tok[None]).to(**d), torch.from_numpy(life[None]).to(**d)
    buf, status = torch.zeros((1, S, RB), dtype=torch.uint8, **d), torch.zeros(1, dtype=torch.int32, **d)
    slots, hit = torch.empty((1, n_q, K), dtype=torch.int32, **d), torch.empty((1, n_q, K), dtype=torch.uint8, **d)
    for t in range(4):
        X = np.stack([rng.choice(70, K, replace=False) for _ in range(n_q)]).astype(np.int32)
        avsg.step_noalloc(tok_d, life_d, buf, torch.from_numpy(X[None]).cuda(), [kv], [4000], max_lifetime=L, slots=slots,
                          hit=hit, status=status)
        r = orc.step(X, 4000, kv.numpy(), RB)
        c, l = orc.export_state()
        assert (slots[0].cpu().numpy() == r.O).all() and (hit[0].cpu().numpy() == r.M).all(), t
        assert (tok_d[0].cpu().numpy() == c).all() and (life_d[0].cpu().numpy() == l).all(), t
        assert int(status.item()) == 0


# clusters of eight and four blocks, and two kernels (state off its alignment); the small sizes of the test above too; rows that
# are asked for early and rows that are too long for that
@pytest.mark.parametrize("n,S,K,n_q,rb", [(2, 64, 16, 4, 64), (1, 4096, 2048, 2, 64), (9, 4096, 2048, 2, 64), (32, 4096, 2048, 2, 64), (3, 8192, 1000, 8, 64),
                                          (2, 64, 16, 4, 1552), (1, 4096, 2047, 2, 1552), (10, 4096, 1365, 3, 1552)])
@pytest.mark.parametrize("aligned", [True, False])
def test_the_last_reservation_of_a_slot_has_its_row(n, S, K, n_q, rb, aligned):
    """Lifetimes above the maximum: a slot that two tokens of a call reserve holds the row of the later one."""
    import torch
    import paper_2609_37538_b200 as avsg
    L, context, calls = 3, 16384, 3
    kv = avsg.pinned_empty(context * rb)
    tr.fill_kv(kv.data_ptr(), 3, 0, context, rb)
    rng = np.random.default_rng([n, S, K])
    d = dict(device="cuda")
    tok_d, life_d = (torch.empty(n * S + 1, dtype=t, **d)[0 if aligned else 1 :][: n * S].view(n, S) for t in (torch.int32, torch.int8))
    buf, status = torch.zeros((n, S, rb), dtype=torch.uint8, **d), torch.zeros(1, dtype=torch.int32, **d)
    slots, hit = torch.empty((n, n_q, K), dtype=torch.int32, **d), torch.empty((n, n_q, K), dtype=torch.uint8, **d)
    orc = [OracleTable(S, rb, L) for _ in range(n)]
    twice = 0
    for c in range(calls):
        tok, life = np.full(S, -1, np.int32), np.full(S, -1, np.int8)
        tok[::2], life[::2] = context - 1 - np.arange(S // 2), 90        # half of the table outlives the call
        for o in orc:
            o.import_state(tok, life)
        tok_d.copy_(torch.from_numpy(tok).expand(n, S)); life_d.copy_(torch.from_numpy(life).expand(n, S))
        X = np.stack([rng.permutation(context - S)[: n_q * K].reshape(n_q, K) for _ in range(n)]).astype(np.int32)
        X[:, 1, 0] = -1                                                   # what is reserved again moves by a row
        avsg.step_noalloc(tok_d, life_d, buf, torch.from_numpy(X).cuda(), [kv] * n, [context] * n, max_lifetime=L, slots=slots,
                          hit=hit, status=status)
        assert int(status.item()) == 0
        for i in range(n):
            r = orc[i].step(X[i], context, kv.numpy(), rb)
            o, l = orc[i].export_state()
            assert (slots[i].cpu().numpy() == r.O).all() and (hit[i].cpu().numpy() == r.M).all(), (c, i)
            assert (tok_d[i].cpu().numpy() == o).all() and (life_d[i].cpu().numpy() == l).all(), (c, i)
            got, want = buf[i].cpu().numpy(), orc[i].rows()
            assert (got == want).all(), (c, i, int((got != want).any(axis=1).sum()))
            taken = r.O[r.O >= 0]
            twice += len(taken) - len(np.unique(taken))
    assert twice > 0


# slots per thread of two, four and eight; the last one takes two kernels
@pytest.mark.parametrize("S,K,n_q", [(32, 8, 2), (256, 31, 3), (1024, 300, 2), (2048, 500, 2), (4096, 1000, 3), (8192, 2048, 2),
                                     (256, 2, 70)])
@pytest.mark.parametrize("tok_at,life_at", [(1, 0), (0, 1), (2, 2), (3, 4), (1, 7)])
def test_caller_owned_state_at_any_place(S, K, n_q, tok_at, life_at):
    """State that begins at any id and any lifetime of a larger allocation (a pool that packs tables); what lies before and
    behind it stays as it is."""
    import torch
    import paper_2609_37538_b200 as avsg
    n, L = 2, 3
    rng = np.random.default_rng([S, K, n_q])
    kv = avsg.pinned_empty(CTX * RB)
    tr.fill_kv(kv.data_ptr(), 1, 0, CTX, RB)
    orc = [OracleTable(S, RB, L) for _ in range(n)]
    d = dict(device="cuda")
    toks, lifes = torch.full((n * S + 8,), -77, dtype=torch.int32, **d), torch.full((n * S + 16,), 77, dtype=torch.int8, **d)
    tok, life = toks[tok_at : tok_at + n * S].view(n, S), lifes[life_at : life_at + n * S].view(n, S)
    tok.fill_(-1); life.fill_(-1)
    buf, status = torch.zeros((n, S, RB), dtype=torch.uint8, **d), torch.zeros(1, dtype=torch.int32, **d)
    slots, hit = torch.empty((n, n_q, K), dtype=torch.int32, **d), torch.empty((n, n_q, K), dtype=torch.uint8, **d)
    for t in range(4):
        X = np.stack([[rng.choice(3 * S // 2 + K, K, replace=False) for _ in range(n_q)] for _ in range(n)]).astype(np.int32)
        N = 3 * S // 2 - 7 * t
        avsg.step_noalloc(tok, life, buf, torch.from_numpy(X).cuda(), [kv] * n, [N] * n, max_lifetime=L, slots=slots, hit=hit,
                          status=status)
        assert int(status.item()) == 0
        for i in range(n):
            r = orc[i].step(X[i], N, kv.numpy(), RB)
            c, l = orc[i].export_state()
            assert (slots[i].cpu().numpy() == r.O).all() and (hit[i].cpu().numpy() == r.M).all(), (t, i)
            assert (tok[i].cpu().numpy() == c).all() and (life[i].cpu().numpy() == l).all(), (t, i)
            assert (buf[i].cpu().numpy() == orc[i].rows()).all(), (t, i)
    assert (toks[:tok_at] == -77).all() and (toks[tok_at + n * S :] == -77).all()
    assert (lifes[:life_at] == 77).all() and (lifes[life_at + n * S :] == 77).all()
