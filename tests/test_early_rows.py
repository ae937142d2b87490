"""Rows that are asked for before their slots are known: the split of a token's positions over the copying blocks (groups of 1
to 32 positions, remainders, fewer groups than blocks), rows up to and above what a warp holds, ids that lose their slots to
earlier tokens of the call (S = N_q K), calls whose sets leave no room (nothing is asked for early), ids in host memory;
compared with the oracle (whole numbers and bytes: nothing to tolerate)."""
import numpy as np
import pytest

import avsg_traces as tr
from oracle import OracleTable

pytestmark = pytest.mark.gpu
CTX = 9000


@pytest.mark.parametrize("n,S,K,n_q,rb", [(1, 32, 1, 5, 48), (2, 256, 31, 3, 48), (1, 256, 33, 2, 1536), (2, 512, 64, 8, 1552), (9, 1024, 196, 3, 48),
                                          (3, 1024, 255, 4, 656), (17, 512, 257, 1, 1040), (2, 4096, 1025, 3, 48), (1, 8192, 2047, 4, 512),
                                          (5, 8192, 8192, 1, 48), (46, 8192, 2048, 4, 48), (46, 4096, 130, 31, 48)])
def test_rows_asked_for_early(n, S, K, n_q, rb):
    import torch
    import paper_2609_37538_b200 as avsg
    rng = np.random.default_rng([n, S, K])
    kv = avsg.pinned_empty(CTX * rb)
    tr.fill_kv(kv.data_ptr(), 1, 0, CTX, rb)
    ctx = avsg.Context(n, S, rb, K, n_q, 3)
    orc = [OracleTable(S, rb, 3) for _ in range(n)]
    done = []
    for c in range(5):
        span = CTX if c == 3 else min(CTX, S + K + 64)   # most ids come back, some after they have lost their slots
        X = np.stack([[rng.permutation(span)[:K] for _ in range(n_q)] for _ in range(n)]).astype(np.int32)
        X[:, :, K // 2 : K // 2 + (K > 8)] = -1          # padding in the middle
        ids = torch.from_numpy(X).pin_memory() if c in (1, 3) else torch.from_numpy(X).cuda()
        done.append((X, (ctx.step_host if c in (1, 3) else ctx.step)(list(range(n)), ids, [kv] * n, [CTX - 10] * n)))
    torch.cuda.synchronize()
    for c, (X, out) in enumerate(done):
        for t in range(n):
            r = orc[t].step(X[t], CTX - 10, kv.numpy(), rb)
            assert (out.slots[t].cpu().numpy() == r.O).all() and (out.hit[t].cpu().numpy() == r.M).all(), (c, t)
            assert (out.miss_count[t].cpu().numpy() == r.n).all(), (c, t)
    for t in range(n):
        assert (ctx.buffer(t).cpu().numpy() == orc[t].rows()).all(), t
    assert ctx.sync_status() == 0
