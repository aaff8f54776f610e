"""The selection kernel at the limits of its two methods: lists around the register limit, ties, a far outlier that leaves all
other scores in one bin, non-finite scores, empty slots.  Order and ids are exact: descending score, then ascending id."""
import numpy as np
import pytest
import torch

import paper_2504_19874_b200 as tq

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def expected(s, i, k):
    keep = np.nonzero(i >= 0)[0]
    order = keep[np.lexsort((i[keep], -s[keep].astype(np.float64)))][:k]
    out_s, out_i = np.full(k, -np.inf, np.float32), np.full(k, -1, np.int32)
    out_s[:order.size], out_i[:order.size] = s[order], i[order]
    return out_s, out_i


@pytest.mark.parametrize("m", [1, 31, 1000, 1025, 4096, 4097, 16384, 16385, 40000])
@pytest.mark.parametrize("kind", ["normal", "ties", "equal", "outlier", "infinite", "empty slots", "crowded"])
def test_selection(m, kind):
    g = np.random.default_rng(m)
    nq = 3
    s = g.standard_normal((nq, m)).astype(np.float32)
    if kind == "ties":
        s = np.round(s, 1)
        s[s == 0] = 0.0
    elif kind == "equal":
        s[:] = 0.25
    elif kind == "outlier":
        s[:, m // 2] = 1e30
    elif kind == "infinite":
        s[0, 0], s[1, m - 1] = np.inf, -np.inf
    elif kind == "crowded":   # the largest scores meet in few threads, so that the threads' maxima say little about them
        s[:, np.arange(m) % 1024 < 40] += 10.0
    ids = np.stack([g.permutation(m) for _ in range(nq)]).astype(np.int32)
    if kind == "empty slots":
        ids[g.random((nq, m)) < 0.9] = -1
    cs, ci = torch.from_numpy(s).to(DEV), torch.from_numpy(ids).to(DEV)
    for k in (1, 10, 256, 257, 1024):
        ts, ti = torch.empty((nq, k), device=DEV), torch.empty((nq, k), dtype=torch.int32, device=DEV)
        tq.tq_select_topk(cs, ci, k, ts, ti)
        for q in range(nq):
            ws, wi = expected(s[q], ids[q], k)
            assert np.array_equal(ti[q].cpu().numpy(), wi) and np.array_equal(ts[q].cpu().numpy(), ws), (q, k)


@pytest.mark.parametrize("m", [6, 300, 2000, 5000])
def test_the_same_pair_given_twice(m):
    """Shards that overlap hand in a (score, id) pair twice: every output slot is written, both copies in place."""
    g = np.random.default_rng(m)
    s, ids = np.repeat(g.standard_normal(m // 2).astype(np.float32), 2), np.repeat(g.permutation(m // 2).astype(np.int32), 2)
    shuffle = g.permutation(m)
    s, ids = s[shuffle], ids[shuffle]
    cs, ci = torch.from_numpy(s[None]).to(DEV), torch.from_numpy(ids[None]).to(DEV)
    for k in (1, 6, 100, 256, 1000):
        ts, ti = torch.full((1, k), -77.0, device=DEV), torch.full((1, k), -77, dtype=torch.int32, device=DEV)
        tq.tq_select_topk(cs, ci, k, ts, ti)
        ws, wi = expected(s, ids, k)
        assert np.array_equal(ti[0].cpu().numpy(), wi) and np.array_equal(ts[0].cpu().numpy(), ws)


def test_the_longest_list():
    """2^31 - 1 candidates: positions and the loop that counts them end at the largest 32-bit integer."""
    m, k = 2**31 - 1, 10
    if torch.cuda.mem_get_info()[0] < 24e9:
        pytest.skip("needs 17 GB of device memory")
    s, ids = torch.empty((1, m), device=DEV), torch.arange(m, dtype=torch.int32, device=DEV)[None]
    s.uniform_(0.0, 1.0)
    at = torch.tensor([m - 1, 0, m - 8192, 5, 8191, m // 2, m - 2, 2**30, 8192, m - 1025], device=DEV)
    s[0, at] = torch.arange(20, 10, -1, device=DEV, dtype=torch.float32)
    ts, ti = torch.empty((1, k), device=DEV), torch.empty((1, k), dtype=torch.int32, device=DEV)
    tq.tq_select_topk(s, ids, k, ts, ti)
    assert torch.equal(ti[0].long(), at) and ts[0].tolist() == list(range(20, 10, -1))
