"""Indexes that a search must not be slow on.  On each of them the first pass once gave thresholds so low that the candidate lists
overflowed and all rows were scored a second time (2 to 100 times the time); here the time is held to that of a plain index of the
same size, and where a dense reference is affordable the result to it."""
import pytest
import torch

import paper_2504_19874_b200 as tq
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
N, D = 1_000_000, 200


def search(su, Q, n, codes, k):
    """(scores, ids, device time of a call in us)."""
    nq = Q.shape[0]
    ts, ti = torch.empty((nq, k), device=DEV), torch.empty((nq, k), dtype=torch.int32, device=DEV)
    ws = torch.empty(tq.tq_workspace_bytes(su.plan, tq.TQ_OP_TOPK, n, nq, k), dtype=torch.uint8, device=DEV)
    times = []
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        tq.tq_topk(su.plan, Q, n, *codes, k, ts, ti, ws)
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    tq.tq_plan_status(su.plan)
    return ts, ti, sorted(times)[2]


def check(su, Q, codes, k, limit):
    ts, ti, us = search(su, Q, N, codes, k)
    if Q.shape[0] <= 8:
        order = torch.sort(su.score(Q, N, *codes), dim=1, descending=True, stable=True)
        assert torch.equal(ts, order.values[:, :k]) and torch.equal(ti.long(), order.indices[:, :k])
    assert us < 2.5 * limit, (us, limit)


def random_codes(su, n, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    idx = torch.randint(0, 256, (n, su.idx_rb), generator=g, dtype=torch.uint8, device=DEV)
    idx[:, su.d * su.mse_bits // 8:] = 0
    return idx, None, None, 0.5 + torch.rand(n, generator=g, device=DEV)


@pytest.mark.parametrize("nq", [1, 8, 64])
@pytest.mark.parametrize("k", [10, 100])
def test_one_row_far_above_the_others(nq, k):
    su = P.Setup(D, 2, tq.TQ_MSE)
    codes = random_codes(su, N, 1)
    Q = torch.randn((nq, D), generator=torch.Generator().manual_seed(nq)).to(DEV)
    plain = search(su, Q, N, codes, k)[2]
    for norm in (1e4, 1e6):
        codes[3][:: N // 8] = norm                    # (row 0 is in any sample of the rows)
        check(su, Q, codes, k, plain)


@pytest.mark.parametrize("bits,mode,layout,nq", [(2, tq.TQ_MSE, None, 1), (2, tq.TQ_MSE, None, 8), (2, tq.TQ_MSE, None, 24), (2, tq.TQ_MSE, None, 64),
                                                 (4, tq.TQ_PROD, tq.TQ_LAYOUT_NIBBLE, 2), (4, tq.TQ_PROD, tq.TQ_LAYOUT_NIBBLE, 8)])
def test_rows_in_the_order_of_their_clusters(bits, mode, layout, nq):
    su = P.Setup(D, bits, mode, layout=layout)
    clusters, g = 1000, torch.Generator(device=DEV).manual_seed(1000)
    centres = torch.randn((clusters, D), generator=g, device=DEV)
    X = centres.repeat_interleave(N // clusters, dim=0) + torch.randn((N, D), generator=g, device=DEV)
    codes = su.quantize(X)
    shuffle = torch.randperm(N, generator=g, device=DEV)
    Q = centres[torch.randint(500, 1000, (nq,), generator=torch.Generator().manual_seed(5))] + torch.randn((nq, D), generator=g, device=DEV)
    for k in (10, 100):
        plain = search(su, Q, N, [None if t is None else t[shuffle].contiguous() for t in codes], k)[2]
        check(su, Q, codes, k, plain)


def test_the_nearest_of_very_many_rows():
    n = 34_000_000                                    # 8,192 candidates per score of the pilot once meant a list of 32,768 at times
    su = P.Setup(128, 1, tq.TQ_MSE)
    codes = random_codes(su, n, 2)
    Q = torch.randn((64, 128), generator=torch.Generator().manual_seed(3)).to(DEV)
    assert search(su, Q, n, codes, 1)[2] < 2.0 * search(su, Q, n, codes, 10)[2]


@pytest.mark.parametrize("nq", [1, 8, 24, 40])
@pytest.mark.parametrize("good", [4, 15])
def test_a_sample_that_misses_the_best_rows(nq, good):
    """The sample is every 16th row here (66,049 rows, 4,096 of them).  The `good` rows that follow each of these score far higher,
    so that the threshold admits them all: 16,512 candidates, more than a CTA's own list holds, or 61,921, more than the global
    lists hold, which is the rescue pass."""
    n, d, k = 66_049, 136, 64
    su = P.Setup(d, 2, tq.TQ_MSE)
    g = torch.Generator().manual_seed(nq)
    X, Q = torch.randn((n, d), generator=g) + 2.0, torch.randn((nq, d), generator=g) + 2.0
    at = torch.arange(n) % 16
    X[~((at >= 1) & (at <= good))] *= 0.01
    codes = su.quantize(X.to(DEV))
    ts, ti, _ = search(su, Q.to(DEV), n, codes, k)
    order = torch.sort(su.score(Q.to(DEV), n, *codes), dim=1, descending=True, stable=True)
    assert torch.equal(ts, order.values[:, :k]) and torch.equal(ti.long(), order.indices[:, :k])
