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
