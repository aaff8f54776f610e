"""The eight-query shape of the register-fed scan (5 to 8 queries on the bit streams): ragged dimensions and row counts around its
256- and 128-row tiles, every bit width, dense scores and top-k.  Its estimates are the single-query shape's bit for bit (the
same exact integers), and the first case of each plan is held to the oracle by the usual criterion."""
import pytest
import torch

import paper_2504_19874_b200 as tq
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d,bits,mode", [(128, 1, tq.TQ_MSE), (200, 3, tq.TQ_PROD), (515, 2, tq.TQ_MSE), (520, 4, tq.TQ_PROD),
                                         (264, 5, tq.TQ_PROD), (1030, 3, tq.TQ_MSE), (768, 1, tq.TQ_PROD), (1032, 4, tq.TQ_MSE)])
def test_eight_queries(d, bits, mode):
    su = P.Setup(d, bits, mode)
    g = torch.Generator(device="cpu").manual_seed(d + bits)
    X, Q = torch.randn((2309, d), generator=g).to(DEV), torch.randn((8, d), generator=g).to(DEV)
    codes = su.quantize(X)
    one = torch.cat([su.score(Q[q:q + 1].clone(), 2309, *codes) for q in range(8)])
    P.check_scores(su, one, Q, *codes)
    for nq, n in ((8, 2309), (5, 1), (6, 127), (7, 257), (8, 2304)):
        part = [None if t is None else t[:n].contiguous() for t in codes]
        assert torch.equal(su.score(Q[:nq].contiguous(), n, *part), one[:nq, :n])
    ts, ti = su.topk(Q, 2309, *codes, 20)
    order = torch.sort(one, dim=1, descending=True, stable=True)
    assert torch.equal(ts, order.values[:, :20]) and torch.equal(ti.long(), order.indices[:, :20])


def test_filter_pass():
    su = P.Setup(136, 2, tq.TQ_MSE)
    g = torch.Generator(device="cpu").manual_seed(5)
    n = 70_003
    X, Q = torch.randn((n, 136), generator=g).to(DEV), torch.randn((8, 136), generator=g).to(DEV)
    codes = su.quantize(X)
    sc = su.score(Q, n, *codes)
    for nq, k in ((8, 100), (5, 1), (7, 1024)):
        ts, ti = su.topk(Q[:nq].contiguous(), n, *codes, k)
        order = torch.sort(sc[:nq], dim=1, descending=True, stable=True)
        assert torch.equal(ts, order.values[:, :k]) and torch.equal(ti.long(), order.indices[:, :k])


@pytest.mark.parametrize("nq", [9, 16, 17, 32, 33, 64])
def test_filter_pass_whose_lanes_hit_unequally(nq):
    """Every seventh row is close to all queries, so that a lane of the tensor-core scans has up to sixteen hits at once and its
    neighbours none."""
    su = P.Setup(136, 2, tq.TQ_MSE)
    g = torch.Generator(device="cpu").manual_seed(nq)
    n = 70_003
    X, Q = torch.randn((n, 136), generator=g), torch.randn((nq, 136), generator=g) + 2.0
    X[::7] += 2.0
    codes = su.quantize(X.to(DEV))
    sc = su.score(Q.to(DEV), n, *codes)
    order = torch.sort(sc, dim=1, descending=True, stable=True)
    for k in (1, 1024):
        ts, ti = su.topk(Q.to(DEV), n, *codes, k)
        tq.tq_plan_status(su.plan)
        assert torch.equal(ts, order.values[:, :k]) and torch.equal(ti.long(), order.indices[:, :k])
