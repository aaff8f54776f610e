"""Top-k by screening: bounds from one fp16 pass decide which rows are scored, so the results are those of sorting the dense
estimates, bit for bit."""
import pytest
import torch

import paper_2504_19874_b200 as tq
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
NIB = tq.TQ_LAYOUT_NIBBLE


def check(su, Q, n, codes, k):
    nq = Q.shape[0]
    ts, ti = torch.empty((nq, k), device=DEV), torch.empty((nq, k), dtype=torch.int32, device=DEV)
    ws = torch.empty(tq.tq_workspace_bytes(su.plan, tq.TQ_OP_TOPK, n, nq, k), dtype=torch.uint8, device=DEV)
    tq.tq_topk(su.plan, Q, n, *codes, k, ts, ti, ws)
    tq.tq_plan_status(su.plan)
    order = torch.sort(su.score(Q, n, *codes), dim=1, descending=True, stable=True)
    assert torch.equal(ts, order.values[:, :k]) and torch.equal(ti.long(), order.indices[:, :k])


# one to four bits with and without signs; d at the edges of K steps (16; one-bit streams 8, 16, 32), k-blocks (64), row groups (128, 256) and of the nibble
# layout's blocks; n and nq at the edges of the row tiles (256) and of the passes' two widths (128, 256 queries)
@pytest.mark.parametrize("d,bits,mode,layout", [
    (128, 1, tq.TQ_MSE, None), (257, 1, tq.TQ_PROD, None), (200, 2, tq.TQ_MSE, None), (384, 2, tq.TQ_PROD, None), (200, 3, tq.TQ_PROD, None),
    (136, 3, tq.TQ_MSE, None), (130, 4, tq.TQ_MSE, None), (768, 4, tq.TQ_PROD, None), (200, 4, tq.TQ_PROD, NIB), (1000, 4, tq.TQ_PROD, NIB),
    (1536, 4, tq.TQ_PROD, NIB), (3072, 2, tq.TQ_PROD, None), (1537, 1, tq.TQ_MSE, None),
    (139, 3, tq.TQ_PROD, None), (171, 4, tq.TQ_PROD, None), (139, 1, tq.TQ_MSE, None), (207, 2, tq.TQ_PROD, None)])
@pytest.mark.parametrize("n,nq,k", [(65_537, 65, 10), (70_000, 128, 1), (65_536, 193, 100), (65_793, 513, 1)])
def test_screened_search_is_the_dense_one(d, bits, mode, layout, n, nq, k):
    su = P.Setup(d, bits, mode, layout=layout)
    g = torch.Generator(device=DEV).manual_seed(d + nq)
    X, Q = torch.randn((n, d), generator=g, device=DEV) + 0.3, torch.randn((nq, d), generator=g, device=DEV) + 0.3
    check(su, Q, n, su.quantize(X), k)


@pytest.mark.parametrize("nq", [80, 200])
def test_rows_and_queries_that_the_bounds_do_not_cover(nq):
    """Norms and gammas outside what the fp16 operands hold, a query of zeros, one of very large and one of very small entries, and
    rows that are all alike (more candidates than the lists hold: every row is scored)."""
    n, d, k = 65_600, 200, 10
    su = P.Setup(d, 3, tq.TQ_PROD)
    g = torch.Generator(device=DEV).manual_seed(1)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    idx, qjl, gamma, norms = su.quantize(X)
    norms[::1000] = 0.0
    norms[7::5000] = 1e-30
    norms[11::20000] = 1e27
    norms[13::20000] = -3.0
    gamma[17::5000] = 1e-7
    gamma[19::20000] = 1e6
    gamma[23::20000] = -2.0
    Q[3] = 0.0
    Q[5] *= 1e15
    Q[9] *= 1e-25
    check(su, Q, n, (idx, qjl, gamma, norms), k)
    same = su.quantize(X[:1].expand(n, d).contiguous())
    check(su, Q[:nq - 5], n, same, k)


@pytest.mark.parametrize("value", [-1.0, float("inf")])
@pytest.mark.parametrize("nq", [65, 80, 300])
def test_a_block_of_rows_that_the_bounds_do_not_cover(nq, value):
    """More such rows in one CTA's share than it collects per query: absent queries (up to the next multiple of 32) have no list, and nothing
    outside the outputs and the workspace changes, whatever the workspace held before."""
    n, d, k, pad = 65_600, 200, 10, 1 << 20
    su = P.Setup(d, 3, tq.TQ_PROD)
    g = torch.Generator(device=DEV).manual_seed(nq)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    codes = su.quantize(X)
    codes[3][1000:1200] = value
    ts, ti = torch.empty((nq, k), device=DEV), torch.empty((nq, k), dtype=torch.int32, device=DEV)
    need = (tq.tq_workspace_bytes(su.plan, tq.TQ_OP_TOPK, n, nq, k) + 255) // 256 * 256
    whole = torch.full((need + 2 * pad,), 0xBF, dtype=torch.uint8, device=DEV)
    tq.tq_topk(su.plan, Q, n, *codes, k, ts, ti, whole[pad:pad + need])
    tq.tq_plan_status(su.plan)
    assert bool((whole[:pad] == 0xBF).all()) and bool((whole[pad + need:] == 0xBF).all())
    order = torch.sort(su.score(Q, n, *codes), dim=1, descending=True, stable=True)
    assert torch.equal(ts, order.values[:, :k]) and torch.equal(ti.long(), order.indices[:, :k])


@pytest.mark.parametrize("d,bits,mode", [(128, 2, tq.TQ_MSE), (128, 1, tq.TQ_PROD), (128, 3, tq.TQ_PROD), (130, 4, tq.TQ_MSE), (256, 3, tq.TQ_MSE),
                                         (320, 2, tq.TQ_MSE), (130, 3, tq.TQ_PROD)])
def test_few_k_blocks_per_tile(d, bits, mode):
    """Two to six k-blocks per tile, even and odd, and some fifty tiles per CTA pair: several tiles within the ring of stages, and expansion
    sets and accumulators that take their turns at any place of it."""
    n, nq, k = 1_000_000, 200, 10
    su = P.Setup(d, bits, mode)
    g = torch.Generator(device=DEV).manual_seed(d)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    check(su, Q, n, su.quantize(X), k)


def test_norms_far_apart_and_negative_estimates():
    """Every estimate is negative and a few rows have norms 10^8 below the others': bounds of theirs that are rounded on the grid of the
    threshold would stand above their estimates.  They lie where the first sample does not look and the second does."""
    n, d, nq, k = 70_000, 200, 128, 10
    su = P.Setup(d, 3, tq.TQ_PROD)
    g = torch.Generator(device=DEV).manual_seed(5)
    X, Q = torch.randn((n, d), generator=g, device=DEV) + 2.0, 0.1 * torch.randn((nq, d), generator=g, device=DEV) - 1.0
    codes = su.quantize(X)
    codes[3].uniform_(0.5e8, 1e8, generator=g)
    codes[3][4:4 + 16 * 200:16] = 1.0
    assert bool((su.score(Q, n, *codes) < 0).all())
    check(su, Q, n, codes, k)


def spoilt(n, rows, spread, g):
    """A block of `rows` rows, or as many spread over the index."""
    return torch.randperm(n, generator=g, device=DEV)[:rows] if spread else torch.arange(1000, 1000 + rows, device=DEV)


@pytest.mark.parametrize("n,nq", [(3000, 3), (3000, 40), (65_600, 8), (65_600, 40), (65_600, 80), (65_600, 300)])
@pytest.mark.parametrize("rows,spread,gamma", [(100, True, False), (200, False, True), (1900, True, True), (5000, True, False), (40_000, False, False)])
def test_rows_without_a_number(n, nq, rows, spread, gamma):
    """Rows whose norm or residual norm is NaN are in no result, however many there are and whichever path the search takes: the exact
    one below 65,536 rows, thresholds, or screening from 65 queries on.  Where nearly all rows are such, the tail is empty."""
    d, k = 200, 10
    rows = min(rows, n - 5 if rows == 40_000 else n // 2)
    su = P.Setup(d, 3, tq.TQ_PROD)
    g = torch.Generator(device=DEV).manual_seed(rows + nq)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    codes = su.quantize(X)
    at = spoilt(n, rows, spread, g) if rows < n - 5 else torch.arange(rows, device=DEV)
    codes[2 if gamma else 3][at] = float("nan")
    ts, ti = su.topk(Q, n, *codes, k)
    tq.tq_plan_status(su.plan)
    scores = su.score(Q, n, *codes)
    assert bool(scores[:, at].isnan().all()) and int(scores.isnan().sum()) == nq * rows
    order = torch.sort(scores.nan_to_num(nan=-float("inf")), dim=1, descending=True, stable=True)
    values, ids = order.values[:, :k], order.indices[:, :k]
    assert torch.equal(ts, values) and torch.equal(ti.long(), torch.where(values == -float("inf"), -1, ids))


@pytest.mark.parametrize("d,bits,mode,layout", [(200, 3, tq.TQ_PROD, None), (200, 2, tq.TQ_MSE, None), (768, 4, tq.TQ_PROD, NIB)])
def test_a_query_that_every_row_passes(d, bits, mode, layout):
    """The atomics of so many hits hold up the warps that read the packed rows: the other queries' estimates of the rows beside them are
    formed from those rows all the same."""
    n, nq, k = 65_600, 200, 10
    su = P.Setup(d, bits, mode, layout=layout)
    g = torch.Generator(device=DEV).manual_seed(d)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    Q[3:6] *= 1e19
    codes = su.quantize(X)
    for _ in range(4):
        check(su, Q, n, codes, k)


@pytest.mark.parametrize("copies", [3000, 7000, 20_000, 40_000])
@pytest.mark.parametrize("d,bits,mode,layout", [(200, 3, tq.TQ_PROD, None), (768, 4, tq.TQ_PROD, NIB)])
def test_equal_rows_at_the_top(d, bits, mode, layout, copies):
    """More equal rows at the top of some queries' results than are scored one by one, than the screening lists hold, and than the lists of the
    exact passes hold: ties go to the lowest ids.  The other queries' passes are not touched by it."""
    n, nq, k = 70_000, 300, 100
    su = P.Setup(d, bits, mode, layout=layout)
    g = torch.Generator(device=DEV).manual_seed(copies)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    X[torch.randperm(n, generator=g, device=DEV)[:copies]] = X[0].clone()
    Q[70:90] += 2.0 * X[0]
    Q[280:] += 2.0 * X[0]
    check(su, Q, n, su.quantize(X), k)


@pytest.mark.parametrize("d,bits,mode,layout", [(200, 3, tq.TQ_PROD, None), (139, 1, tq.TQ_PROD, None), (200, 2, tq.TQ_MSE, None), (200, 4, tq.TQ_PROD, NIB)])
@pytest.mark.parametrize("rows", [0, 50, 1500])
def test_queries_of_zeros_and_without_a_number(d, bits, mode, layout, rows):
    """A batch padded with zeros gets the first k rows that have an estimate (behind `rows` rows without one), a query with a NaN an empty
    result, and the other queries what they get without them."""
    n, nq, k = 70_000, 200, 100
    su = P.Setup(d, bits, mode, layout=layout)
    g = torch.Generator(device=DEV).manual_seed(rows)
    X, Q = torch.randn((n, d), generator=g, device=DEV), torch.randn((nq, d), generator=g, device=DEV)
    codes = su.quantize(X)
    codes[3][:rows] = float("nan")
    Q[150:], Q[7, 3] = 0.0, float("nan")
    ts, ti = su.topk(Q, n, *codes, k)
    tq.tq_plan_status(su.plan)
    order = torch.sort(su.score(Q, n, *codes).nan_to_num(nan=-float("inf")), dim=1, descending=True, stable=True)
    values, ids = order.values[:, :k], order.indices[:, :k]
    assert torch.equal(ts, values) and torch.equal(ti.long(), torch.where(values == -float("inf"), -1, ids))
    assert bool((ti[7] == -1).all()) and torch.equal(ti[199].long(), torch.arange(rows, rows + k, device=DEV))


@pytest.mark.parametrize("n", [100, 9000])
def test_rows_without_a_number_in_short_vectors(n):
    """The same rule where the scans run on CUDA cores: what is left of k is empty."""
    d, k, nq = 64, 10, 3
    su = P.Setup(d, 3, tq.TQ_PROD)
    g = torch.Generator(device=DEV).manual_seed(n)
    codes = su.quantize(torch.randn((n, d), generator=g, device=DEV))
    codes[3][4:] = float("nan")
    ts, ti = su.topk(torch.randn((nq, d), generator=g, device=DEV), n, *codes, k)
    assert bool((ti[:, 4:] == -1).all()) and bool((ts[:, 4:] == -float("inf")).all())
    assert torch.equal(ti[:, :4].sort(dim=1).values.long(), torch.arange(4, device=DEV).expand(nq, 4))
