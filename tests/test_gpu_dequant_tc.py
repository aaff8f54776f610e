"""The tensor-core reconstruction at the edges of its tiles, k-blocks, K splits and store paths, against the oracle.

Bound: the codes, norms and matrices are the same on both sides, so only the arithmetic differs.  The fp16 limb products keep
2^-23 of each product and an accumulation truncates at most 2 x 16 x 4 = 128 times (fewer for d < 3072) by 2^-23 of a partial
sum; a reconstructed row (norm nu up to 1 + the sign term) is therefore within sqrt(128) 2^-23 + 2^-22 < 2e-6 of its norm for
errors that do not all point one way, and a row of a few hundred coordinates shows a tenth of that."""
import numpy as np
import pytest
import torch

import paper_2504_19874_b200 as tq
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
NIB = tq.TQ_LAYOUT_NIBBLE


@pytest.mark.parametrize("d,bits,mode,layout,n,pad", [
    (128, 1, tq.TQ_MSE, None, 1, 0), (128, 2, tq.TQ_MSE, None, 129, 0), (131, 4, tq.TQ_MSE, None, 127, 0),
    (192, 3, tq.TQ_MSE, None, 257, 4), (200, 3, tq.TQ_PROD, None, 128, 3), (201, 1, tq.TQ_PROD, None, 70, 0),
    (320, 5, tq.TQ_PROD, None, 33, 0), (582, 4, tq.TQ_PROD, None, 300, 0), (1026, 2, tq.TQ_PROD, None, 5, 0),
    (136, 4, tq.TQ_PROD, NIB, 19000, 0), (136, 3, tq.TQ_PROD, None, 19013, 1), (264, 2, tq.TQ_MSE, None, 9600, 0),
    (1536, 4, tq.TQ_PROD, NIB, 600, 0), (1536, 3, tq.TQ_MSE, None, 3100, 0)])
def test_reconstruction_at_tile_edges(d, bits, mode, layout, n, pad):
    su = P.Setup(d, bits, mode, layout=layout)
    g = torch.Generator(device="cpu").manual_seed(11 * d + n)
    X = torch.randn((n, d), generator=g).to(DEV)
    codes = list(su.quantize(X))
    if mode == tq.TQ_PROD:
        codes[2][:: max(n // 3, 1)] = 0.0                       # rows without a sign term
    out = torch.full((n, d + pad), 7.0, device=DEV)
    tq.tq_dequantize(su.plan, n, *codes, out[:, :d])
    tq.tq_plan_status(su.plan)
    assert bool((out[:, d:] == 7.0).all()), "columns past d must stay as they are"
    rows = sorted({r for r in (0, 1, 31, 127, 128, 255, 256, n // 2, n - 2, n - 1) if 0 <= r < n})
    part = [None if t is None else t[rows] for t in codes]
    ref = P.oracle_dequant(su, *part)
    err = np.linalg.norm(P.as_f64(out[rows][:, :d]) - ref, axis=1) / np.maximum(np.linalg.norm(ref, axis=1), 1e-30)
    assert err.max() <= 2e-6, err.max()
    again = torch.empty((n, d), device=DEV)                     # unit norms
    tq.tq_dequantize(su.plan, n, codes[0], codes[1], codes[2], None, again)
    tq.tq_plan_status(su.plan)
    assert torch.allclose(again * codes[3][:, None], out[:, :d], rtol=1e-6, atol=0)


@pytest.mark.parametrize("n", [40, 3000])                       # both tiles
@pytest.mark.parametrize("bits,mode", [(3, tq.TQ_MSE), (3, tq.TQ_PROD)])
def test_norms_and_residual_norms_of_any_size(bits, mode, n):
    """Scaling a row's norm or its gamma scales the row: to 1e-6 of it where the result is a normal number (a quotient of two
    fp32 results of the same sums errs by three roundings, 3 x 2^-24), also at 1e-34 and at 1e30."""
    d = 256
    su = P.Setup(d, bits, mode)
    X = torch.randn((n, d), generator=torch.Generator().manual_seed(n)).to(DEV)
    idx, qjl, gamma, _ = su.quantize(X)
    ones = torch.ones(n, device=DEV)
    base = su.dequantize(n, idx, qjl, gamma, ones).double()
    for nu in (1e-34, 1e-30, 1e-20, 1e20, 1e30):
        out = su.dequantize(n, idx, qjl, gamma, ones * nu).double()
        assert ((out - base * float(np.float32(nu))).norm(dim=1) <= 1e-6 * (base * nu).norm(dim=1)).all(), nu
    if mode == tq.TQ_PROD:
        sign = su.dequantize(n, idx, qjl, ones * 2.0 ** 40, None).double()        # the centroid term is 2^-40 of this
        for g in (2.0 ** 60, 2.0 ** 100):
            out = su.dequantize(n, idx, qjl, ones * g, None).double()
            assert ((out - sign * (g / 2.0 ** 40)).norm(dim=1) <= 1e-6 * out.norm(dim=1)).all(), g
