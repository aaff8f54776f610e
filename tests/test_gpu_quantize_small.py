"""The one-launch quantiser (d = 32, 64, 96) at the edges of its 64-row tiles and over its bit widths, types and strides,
against the oracle by the criteria of the other quantiser tests."""
import numpy as np
import pytest
import torch

import paper_2504_19874_b200 as tq
from oracle import turboquant_oracle as orc
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("d", [32, 64, 96])
@pytest.mark.parametrize("bits,mode", [(1, tq.TQ_MSE), (2, tq.TQ_MSE), (3, tq.TQ_MSE), (4, tq.TQ_MSE),
                                       (1, tq.TQ_PROD), (2, tq.TQ_PROD), (3, tq.TQ_PROD), (4, tq.TQ_PROD), (5, tq.TQ_PROD)])
def test_codes_norms_and_residuals(d, bits, mode):
    su = P.Setup(d, bits, mode)
    for n, dtype, pad in ((1, torch.float32, 0), (63, torch.bfloat16, 0), (127, torch.float32, 1), (130, torch.bfloat16, 3)):
        g = torch.Generator(device="cpu").manual_seed(100 * d + 10 * bits + n)
        X = torch.randn((n, d + pad), generator=g)
        X[:, :4] *= 10.0                                        # outlier channels
        X[n // 2] = 0.0 if n > 1 else X[0]                      # a zero row
        X[0] *= 1e-6
        X = X.to(dtype).to(DEV)[:, :d]
        idx, qjl, gamma, norms = su.quantize(X)
        P.check_quantize(su, X, idx, qjl, gamma, norms)
        if su.mse_bits:
            P.check_pad_bits_zero(idx, su.mse_bits, d)
        if qjl is not None:
            P.check_pad_bits_zero(qjl, 1, d)
        if n == 127:                                            # rows taken as unit-norm
            U = torch.nn.functional.normalize(X, dim=1)
            U[n // 2] = U[1]                                    # (a zero row is not unit-norm: the oracle has no residual for it)
            P.check_quantize(su, U, *su.quantize(U, with_norms=False)[:3], None, unit_input=True)


@pytest.mark.parametrize("d", [32, 64, 96])
def test_rows_whose_norm_overflows(d):
    """The norm of such a row is inf and 1 / inf is 0: its residual is -c[idx], and a zero row's stays zero."""
    su = P.Setup(d, 3, tq.TQ_PROD)
    X = 1e20 * torch.randn((70, d), generator=torch.Generator().manual_seed(d)).to(DEV)
    X[3] = 0.0
    idx, qjl, gamma, norms = su.quantize(X)
    assert torch.isinf(norms[4]) and norms[3] == 0 and gamma[3] == 0
    e = -su.c[orc.unpack_bits(idx.cpu().numpy(), su.mse_bits, d)].astype(np.float64)
    e[3] = 0.0
    np.testing.assert_allclose(gamma.cpu().numpy(), np.linalg.norm(e, axis=1), rtol=1e-5, atol=0)
    z = e @ (su.S.astype(np.float64) @ su.Pi.astype(np.float64).T).T
    bits = np.unpackbits(qjl.cpu().numpy(), axis=1, bitorder="little")[:, :d]
    sure = np.abs(z) > 1e-5 * np.linalg.norm(z, axis=1, keepdims=True)
    sure[3] = True
    assert ((bits == 1) == (z >= 0))[sure].all()
