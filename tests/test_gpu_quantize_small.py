"""The one-launch quantiser (d = 32, 64, 96) at the edges of its 64-row tiles and over its bit widths, types and strides,
against the oracle by the criteria of the other quantiser tests."""
import pytest
import torch

import paper_2504_19874_b200 as tq
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
