"""Tiles of the tensor-core quantiser: every output is one sum in one order on all of them, so the codes of a row are the same
bits however many rows come with it -- 128 x 64 tiles for a few rows, CTA pairs of 128, 192 and 256 columns for more, one block
of rows or two."""
import pytest
import torch

import paper_2504_19874_b200 as tq

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def quantize(plan, X, mode):
    n = X.shape[0]
    idx = torch.full((n, plan.idx_row_bytes), 7, dtype=torch.uint8, device=DEV)
    norms = torch.zeros(n, device=DEV)
    scratch = torch.empty(max(tq.tq_workspace_bytes(plan, tq.TQ_OP_QUANTIZE, n), 256), dtype=torch.uint8, device=DEV)
    if mode == tq.TQ_MSE:
        tq.tq_quantize_mse(plan, X, idx, norms, scratch)
        return idx, norms
    qjl = torch.full((n, plan.qjl_row_bytes), 7, dtype=torch.uint8, device=DEV)
    gamma = torch.zeros(n, device=DEV)
    tq.tq_quantize_prod(plan, X, idx, qjl, gamma, norms, scratch)
    return idx, qjl, gamma, norms


@pytest.mark.parametrize("d,n", [(129, 9000), (200, 20000), (384, 20000), (600, 9000), (1536, 9000), (3072, 5000)])
@pytest.mark.parametrize("mode,bits,nibble", [(tq.TQ_PROD, 4, True), (tq.TQ_PROD, 2, False), (tq.TQ_MSE, 2, False)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_codes_do_not_depend_on_the_number_of_rows(d, n, mode, bits, nibble, dtype):
    prod = mode == tq.TQ_PROD
    cent, _ = tq.tq_codebook(d, bits - 1 if prod else bits)
    plan = tq.Plan(d, bits, mode, tq.tq_rotation(d, 5), tq.tq_rotation(d, 6, tq.TQ_GAUSSIAN) if prod else None, cent)
    if nibble:
        plan.set_layout(tq.TQ_LAYOUT_NIBBLE)
    X = torch.randn((n, d), generator=torch.Generator(device=DEV).manual_seed(d), device=DEV).to(dtype)
    whole = quantize(plan, X, mode)
    for rows in (1, 127, 128, 129, 300, 1001, 2049, 4097):
        for part, full in zip(quantize(plan, X[:rows], mode), whole):
            assert torch.equal(part, full[:rows]), rows
    # rows that are not 16-byte aligned (fp32 rows of whole 16-byte pieces take another order of the norm's sum when they are)
    Y = torch.zeros((300, d + 1), dtype=dtype, device=DEV)
    Y[:, :d] = X[:300]
    for part, full in zip(quantize(plan, Y[:, :d], mode), whole):
        if dtype == torch.bfloat16 or d % 4:
            assert torch.equal(part, full[:300])


@pytest.mark.parametrize("d,n", [(129, 70), (384, 300), (3072, 130), (5000, 40)])
@pytest.mark.parametrize("mode,bits", [(tq.TQ_PROD, 3), (tq.TQ_MSE, 2)])
def test_bf16_rows_at_any_scale(d, n, mode, bits):
    """Rows enter the rotation scaled by a power of two: codes are those of the same rows at another power of two, bit for bit, and rows
    of zeros, of a norm that overflows or of a NaN are coded as the fp32 rows are."""
    prod = mode == tq.TQ_PROD
    cent, _ = tq.tq_codebook(d, bits - 1 if prod else bits)
    plan = tq.Plan(d, bits, mode, tq.tq_rotation(d, 5), tq.tq_rotation(d, 6, tq.TQ_GAUSSIAN) if prod else None, cent)
    X = torch.randn((n, d), generator=torch.Generator(device=DEV).manual_seed(d), device=DEV).bfloat16()
    base = quantize(plan, X, mode)
    for e in (-50, 40):                                # squares stay inside fp32
        out = quantize(plan, X * 2.0 ** e, mode)
        for a, b in zip(out[:-1], base[:-1]):
            assert torch.equal(a, b), e
        assert torch.equal(out[-1], base[-1] * 2.0 ** e)
    X[3] = 0.0
    X[5, 7] = 1e30
    X[7, 2] = float("nan")
    X[9] = 1e-30
    for a, b in zip(quantize(plan, X, mode)[:-1], quantize(plan, X.float(), mode)[:-1]):
        for r in (3, 5, 7, 9):
            assert torch.equal(a[r], b[r]) or (a.dtype == torch.float32 and torch.isnan(a[r]) and torch.isnan(b[r])), r
