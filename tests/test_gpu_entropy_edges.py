"""Entropy coder at the edges of its work split: rows of fewer groups than lanes, groups and pairs cut by the end of the row,
long and incomplete codes, the 12-bit look-up, and so many rows that the offsets take their second level.  Whole numbers:
streams equal the oracle's and indices come back bit for bit."""
import numpy as np
import pytest
import torch

import paper_2504_19874_b200 as tq
from oracle import turboquant_oracle as orc
from tests import parity as P

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def random_rows(plan, d, bits, n, seed):
    g = np.random.default_rng(seed)
    sym = g.integers(0, 1 << bits, size=(n, d), dtype=np.uint8)
    b = ((sym[:, :, None] >> np.arange(bits)) & 1).astype(np.uint8).reshape(n, d * bits)
    rows = np.zeros((n, plan.idx_row_bytes), dtype=np.uint8)
    packed = np.packbits(b, axis=1, bitorder="little")
    rows[:, :packed.shape[1]] = packed
    return sym, torch.from_numpy(rows).to(DEV)


LONG = [2, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 12, 12, 12, 12]   # incomplete, up to 12 bits
DEEP = [10, 10, 9, 8, 7, 6, 5, 4, 3, 2, 2, 4, 6, 8, 9, 10]


@pytest.mark.parametrize("d,bits,lengths", [
    (8, 1, [1, 1]), (9, 1, [1, 2]), (15, 2, [1, 2, 3, 3]), (64, 3, [3] * 8), (131, 3, [1, 2, 3, 4, 5, 6, 7, 7]),
    (127, 4, LONG), (201, 4, DEEP), (257, 2, [3, 1, 2, 3]), (1537, 4, LONG), (2049, 1, [2, 1])])
def test_streams_and_round_trip(d, bits, lengths):
    su = P.Setup(d, bits, tq.TQ_MSE)
    lengths = np.array(lengths, dtype=np.uint8)
    assert np.sum(2.0 ** -lengths.astype(float)) <= 1.0
    codes = orc.canonical_codes(lengths)
    for n in (1, 9, 200):
        sym, idx = random_rows(su.plan, d, bits, n, d + n)
        packed, offsets = tq.tq_entropy_pack(su.plan, lengths, n, idx)
        tq.tq_plan_status(su.plan)
        off, data = offsets.cpu().numpy(), packed.cpu().numpy()
        bits_of = lengths[sym].astype(np.int64).sum(axis=1)
        assert np.array_equal(np.diff(off), (bits_of + 31) // 32 * 4) and off[0] == 0
        for r in sorted({0, n // 2, n - 1}):
            want, _ = orc.entropy_encode_row(sym[r], lengths, codes)
            row = data[off[r]:off[r + 1]]
            assert np.array_equal(row[:want.size], want) and not row[want.size:].any()
        back = torch.full_like(idx, 0xEE)
        tq.tq_entropy_unpack(su.plan, lengths, n, packed, offsets, back)
        assert torch.equal(back, idx)


@pytest.mark.parametrize("n", [1023, 1025, 40_000, (1 << 21) + 777])
def test_offsets_of_many_rows(n):
    su = P.Setup(8, 2, tq.TQ_MSE)
    idx = torch.zeros((n, su.plan.idx_row_bytes), dtype=torch.uint8, device=DEV)
    idx[:, :2] = torch.randint(0, 256, (n, 2), generator=torch.Generator().manual_seed(n), dtype=torch.uint8).to(DEV)
    lengths = np.array([1, 4, 12, 12], dtype=np.uint8)          # 8 .. 96 bits per row
    sym = (idx[:, :2].long()[:, :, None] >> torch.arange(0, 8, 2, device=DEV)) & 3
    size = (torch.tensor([1, 4, 12, 12], device=DEV)[sym].sum(dim=(1, 2)) + 31) // 32 * 4
    packed, offsets = tq.tq_entropy_pack(su.plan, lengths, n, idx)
    tq.tq_plan_status(su.plan)
    assert int(offsets[0]) == 0 and torch.equal(offsets[1:], size.cumsum(0)) and packed.numel() == int(offsets[n])
    back = torch.full_like(idx, 0xEE)
    tq.tq_entropy_unpack(su.plan, lengths, n, packed, offsets, back)
    assert torch.equal(back, idx)


@pytest.mark.parametrize("bits,lengths", [(1, [1, 1]), (2, [1, 2, 3, 3]), (3, [3] * 8), (4, DEEP)])
def test_rows_at_any_address(bits, lengths):
    """Index rows inside a larger buffer, off the 4-byte grid, and a workspace on no more than that grid: the same stream."""
    d, n = 203, 77
    su = P.Setup(d, bits, tq.TQ_MSE)
    lengths = np.array(lengths, dtype=np.uint8)
    _, idx = random_rows(su.plan, d, bits, n, bits)
    want, want_offsets = tq.tq_entropy_pack(su.plan, lengths, n, idx)
    for shift in (1, 2, 3, 4):
        buf = torch.full((idx.numel() + 8,), 0xA5, dtype=torch.uint8, device=DEV)
        moved = buf[shift:shift + idx.numel()].view(n, -1)
        moved.copy_(idx)
        packed, offsets = tq.tq_entropy_pack(su.plan, lengths, n, moved)
        tq.tq_plan_status(su.plan)
        assert torch.equal(packed, want) and torch.equal(offsets, want_offsets)
    need = tq.lib().tq_entropy_workspace_bytes(n)
    ws, offsets = torch.empty(need + 8, dtype=torch.uint8, device=DEV), torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    measure = lambda shift, at: tq.lib().tq_entropy_measure(su.plan.handle, lengths.ctypes.data, n, idx.data_ptr(), offsets.data_ptr() + at,  # noqa: E731
                                                            ws.data_ptr() + shift, need, torch.cuda.current_stream().cuda_stream)
    assert measure(4, 0) == 0 and torch.equal(offsets, want_offsets)
    assert measure(2, 0) == 3 and measure(0, 4) == 3          # TQ_ERR_ALIGNMENT, nothing launched


@pytest.mark.parametrize("d,bits,lengths", [(131, 4, LONG), (203, 3, [1, 2, 3, 4, 5, 6, 7, 7]), (9, 1, [1, 2]), (1537, 2, [3, 1, 2, 3])])
def test_bits_past_the_last_coordinate_do_not_count(d, bits, lengths):
    su = P.Setup(d, bits, tq.TQ_MSE)
    lengths = np.array(lengths, dtype=np.uint8)
    for n in (5, 200):
        _, idx = random_rows(su.plan, d, bits, n, n)
        want, want_offsets = tq.tq_entropy_pack(su.plan, lengths, n, idx)
        used = torch.zeros(idx.shape[1] * 8, dtype=torch.bool)
        used[:d * bits] = True
        pad = torch.from_numpy(np.packbits(~used.numpy(), bitorder="little")).to(DEV)
        for fill in (0xFF, 0x55):
            packed, offsets = tq.tq_entropy_pack(su.plan, lengths, n, idx | (pad & fill))
            tq.tq_plan_status(su.plan)
            assert torch.equal(offsets, want_offsets) and torch.equal(packed, want)


def test_bytes_of_the_output_that_hold_no_stream_are_zero():
    """A longer buffer, rows that the caller spaced out, and a buffer that is too small: nothing old shines through."""
    d, bits, n = 203, 3, 67
    su = P.Setup(d, bits, tq.TQ_MSE)
    lengths = np.array([1, 2, 3, 4, 5, 6, 7, 7], dtype=np.uint8)
    _, idx = random_rows(su.plan, d, bits, n, 4)
    packed, offsets = tq.tq_entropy_pack(su.plan, lengths, n, idx)
    streams, off = packed.cpu().numpy(), offsets.cpu().numpy()

    def pack(at, size):
        out = torch.full((size,), 0xFF, dtype=torch.uint8, device=DEV)
        at = torch.from_numpy(at).to(DEV)
        assert tq.lib().tq_entropy_pack(su.plan.handle, lengths.ctypes.data, n, idx.data_ptr(), at.data_ptr(), out.data_ptr(), size,
                                        torch.cuda.current_stream().cuda_stream) == 0
        return out.cpu().numpy()

    for spare in (0, 1, 6, 4099):
        got = pack(off, streams.size + spare)
        assert np.array_equal(got[:streams.size], streams) and not got[streams.size:].any()
    spaced = np.arange(n + 1, dtype=np.int64) * 200 + 16               # 200 > the longest stream of this code
    want = np.zeros(int(spaced[n]) + 5, dtype=np.uint8)
    for r in range(n):
        want[spaced[r]:spaced[r] + off[r + 1] - off[r]] = streams[off[r]:off[r + 1]]
    assert np.array_equal(pack(spaced, want.size), want)
    tq.tq_plan_status(su.plan)
    size = int(off[n // 2]) + 7                                         # row n / 2 does not fit
    want = np.zeros(size, dtype=np.uint8)
    want[:off[n // 2]] = streams[:off[n // 2]]
    assert np.array_equal(pack(off, size), want)
    with pytest.raises(tq.TqError):
        tq.tq_plan_status(su.plan)
