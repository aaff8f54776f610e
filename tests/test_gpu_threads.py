"""Calls of different sizes from several host threads at once, each on its own stream: none of them may fail because another one
has set up the same kernel for less shared memory."""
import threading

import numpy as np
import pytest
import torch

import paper_2504_19874_b200 as tq

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
LONG = np.array([2, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 12, 12, 12, 12], dtype=np.uint8)


def plan(d, bits, mode=tq.TQ_MSE):
    eye = np.eye(d, dtype=np.float32)
    return tq.Plan(d, bits, mode, eye, eye if mode == tq.TQ_PROD else None, tq.tq_codebook(d, bits - (mode == tq.TQ_PROD))[0])


def pack_calls(p, errors):
    n = 64
    idx = torch.zeros((n, p.idx_row_bytes), dtype=torch.uint8, device=DEV)
    packed, offsets = tq.tq_entropy_pack(p, LONG, n, idx)

    def call(stream):
        rc = tq.lib().tq_entropy_pack(p.handle, LONG.ctypes.data, n, idx.data_ptr(), offsets.data_ptr(), packed.data_ptr(), packed.numel(), stream)
        if rc != 0:
            errors.append((p.d, rc, tq.lib().tq_last_error()))
    return call


def score_calls(p, errors):
    n, nq = 300, 2
    codes = [torch.zeros((n, p.idx_row_bytes), dtype=torch.uint8, device=DEV), torch.zeros((n, p.qjl_row_bytes), dtype=torch.uint8, device=DEV),
             torch.ones(n, device=DEV), torch.ones(n, device=DEV)]
    Q, scores = torch.ones((nq, p.d), device=DEV), torch.zeros((nq, n), device=DEV)
    ws = torch.zeros(tq.tq_workspace_bytes(p, tq.TQ_OP_SCORE, n, nq), dtype=torch.uint8, device=DEV)

    def call(stream):
        try:
            tq.tq_score(p, Q, n, *codes, scores, ws)
        except tq.TqError as e:
            errors.append((p.d, str(e)))
    return call


@pytest.mark.parametrize("kind", ["pack", "score"])
def test_calls_of_different_sizes_from_several_threads(kind):
    errors = []
    if kind == "pack":
        calls = [pack_calls(plan(d, 4), errors) for d in (4096, 1400, 4096, 1400)]
    else:
        plans = [plan(d, 4, tq.TQ_PROD) for d in (1536, 256, 1536, 256)]
        for p in plans:
            p.set_layout(tq.TQ_LAYOUT_NIBBLE)
        calls = [score_calls(p, errors) for p in plans]

    def work(call):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            for _ in range(3000):
                if errors:
                    return
                call(stream.cuda_stream)
        stream.synchronize()
    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:2]
