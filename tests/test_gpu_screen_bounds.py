"""The bounds of the screening pass against the exact estimates, every pair of them, where they have least room: products of equal sign, so
that the tensor core's truncations add up, and operands that fp16 holds exactly, so that nothing else is in the constant.  The bounds are
not part of the interface: the debug build has a hook for them, and runs a screened search with its index checks on.  Runs in a child process,
because the library variant is chosen when the binding loads."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

_CHILD = r"""
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import torch
import paper_2504_19874_b200 as tq
import paper_2504_19874_b200.binding as B
from tests import parity as P
assert B._LIB_PATH.endswith("libtq_debug.so"), B._LIB_PATH
DEV, NIB = "cuda:0", tq.TQ_LAYOUT_NIBBLE
tightest = 0.0
for d, bits, mode, layout in ((128, 2, tq.TQ_MSE, None), (129, 1, tq.TQ_PROD, None), (200, 3, tq.TQ_PROD, None), (777, 4, tq.TQ_MSE, None),
                              (1000, 4, tq.TQ_PROD, NIB), (1537, 1, tq.TQ_MSE, None), (1536, 4, tq.TQ_PROD, None), (3072, 2, tq.TQ_PROD, None),
                              (3072, 4, tq.TQ_PROD, NIB), (3072, 3, tq.TQ_MSE, None)):
    su = P.Setup(d, bits, mode, layout=layout)
    g = torch.Generator(device=DEV).manual_seed(d + bits)
    n = 2100
    rand = lambda *shape: torch.randn(shape, generator=g, device=DEV)
    idx, qjl, gamma, norms = su.quantize(rand(n, d) + 0.2)
    for part in (idx, qjl):             # rows of equal codes: the largest centroid and signs up, the smallest and signs down
        if part is not None and part.numel():
            part[:300], part[300:600] = 0xFF, 0
    Pi = torch.from_numpy(su.Pi).to(DEV)
    norms[:] = 10.0 ** (12.0 * torch.rand(n, generator=g, device=DEV) - 6.0)
    if gamma is not None:
        gamma[:] = 2.0 * torch.rand(n, generator=g, device=DEV)
        gamma[::7] = 0.0
        gamma[1::7] = 1.0
    for nq in (70, 256):
        y = rand(nq, d)
        y[0], y[1], y[2:20], y[20:40] = 1.0, 0.75, y[2:20].abs(), torch.exp2(torch.floor(y[20:40].abs() * 3))   # rotated queries of equal sign
        Q = (y @ Pi).contiguous()
        if mode == tq.TQ_PROD:          # projections of equal sign
            Q[48:60] = torch.linalg.solve(torch.from_numpy(su.S).to(DEV).double(), y[8:20].double().T).T.float()
        Q[40:44] *= 1e12
        Q[44:48] *= 1e-12
        ws = torch.empty(1 << 24, dtype=torch.uint8, device=DEV)
        low, terms = torch.empty((nq, n), device=DEV), torch.empty((nq, 2), device=DEV)
        ptr = lambda t: ctypes.c_void_p(t.data_ptr() if t is not None else 0)
        f = B.lib().tq_debug_screen_bounds
        f.restype = ctypes.c_int
        rc = f(ctypes.c_void_p(su.plan.handle), ptr(Q), ctypes.c_int(nq), ctypes.c_int64(n), ptr(idx), ptr(qjl), ptr(gamma),
               ptr(norms), ptr(low), ptr(terms), ptr(ws), ctypes.c_size_t(ws.numel()), ctypes.c_void_p(0))
        assert rc == 0
        torch.cuda.synchronize()
        tq.tq_plan_status(su.plan)
        est = su.score(Q, n, idx, qjl, gamma, norms).double()
        rho = norms.double() * (1.0 + (gamma.double() if gamma is not None else 0.0))
        half = rho[None, :] * (terms[:, 0].double() * terms[:, 1].double())[:, None]
        mid = low.double() + half
        assert bool((terms[:, 0] > 0).all()) and bool((low.double() <= est).all()) and bool((est <= mid + half).all()), (d, bits, mode)
        tightest = max(tightest, float(((est - mid).abs() / half).max()))
print("tightest", tightest)
# a screened search with the index checks of the debug build
su = P.Setup(200, 3, tq.TQ_PROD)
g = torch.Generator(device=DEV).manual_seed(3)
X, Q = torch.randn((65_600, 200), generator=g, device=DEV), torch.randn((80, 200), generator=g, device=DEV)
codes = su.quantize(X)
codes[3][1000:1200] = -1.0
ts, ti = su.topk(Q, 65_600, *codes, 10)
tq.tq_plan_status(su.plan)
order = torch.sort(su.score(Q, 65_600, *codes), dim=1, descending=True, stable=True)
assert torch.equal(ts, order.values[:, :10]) and torch.equal(ti.long(), order.indices[:, :10])
print("bounds ok")
"""


def test_bounds_hold_for_every_pair():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    sys.path.insert(0, root)
    from paper_2504_19874_b200 import build as tq_build
    tq_build.build(debug=True)          # a no-op when libtq_debug.so is up to date
    env = dict(os.environ, TQ_LIB_VARIANT="debug")
    r = subprocess.run([sys.executable, "-c", _CHILD, root], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "bounds ok" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
