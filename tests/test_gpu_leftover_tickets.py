"""A call whose bounded wait gave up can leave the solver's tickets mid-count
(SW_ETIMEOUT).  The next call on the context, whichever driver or ensemble
takes it, must start from clean ones: with leftover counts planted
(sw_check_inject, checked build, in a process of its own) it gives what a
fresh context gives.  No wait of these calls depends on the planted counts."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WORKER = r"""
import sys
import torch
from paper_2101_05617_gb300 import swepi
from tests.gpu_common import oracle_case, scaled_direction

_, g, q, _ = oracle_case(4, 4, seed=1)
qd = torch.tensor(q.reshape(-1), device="cuda")
b = [torch.tensor(scaled_direction(q, k).reshape(-1), device="cuda") for k in range(3)]
big = [None] + [1024.0 * x for x in b[1:]]


def context(driver, mode):
    ctx = swepi.SWContext(g.ne, g.ns - 1, g.rotation)
    ctx.set_jvp_mode(mode)
    ctx.set_kiops_driver(driver)
    ctx.kiops_phi(qd, 30.0, b, tol=1e-8, m_init=12, iop=3)
    return ctx


for driver in (0, 1):
    for mode in (1, 2):
        res = []
        for planted in (False, True):
            ctx = context(driver, mode)
            if planted:
                swepi.sw_check_inject(ctx.handle, 2)
            w, st = ctx.kiops_phi(qd, 30.0, big, tol=1e-8, m_init=12, iop=3)
            assert torch.isfinite(w).all()
            res.append((w.clone(), st))
        assert res[0][1] == res[1][1], (driver, mode, res[0][1], res[1][1])
        assert torch.equal(res[0][0], res[1][0]), (driver, mode)

# the complex64-bulk product alone: its bounded waits have a place to report to from the linearisation on
ctx = swepi.SWContext(g.ne, g.ns - 1, g.rotation)
ctx.set_jvp_mode(2)
ctx.linearize(qd)
swepi.sw_check_inject(ctx.handle, 2)   # refused while the context has no flags
assert torch.isfinite(ctx.jvp_linearized(b[1])).all()

res = []
for planted in (False, True):
    ctxs = [context(0, 1) for _ in range(2)]
    if planted:
        for c in ctxs:
            swepi.sw_check_inject(c.handle, 2)
    ens = swepi.SWEnsemble(ctxs)
    ys = [qd.clone() for _ in ctxs]
    st = ens.epi_run(2, [4, 4], [900.0, 900.0], ys, tol=1e-10)
    res.append((ys, [s["krylov_iters"] for s in st]))
    ens.close()
assert res[0][1] == res[1][1], (res[0][1], res[1][1])
for a, c in zip(res[0][0], res[1][0]):
    assert torch.linalg.norm(a - c) < 1e-12 * torch.linalg.norm(a)
print("ok")
"""


def test_calls_after_leftover_counts():
    from paper_2101_05617_gb300 import build as b
    b.build(checked=True)
    r = subprocess.run([sys.executable, "-c", WORKER], cwd=ROOT, env=dict(os.environ, SWEPI_CHECKED="1"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, (r.stdout[-2000:], r.stderr[-3000:])
