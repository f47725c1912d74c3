"""Phi-function calls at p = 0 and 1, where an element has one or four nodes
and the kernels take forms of their own (N_s = 1: the split product from
registers; the window of three with five dots a node): both windows, the
split and the full product, the host's and the device's controller, against
the oracle (the same Krylov, substep and rejection counts, the product to
1e-10 as in the other parity tests)."""
import numpy as np
import pytest

from oracle import kiops as okiops
from oracle import shallow_water as osw
from tests.gpu_common import oracle_case, rel_l2_per_var, scaled_direction

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,driver", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("iop", [2, 3])
@pytest.mark.parametrize("ne,ns", [(5, 1), (17, 1), (4, 2)])
def test_phi_parity(ne, ns, iop, mode, driver):
    from paper_2101_05617_gb300.swepi import SWContext
    _, g, q, _ = oracle_case(ne, ns, seed=12)
    dt, tol = 3600.0, 1e-10
    bs = [None, dt * osw.rhs_real(g, q)] + [1e-3 * dt * scaled_direction(q, 70 + k) for k in range(2)]
    ctx = SWContext(g.ne, g.ns - 1, g.rotation)
    ctx.set_jvp_mode(mode)
    ctx.set_kiops_driver(driver)
    qd = torch.tensor(q.reshape(-1), device="cuda")
    bd = [None if b is None else torch.tensor(b.reshape(-1), device="cuda") for b in bs]
    w, st = ctx.kiops_phi(qd, dt, bd, tol=tol, iop=iop)
    ref, rst = okiops.kiops(1.0, lambda x: dt * osw.jvp(g, q, x.reshape(q.shape)).reshape(-1),
                            [np.zeros(q.size)] + [b.reshape(-1) for b in bs[1:]], tol=tol, iop=iop)
    err = rel_l2_per_var(w.cpu().numpy(), ref)
    assert max(err) < 1e-10, (err, st, rst)
    assert (st["krylov_iters"], st["substeps"], st["rejects"]) == \
        (rst["krylov_iters"], rst["substeps"], rst["rejects"]), (st, rst)
