"""The packed coefficients of the split product (lin_node_kernel) where their
classes' magnitudes lie far apart: an element's exponents for u, A, S^i_j and
S^i_0 are chosen for one another, and none may cost another class its bits.
Elements that stay unpacked (a class out of the format's range) sit beside
packed ones, and all-zero classes (no wind, no rotation) are held too.  Split
and full product against the oracle, element by element, to the parity bound
of the JVP tests (8e-14 of the term scale of each variable)."""
import numpy as np
import pytest

from oracle import fields as ofields
from oracle import shallow_water as osw
from tests.gpu_common import oracle_case, scaled_direction, scaled_err_per_var, term_scale

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_JVP = 8e-14
OMEGA = 7.292e-5


def _products(g, q, v, hB=None, omega=OMEGA):
    from paper_2101_05617_gb300.swepi import SWContext
    ctx = SWContext(g.ne, g.ns - 1, g.rotation, omega=omega)
    if hB is not None:
        ctx.set_bottom(hB.reshape(-1))
    qd = torch.tensor(q.reshape(-1), device="cuda")
    vd = torch.tensor(v.reshape(-1), device="cuda")
    ctx.linearize(qd)
    out = [ctx.jvp_linearized(vd), ctx.jvp(qd, vd)]
    return [x.cpu().numpy().reshape(q.shape) for x in out]


def _check(g, q, v, hB=None, omega=OMEGA):
    ref, scale = osw.jvp(g, q, v), term_scale(g, q, v)
    for got in _products(g, q, v, hB, omega):
        err = scaled_err_per_var(got, ref, scale)
        assert max(err) < TOL_JVP, err


@pytest.mark.parametrize("depth,speed", [(8000.0, 20.0), (0.01, 0.5)])
@pytest.mark.parametrize("omega", [OMEGA, 0.0])
@pytest.mark.parametrize("ne,ns", [(1, 1), (3, 1), (23, 1), (5, 2), (3, 3), (2, 6)])
def test_sources_far_below_the_fluxes(ne, ns, omega, depth, speed):
    """An unrotated grid has panel-centre nodes (N_s = 1, odd n_e) with no
    Christoffel and, on the equator or without rotation, no Coriolis term, so
    S^i_j is zero there while u and A are not; over a thin layer A lies 23
    bits below u."""
    g = osw.Grid(ne, ns, (0.0, 0.0, 0.0), omega=omega)
    x, y, z = g.node_xyz()
    h = depth * (1.0 + 0.05 * x + 0.03 * y * z)
    V = speed * np.stack([0.3 * z - y, x - 0.2 * z, 0.2 * y - 0.3 * x])   # solid-body rotation
    hB = 0.1 * depth * (x * y + 0.5 * z)
    g.set_bottom(hB)
    q = ofields.state_from_fields(g, h, hB, V)
    _check(g, q, scaled_direction(q, 3), hB, omega)


@pytest.mark.parametrize("factor", [0.0, 1e-200])
@pytest.mark.parametrize("ne,ns", [(3, 1), (2, 2), (3, 4), (2, 6), (1, 8)])
def test_unpacked_and_packed_elements_side_by_side(ne, ns, factor):
    """One element's wind zero, or below the format (its coefficients stay FP64
    values), the others as they are; then the wind of the whole grid."""
    _, g, q, _ = oracle_case(ne, ns, seed=2)
    one = q.copy()
    one[1:, 1, 0, 0] *= factor
    still = q.copy()
    still[1:] *= factor
    v = scaled_direction(q, 4)
    for state in (one, still):
        _check(g, state, v)


@pytest.mark.parametrize("var", [0, 1, 2])
@pytest.mark.parametrize("ne,ns", [(3, 2), (3, 4), (2, 6), (2, 8)])
def test_directions_of_one_variable(ne, ns, var):
    """A direction in one variable alone leaves a momentum component with far
    smaller fluxes than the other's, which shares its exponent; each
    variable's error is measured against its own terms (the nodal fluxes, or the
    interface fluxes behind the result where those are larger)."""
    _, g, q, _ = oracle_case(ne, ns, seed=6)
    v = scaled_direction(q, 9)
    v[[k for k in range(3) if k != var]] = 0.0
    ref = osw.jvp(g, q, v)
    scale = [max(s, np.max(np.abs(r))) for s, r in zip(term_scale(g, q, v), ref)]
    for got in _products(g, q, v):
        err = scaled_err_per_var(got, ref, scale)
        assert max(err) < TOL_JVP, err


@pytest.mark.parametrize("ns", [2, 5])
def test_zero_entries_beside_huge_coefficients(ns):
    """Entries that are zero contribute nothing however large the exponent of
    their coefficient (a bottom of 1e200 m lifts S^i_0 and with it A) and
    however small the direction."""
    _, g, q, _ = oracle_case(2, ns, seed=3)
    x, y, z = g.node_xyz()
    hB = 1e200 * (x * y + 0.5 * z)
    g.set_bottom(hB)
    v = scaled_direction(q, 5)
    v[0] = 0.0
    for k in (0, -260, -320, -340, -360, -400):
        _check(g, q, np.ldexp(v, k), hB)
