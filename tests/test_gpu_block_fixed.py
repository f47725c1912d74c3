"""The block fixed-point sweeps of the DFR kernels at the edges of their
format: elements whose fluxes the 58-bit blocks cannot hold (values outside
2^-623 .. 2^677, NaN, infinities) take the FP64 chain, element by element, and
an all-zero element is exact.  The product is linear in v and a power of two
commutes with every rounding of both forms, so a scaled vector must give the
scaled product to the parity bound of the JVP tests (8e-14 of the term scale)
whichever form an element takes."""
import numpy as np
import pytest

from tests.gpu_common import oracle_case, scaled_direction, scaled_err_per_var, term_scale

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_JVP = 8e-14


def _ctx(g):
    from paper_2101_05617_gb300.swepi import SWContext
    return SWContext(g.ne, g.ns - 1, g.rotation)


def _product(ctx, split, qd, v):
    vd = torch.tensor(v.reshape(-1), device="cuda")
    return (ctx.jvp_linearized(vd) if split else ctx.jvp(qd, vd)).cpu().numpy().reshape(v.shape)


@pytest.mark.parametrize("split", [True, False])
@pytest.mark.parametrize("ne,ns", [(2, 1), (2, 2), (3, 3), (2, 5), (2, 6), (1, 8)])
def test_scaled_vectors_take_either_form(ne, ns, split):
    _, g, q, _ = oracle_case(ne, ns, seed=5)
    ctx = _ctx(g)
    qd = torch.tensor(q.reshape(-1), device="cuda")
    ctx.linearize(qd)
    v = scaled_direction(q, 6)
    ref = _product(ctx, split, qd, v)
    scale = term_scale(g, q, v)
    # 2^-700 (and, past the complex step's eps = 1e-30 ~ 2^-100, 2^-600) leave the format; 2^600 stays with eps
    for k in (-700, -600, -400, 300, 600):
        got = np.ldexp(_product(ctx, split, qd, np.ldexp(v, k)), -k)
        err = scaled_err_per_var(got, ref, scale)
        assert max(err) < TOL_JVP, (k, err)
    # one element scaled out of the format, its neighbours not: linearity again
    e = np.zeros_like(v)
    e[:, 0, 0, 0] = v[:, 0, 0, 0]
    small = np.ldexp(e, -900)
    assert np.array_equal(_product(ctx, split, qd, v - e + small), _product(ctx, split, qd, v - e)) or \
        max(scaled_err_per_var(_product(ctx, split, qd, v - e + small), _product(ctx, split, qd, v - e), scale)) < TOL_JVP


@pytest.mark.parametrize("split", [True, False])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("ns", [3, 6])
def test_nonfinite_values_stay_in_their_neighbourhood(ns, bad, split):
    """A NaN or infinity in v reaches its element (every line through the node)
    and its neighbours through their shared interfaces, and nothing else."""
    _, g, q, _ = oracle_case(4, ns, seed=3)
    ctx = _ctx(g)
    qd = torch.tensor(q.reshape(-1), device="cuda")
    ctx.linearize(qd)
    v = scaled_direction(q, 8)
    ref = _product(ctx, split, qd, v)
    w = v.copy()
    w[1, 2, 1, 2, 0, 0] = bad          # panel 2, interior element (e2, e1) = (1, 2)
    got = _product(ctx, split, qd, w)
    near = np.zeros(got.shape[1:4], dtype=bool)
    for d2, d1 in ((0, 0), (1, 0), (-1, 0), (0, 1), (0, -1)):
        near[2, 1 + d2, 2 + d1] = True
    assert not np.isfinite(got[:, 2, 1, 2, 0, 0]).all()
    assert np.isfinite(got[:, ~near]).all()
    assert np.array_equal(got[:, ~near], ref[:, ~near])


def test_zero_vector_and_zero_operator():
    """Krylov vectors start with an all-zero state block, and dt = 0 makes the sweeps' scale zero."""
    _, g, q, _ = oracle_case(3, 6, seed=4)
    ctx = _ctx(g)
    qd = torch.tensor(q.reshape(-1), device="cuda")
    ctx.linearize(qd)
    assert not ctx.jvp_linearized(torch.zeros_like(qd)).any()
    b = [torch.tensor(scaled_direction(q, k).reshape(-1), device="cuda") for k in range(3)]
    w, _ = ctx.kiops_phi(qd, 0.0, b, tol=1e-13)
    ref = b[0] + b[1] + b[2] / 2
    assert torch.linalg.norm(w - ref) < 1e-11 * torch.linalg.norm(ref)
