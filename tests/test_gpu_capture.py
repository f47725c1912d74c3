"""The calls that only enqueue work (right-hand side, full product,
linearisation, split product in both forms) recorded in a CUDA graph after a
first call: their kernels are linked by programmatic dependent launch, and a
replay gives what the direct calls give, bit for bit, for new input values."""
import pytest

from tests.gpu_common import oracle_case, scaled_direction

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", [1, 2])
def test_enqueued_calls_under_capture(mode):
    from paper_2101_05617_gb300.swepi import SWContext
    _, g, q, _ = oracle_case(4, 4, seed=2)
    ctx = SWContext(g.ne, g.ns - 1, g.rotation)
    ctx.set_jvp_mode(mode)
    qd = torch.tensor(q.reshape(-1), device="cuda")
    vd = torch.tensor(scaled_direction(q, 3).reshape(-1), device="cuda")
    outs = [torch.empty_like(qd) for _ in range(3)]

    def calls():
        ctx.rhs(qd, out=outs[0])
        ctx.jvp(qd, vd, out=outs[1])
        ctx.linearize(qd)
        ctx.jvp_linearized(vd, out=outs[2])
    calls()   # tables and workspace are allocated by the first calls
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    qd.mul_(1.0 + 2.0 ** -20)
    vd.mul_(-3.0)
    calls()
    ref = [o.clone() for o in outs]
    for o in outs:
        o.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for o, r in zip(outs, ref):
        assert torch.isfinite(r).all() and torch.equal(o, r)
