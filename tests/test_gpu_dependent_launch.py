"""The right-hand side and the full product are pairs of kernels linked by
programmatic dependent launch.  Waiting successors must not keep a grid of
about one wave from spreading over the SMs: a grid with 1.56 times the
elements takes no more than 1.56 times as long (both fit one wave, so a
sound placement takes about the same; two face CTAs on an SM take twice)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _replay_us(f, calls=20, replays=20, rounds=7):
    f()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(calls):
            f()
    best = float("inf")
    for _ in range(rounds):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(replays):
            graph.replay()
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e3 / (calls * replays))
    return best


@pytest.mark.parametrize("call", ["rhs", "jvp"])
def test_time_grows_no_faster_than_the_work(call):
    from paper_2101_05617_gb300 import synth
    from paper_2101_05617_gb300.swepi import SWContext
    us = []
    for ne in (16, 20):
        f = synth.make_fields("small_ne4_p3", 1)
        ctx = SWContext(ne, 3, f.rotation)
        q = torch.tensor(ctx.state_from_fields(*f.evaluate(ctx.node_xyz())).reshape(-1), device="cuda")
        v, out = q * 1e-3, torch.empty_like(q)
        us.append(_replay_us((lambda: ctx.rhs(q, out=out)) if call == "rhs" else (lambda: ctx.jvp(q, v, out=out))))
    assert us[1] < (20 / 16) ** 2 * us[0], us
