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


@pytest.mark.parametrize("mode", [1, 2])
def test_captured_behind_joins_and_copies(mode):
    """Calls recorded after a join of two streams, after a copy and after a
    fill, and on a second stream of the capture: the linked kernels' first node
    then depends on several nodes, or on ones that are not kernels."""
    from paper_2101_05617_gb300 import synth
    from paper_2101_05617_gb300.swepi import SWContext
    f = synth.make_fields("small_ne4_p3", 2)
    ctx = SWContext(4, 3, f.rotation)
    ctx.set_jvp_mode(mode)
    q0 = torch.tensor(ctx.state_from_fields(*f.evaluate(ctx.node_xyz())).reshape(-1), device="cuda")
    v0 = q0 * 1e-3
    q, v = q0.clone(), v0.clone()
    outs = [torch.empty_like(q) for _ in range(4)]
    side = torch.cuda.Stream()

    def calls():
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            v.copy_(v0)
            v.mul_(2.0)
        q.copy_(q0)
        main.wait_stream(side)
        ctx.rhs(q, out=outs[0])               # behind a join
        outs[1].zero_()
        ctx.jvp(q, v, out=outs[1])            # behind a fill
        v.copy_(v0)
        ctx.linearize(q)                      # behind a copy
        ctx.jvp_linearized(v, out=outs[2])
        side.wait_stream(main)
        with torch.cuda.stream(side):
            ctx.rhs(v0 + q0, out=outs[3])     # on the capture's second stream
        main.wait_stream(side)
    calls()
    torch.cuda.synchronize()
    ref = [o.clone() for o in outs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    for o in outs:
        o.zero_()
    graph.replay()
    torch.cuda.synchronize()
    for o, r in zip(outs, ref):
        assert torch.isfinite(r).all() and torch.equal(o, r)
