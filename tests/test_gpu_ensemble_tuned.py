"""A tuned ensemble is not slower than an untuned one (to the scatter of two
runs and the share of a run that the tuner's full iterations do not show:
8 %), whatever its members: one member of each of twelve classes, where tiles
searched class by class are too fine beside one another, and a few members of
one class."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TWELVE = [((8, 16, 24, 32)[k % 4], (3, 4, 5)[k // 4]) for k in range(12)]


@pytest.mark.parametrize("spec", [TWELVE, [(8, 3)] * 4])
def test_tuned_is_not_slower(spec):
    from paper_2101_05617_gb300 import swepi, synth
    ctxs, qs = [], []
    for i, (ne, p) in enumerate(spec):
        f = synth.make_fields("small_ne4_p3", i)
        ctxs.append(swepi.SWContext(ne, p, f.rotation))
        qs.append(torch.tensor(ctxs[-1].state_from_fields(*f.evaluate(ctxs[-1].node_xyz())).reshape(-1), device="cuda"))
    ens = swepi.SWEnsemble(ctxs)

    def run():
        for c in ctxs:
            c.epi_reset()
        ys = [q.clone() for q in qs]
        torch.cuda.synchronize()
        t = time.perf_counter()
        ens.epi_run(2, [4] * len(ys), [600.0] * len(ys), ys, m_init=48)
        return time.perf_counter() - t

    run()
    untuned = min(run() for _ in range(8))
    ens.tune(qs)
    run()
    tuned = min(run() for _ in range(8))
    ens.close()
    assert tuned < 1.08 * untuned, (tuned, untuned)
