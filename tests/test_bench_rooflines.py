"""The benchmark's reported rooflines (CPU): the kernels that run most of their
flops as integers carry no fraction of the FP64 peak, and the vector passes
are reported as the one launch that is timed."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _prof(orth_count=20):
    prof = {k: {"ms": 0.0, "count": 0} for k in ("volume_jvp", "face_jvp", "orthogonalisation", "expm", "linearize")}
    prof["volume_jvp"] = {"ms": 0.8, "count": 10}
    prof["face_jvp"] = {"ms": 0.2, "count": 10}
    prof["orthogonalisation"] = {"ms": 0.3, "count": orth_count}
    return prof


def _keys(x):
    for k, v in x.items():
        yield k
        if isinstance(v, dict):
            yield from _keys(v)


def test_reported_kernels_are_set_against_bytes():
    import bench
    from paper_2101_05617_gb300 import synth
    wl = synth.WORKLOADS["ne60_p5"]
    nodes = 6 * 60 * 60 * 36
    for mode, w in ((1, 8), (2, 4)):
        r = bench.kernel_rooflines(_prof(), wl, mode, 2, 10.0, fused=True)
        assert not any("fp64" in k for k in _keys(r))
        # v, 18 coefficients and twice three fluxes at 2 / 6 points a node, 20 us a launch
        fb = nodes * (3 * w + 24 * w / 3.0)
        assert abs(r["face"]["bytes"] - fb) < 1e-9 * fb
        assert abs(r["face"]["gbs"] - fb / 2e-5 / 1e9) < 1e-9 * r["face"]["gbs"]
        assert r["orthogonalisation"]["bytes_per_iteration"] == (32 + (4 if mode == 2 else 0)) * (wl.n_unknowns + 4)


def test_vector_passes_reported_as_one_launch():
    import bench
    from paper_2101_05617_gb300 import synth
    wl = synth.WORKLOADS["ne60_p5"]
    assert bench.ortho_roofline(_prof(), wl, True)["bytes_per_iteration"] == 32 * (wl.n_unknowns + 4)
    assert bench.ortho_roofline(_prof(), wl, False) is None


def test_full_evaluation_bytes():
    import bench
    # 6 nodes a line, four b-columns, window of two: q, v, Jv 72, 13 coefficients, fluxes, window, b-columns
    assert bench.full_bytes_per_node(6, "volume", 2, 4) == 72 + 104 + 16 + 48 + 96
    assert bench.full_bytes_per_node(6, "face", 2, 4) == 48 + (96 + 48) / 3
