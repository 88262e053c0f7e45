"""The edges of the range in which FP64 scenes take the steps of rt_split.cuh: the
step that ran, and its rays against those of the general step."""
import math

import numpy as np
import pytest

from paper_1012_5107_gb300 import inputs

pytestmark = pytest.mark.gpu


def edge(kA, scale):
    """scale times the largest RK4 step in range at kA: |D| <= 1/16 up to kA = 0.1, then |D|/(1 - kA) <= 0.06"""
    return scale * (1.0 / 16.0 if kA <= 0.1 else 0.06 * (1.0 - kA)) * (1.0 - kA) / 1.001 / (2.0 * math.pi)


def rk4(kA, h, **over):
    return dict(A=kA / (2.0 * math.pi), h=h, integrator=0, **over)


def dp45(kA, h_max, tol, **over):
    return dict(A=kA / (2.0 * math.pi), h=0.005, h_max=h_max, integrator=1, rtol=tol, atol=tol, **over)


# The general step counts the Newton steps of its solves, the split ones a fixed
# number a step, so the counts of the wavefront loop and of the per-lane loop,
# which steps in FP64 always, are equal where both took the general step and
# differ where not.  The bar on the exits is that of the launch variants (1e-10).
@pytest.mark.parametrize("over,inside", [
    (rk4(0.2999, edge(0.2999, 0.999)), True), (rk4(0.2999, edge(0.2999, 1.001)), False),
    (rk4(0.3001, 0.002), False), (rk4(0.0999, edge(0.0999, 0.999)), True), (rk4(0.0999, edge(0.0999, 1.001)), False),
    (rk4(0.1001, edge(0.1001, 0.999)), True), (rk4(0.1001, edge(0.1001, 1.001)), False),
    (rk4(0.02, edge(0.02, 0.999), H=0.08, E=6.0), True), (rk4(0.2513274, 0.005), True),
    (rk4(0.2513274, 0.005, E=32.0, cam_dist=40.0), True),        # abscissae of many periods
    (rk4(0.2513274, 0.005, E=60.0, cam_dist=70.0, azim_deg=10.0), True),
    (dp45(0.2799, 0.0625, 1e-6), True), (dp45(0.2801, 0.0625, 1e-6), False), (dp45(0.2513274, 0.0625, 1e-7), True),
    (dp45(0.2513274, 0.067, 1e-7), False), (dp45(0.1, 0.08, 1.1e-6), False), (dp45(0.1, 0.08, 1e-6), True),
])
def test_edges_of_the_range(over, inside):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    p = inputs.base_scene(**{**dict(width=40, height=32, spp=1, precision=1), **over})
    out = []
    for variant in (0, 3):
        sc = rt.Scene(p)
        sc.set_launch(variant, 0)
        rgb = torch.zeros(sc.shape, dtype=torch.float32, device="cuda")
        rec = torch.zeros(40 * 32 * 80, dtype=torch.uint8, device="cuda")
        sc.render(rgb, rec=rec)
        out.append((rgb.cpu().numpy(), rt.records_to_numpy(rec), sc.stats()))
    (a_rgb, a, a_st), (b_rgb, b, b_st) = out
    assert (a_st["newton"] == b_st["newton"]) == (not inside)
    for name in ("status", "bounces", "events", "steps"):
        assert np.array_equal(a[name], b[name]), name
    assert np.abs(a["pos"] - b["pos"]).max() <= 1e-10 and np.abs(a["dir"] - b["dir"]).max() <= 1e-10
    assert np.array_equal(a_rgb, b_rgb)
