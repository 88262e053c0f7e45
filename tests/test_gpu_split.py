"""The FP64 RK4 step in two- and three-float arithmetic (rt_split.cuh) against
the general FP64 step, which the per-lane loop takes, and against the oracle's
paths, at the edges of the step's bounds and just past them."""
import numpy as np
import pytest

from paper_1012_5107_gb300 import inputs

pytestmark = pytest.mark.gpu


def render(rt, torch, p, variant):
    sc = rt.Scene(p)
    sc.set_launch(variant, 0)
    n = sc.height * sc.wout * sc.spp
    rgb = torch.zeros(sc.shape, dtype=torch.float32, device="cuda")
    rec = torch.zeros(n * 80, dtype=torch.uint8, device="cuda")
    sc.render(rgb, rec=rec)
    torch.cuda.synchronize()
    return rgb.cpu().numpy(), rt.records_to_numpy(rec), sc.stats()


# Both steps round at about 1e-16 a step; over some 1000 steps and the
# amplification of the rays that graze the grating, exits agree to 1e-12 on
# nearly all rays, and the bar is the one of the launch variants (1e-10).
@pytest.mark.parametrize("over", [
    dict(),
    dict(A=0.0),                                        # W0 = 0 everywhere
    dict(A=1e-6),                                       # a force far below the rounding of the momentum
    dict(A=0.0477),                                     # kA = 0.2997, the largest the step takes
    dict(A=0.048, width=24, height=20),                 # just past it: the general step
    dict(h=1.0 / 110.0, A=0.02),                        # |D| = 0.0653 at n_max: the general step
    dict(h=1.0 / 117.0, A=0.02),                        # 0.0614: within the bound
    dict(h=1.0 / 900.0, width=16, height=12),           # short steps
    dict(H=7.9, E=24.0, cam_dist=30.0, width=24, height=20),   # |W0| = 1e-22 at the box's top
    dict(H=8.1, E=24.0, cam_dist=30.0, width=12, height=8),    # past the bound on the box's height
    dict(H=0.11, E=6.0),                                # a box barely above the crests
    dict(E=0.7, elev_deg=12.0),                         # faces within a few steps of one another
    dict(E=32.0, cam_dist=40.0, width=24, height=20),
    dict(max_steps=50),                                 # the guard inside the cloak
    dict(max_bounces=0),
    dict(azim_deg=90.0, elev_deg=15.0),                 # along the grooves
    dict(width=7, height=5, spp=3, Lambda=0.6, A=0.02, E=4.8, H=1.2, h=0.003, cam_dist=7.2, bg_cell=0.3),
])
def test_split_step_equals_general_step(over):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    p = inputs.base_scene(**{**dict(width=40, height=32, spp=1, precision=1), **over})
    a_rgb, a, a_st = render(rt, torch, p, 0)
    b_rgb, b, b_st = render(rt, torch, p, 3)
    assert a_st["rays"] == b_st["rays"] and a_st["steps"] == b_st["steps"] and a_st["status"] == b_st["status"]
    assert b_st["evals"] >= 4 * b_st["steps"]
    for name in ("status", "bounces", "events", "steps"):
        assert np.array_equal(a[name], b[name]), name
    assert np.abs(a["pos"] - b["pos"]).max() <= 1e-10 * p["Lambda"]
    assert np.abs(a["dir"] - b["dir"]).max() <= 1e-10
    assert np.array_equal(a_rgb, b_rgb)


def test_split_render_repeats_and_matches_for_every_grouping():
    """The grouping of rays into warps changes no bit of the records."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    p = inputs.base_scene(width=72, height=50, spp=4, seed=5, precision=1)
    sc = rt.Scene(p)
    out = []
    for min_active in (1, 16, 28, 32, 28):
        sc.set_launch(3, min_active)
        rec = torch.zeros(72 * 50 * 4 * 80, dtype=torch.uint8, device="cuda")
        rgb = torch.zeros(sc.shape, dtype=torch.float32, device="cuda")
        sc.render(rgb, rec=rec)
        out.append(rec.cpu().numpy())
    assert all(np.array_equal(out[0], o) for o in out[1:])


# Dormand-Prince: the steps' sizes follow the error estimates, whose rounding is
# 1e-10 of them on both sides, so the two sides' exits differ by 1e-10 of the
# tolerance (1e-7) and by their rounding; the bar is again 1e-10.
@pytest.mark.parametrize("over", [
    dict(),
    dict(A=0.0),
    dict(A=0.0477),
    dict(A=0.048, width=24, height=20),                 # past kA = 0.3: the general step
    dict(rtol=1e-3, atol=1e-3),                         # steps of h_max: the general step
    dict(rtol=1e-6, atol=1e-6, A=0.01),                 # the loosest tolerance, weak forces: the longest steps
    dict(rtol=1e-10, atol=1e-10, width=20, height=16),
    dict(h_max=1.0 / 15.0, A=0.04),                     # |D| = 0.56 at n_max: the general step
    dict(h=0.5, h_max=0.06),                            # a first step past the bound: the general step
    dict(H=7.9, E=24.0, cam_dist=30.0, width=24, height=20),
    dict(H=0.11, E=6.0),
    dict(E=0.7, elev_deg=12.0),
    dict(max_steps=12),
    dict(azim_deg=90.0, elev_deg=15.0),
    dict(width=7, height=5, spp=3, Lambda=0.6, A=0.02, E=4.8, H=1.2, h=0.003, h_max=0.0375, cam_dist=7.2, bg_cell=0.3),
])
def test_wide_stages_equal_general_step(over):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    p = inputs.base_scene(**{**dict(width=40, height=32, spp=1, precision=1, integrator=inputs.DP45, rtol=1e-7, atol=1e-7),
                             **over})
    a_rgb, a, a_st = render(rt, torch, p, 0)
    b_rgb, b, b_st = render(rt, torch, p, 3)
    assert a_st["rays"] == b_st["rays"] and a_st["steps"] == b_st["steps"] and a_st["status"] == b_st["status"]
    for name in ("status", "bounces", "events", "steps"):
        assert np.array_equal(a[name], b[name]), name
    assert np.abs(a["pos"] - b["pos"]).max() <= 1e-10 * p["Lambda"]
    assert np.abs(a["dir"] - b["dir"]).max() <= 1e-10
    assert np.array_equal(a_rgb, b_rgb)


@pytest.mark.parametrize("integrator", [0, 1])
def test_batches_and_server_take_the_same_steps(integrator):
    """FP64 batches (all scenes within the bounds, one past them, an update from
    one to the other and back) and served requests equal the renders alone."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    base = dict(precision=1, integrator=integrator, rtol=1e-7, atol=1e-7, spp=4, seed=3)
    inside = [inputs.base_scene(width=40, height=28, **base), inputs.base_scene(width=33, height=20, A=0.02, azim_deg=20.0, **base)]
    past = [inside[0], dict(inside[1], A=0.05)]          # kA = 0.314
    bare = inputs.three_renders(inside[0])["bare"]

    def alone(p):
        sc = rt.Scene(p)
        rgb = torch.zeros(sc.shape, dtype=torch.float32, device="cuda")
        sc.render(rgb)
        return rgb.cpu().numpy()

    ref = {k: [alone(p) for p in ps] for k, ps in (("inside", inside + [bare]), ("past", past + [bare]))}
    scenes = [rt.Scene(p) for p in inside + [bare]]
    img = [torch.zeros(s.shape, dtype=torch.float32, device="cuda") for s in scenes]
    b = rt.Batch(scenes)
    for kind, ps in (("inside", inside), ("past", past), ("inside", inside)):
        b.update(ps + [bare])
        b.render(img)
        for t, r in zip(img, ref[kind]):
            assert np.array_equal(t.cpu().numpy(), r)
    assert b.stats()["sched_timeouts"] == 0
    s = rt.Server(1 << 28, max_inflight=2)
    out = [torch.zeros(sc.shape, dtype=torch.float32, device="cuda") for sc in scenes[:2] for _ in range(2)]
    tickets = [s.submit(p, t) for p, t in zip([inside[0], past[0], inside[1], past[1]], out)]
    for t in tickets:
        while s.poll(t, 1_000_000) is None:
            pass
    for t, r in zip(out, [ref["inside"][0], ref["past"][0], ref["inside"][1], ref["past"][1]]):
        assert np.array_equal(t.cpu().numpy(), r)
    s.close()
