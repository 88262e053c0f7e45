"""How the wavefront loop cuts its integration tasks (rt_wave.cuh), and the
launch configuration's setters and tuner: nothing of it changes a result."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1012_5107_gb300 import inputs

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


# Rays across the grooves at grazing elevation leave the box so far apart that
# the FP32 loops begin to cut their tasks (wave_ragged, from some 100,000 steps
# of uncut tasks on); the last camera keeps them together.
@pytest.mark.parametrize("integrator", [0, 1, 2])
@pytest.mark.parametrize("over", [
    dict(azim_deg=90.0, elev_deg=10.0, E=32.0, cam_dist=40.0),
    dict(azim_deg=60.0, elev_deg=12.0, E=16.0, cam_dist=24.0, A=0.02),
    dict(azim_deg=90.0, elev_deg=10.0, E=32.0, cam_dist=40.0, A=0.06, flags=1),
    dict(),
])
def test_cut_tasks_change_nothing(integrator, over):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    p = inputs.base_scene(**{**dict(width=200, height=168, spp=4, precision=0, integrator=integrator, rtol=1e-5,
                                    atol=1e-5, seed=9, max_steps=40000), **over})
    out = []
    for min_active in (0, 1, 32, 0):
        sc = rt.Scene(p)
        sc.set_launch(3, min_active)
        rgb = torch.zeros(sc.shape, dtype=torch.float32, device="cuda")
        rec = torch.zeros(200 * 168 * 4 * 80, dtype=torch.uint8, device="cuda")
        sc.render(rgb, rec=rec)
        st = sc.stats()
        assert st["sched_timeouts"] == 0 and st["rays"] == 200 * 168 * 4
        out.append((rgb.cpu().numpy(), rec.cpu().numpy(), st["steps"]))
    for o in out[1:]:
        assert np.array_equal(out[0][0], o[0], equal_nan=True) and np.array_equal(out[0][1], o[1]) and out[0][2] == o[2]


@pytest.mark.parametrize("integrator", [0, 1, 2])
def test_batches_of_either_schedule(integrator):
    """A scene's image is the same in a batch most of whose scenes look across the
    grooves (cut tasks) and in one of scenes that do not (uncut), and after an
    update from the one to the other."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt

    def scene(q, az):
        return inputs.base_scene(width=112, height=80, spp=4, precision=0, integrator=integrator, rtol=1e-5, atol=1e-5,
                                 seed=q, E=32.0, cam_dist=40.0, elev_deg=14.0, azim_deg=az)

    across = [scene(q, az) for q, az in enumerate((90.0, 80.0, 75.0))]
    along = [scene(10 + q, az) for q, az in enumerate((0.0, 4.0, -7.0))]
    sets = {"cut": across + along[:1], "uncut": across[:1] + along, "cut again": across + along[:1]}
    scenes = [rt.Scene(p) for p in sets["cut"]]
    b = rt.Batch(scenes)
    out = {}
    for name, ps in sets.items():
        b.update(ps)
        img = [torch.zeros(sc.shape, dtype=torch.float32, device="cuda") for sc in scenes]
        b.render(img)
        assert b.stats()["sched_timeouts"] == 0
        out[name] = img
    b.close()
    assert torch.equal(out["cut"][0], out["uncut"][0]) and torch.equal(out["cut"][3], out["uncut"][1])
    assert all(torch.equal(x, y) for x, y in zip(out["cut"], out["cut again"]))


def test_served_views_across_the_grooves():
    """Requests that look across the grooves, then along them, then across again:
    the images of the scenes alone."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    ps = [inputs.base_scene(width=120 + q, height=88, spp=4, precision=0, seed=30 + q, azim_deg=az)
          for q, az in enumerate((90.0, 85.0, 78.0, 0.0, 3.0, 1.0, 88.0, 90.0))]
    s = rt.Server(1 << 28, max_inflight=2)
    out = [torch.zeros((p["height"], p["width"], 3), dtype=torch.float32, device="cuda") for p in ps]
    tickets = [s.submit(p, t) for p, t in zip(ps, out)]
    for t in tickets:
        while s.poll(t, 1_000_000) is None:
            pass
    s.close()
    for p, t in zip(ps, out):
        sc = rt.Scene(p)
        ref = torch.zeros_like(t)
        sc.render(ref)
        torch.cuda.synchronize()
        assert torch.equal(t, ref)


@pytest.mark.parametrize("over", [dict(E=12.0, elev_deg=20.0), dict(E=32.0, elev_deg=10.0, cam_dist=40.0),
                                  dict(E=32.0, elev_deg=8.0, cam_dist=40.0, integrator=1)])
def test_served_across_a_long_box(over):
    """Requests across the grooves of a long box, in flight by themselves (tasks
    are cut) and beside one along them (tasks run uncut): the same images."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    ps = [inputs.base_scene(width=100 + q, height=72, spp=3, precision=0, seed=50 + q, azim_deg=90.0 - 4 * q, **over)
          for q in range(3)]
    along = inputs.base_scene(width=256, height=256, spp=16, precision=0, seed=60, azim_deg=0.0)
    got = []
    for first in ([], [along]):
        s = rt.Server(1 << 28, max_inflight=2)
        out = [torch.zeros((p["height"], p["width"], 3), dtype=torch.float32, device="cuda") for p in first + ps]
        tickets = [s.submit(p, t) for p, t in zip(first + ps, out)]
        for t in tickets:
            while s.poll(t, 1_000_000) is None:
                pass
        s.close()
        got.append(out[len(first):])
    for a, b in zip(*got):
        assert float(a.abs().sum()) > 0.0
        assert torch.equal(a, b)


@pytest.mark.parametrize("over", [
    dict(precision=0), dict(precision=1), dict(precision=1, A=0.06), dict(precision=0, integrator=1),
    dict(precision=1, integrator=1),
])
def test_set_launch_keeps_min_active(over):
    """min_active 0 keeps the current one, also where the variant changes."""
    pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    sc = rt.Scene(inputs.base_scene(width=16, height=16, **over))
    first = sc.get_launch()["min_active"]
    sc.set_launch(0, 0)
    assert sc.get_launch()["min_active"] == first
    sc.set_launch(3, 0)
    assert sc.get_launch()["min_active"] == first
    sc.set_launch(-1, 19)
    sc.set_launch(0, 0)
    assert sc.get_launch()["min_active"] == 19


TUNE = """
import torch
from paper_1012_5107_gb300 import inputs, rt
for over in (dict(), dict(A=0.06), dict(integrator=1), dict(integrator=1, rtol=1e-4, atol=1e-4)):
    p = inputs.base_scene(width=24, height=20, spp=1, precision=1, **over)
    sc = rt.Scene(p)
    print(sc.autotune(torch.zeros(sc.shape, dtype=torch.float32, device="cuda"), trials=1)["variant"])
    b = rt.Batch([sc])
    b.autotune([torch.zeros(sc.shape, dtype=torch.float32, device="cuda")], trials=1)
"""


def test_tuned_choices_are_kept_apart(tmp_path):
    """Scenes that take different FP64 steps are tuned apart, and choices that a
    file holds from an earlier build's kernels are left alone and not taken."""
    pytest.importorskip("torch")
    cache = tmp_path / "tune"
    old = ["batch/p1/i0/n1 0 13", "batch/p1/i1/n1 0 13", "scene/p1/i0/c1/m1/f0/log2n8 0 13", "scene/p1/i1/c1/m1/f0/log2n8 0 13"]
    cache.write_text("\n".join(old) + "\n")
    run = subprocess.run([sys.executable, "-c", TUNE], cwd=ROOT, capture_output=True, text=True, timeout=300,
                         env=dict(os.environ, RT_AUTOTUNE_CACHE=str(cache)))
    assert run.returncode == 0, run.stderr[-2000:]
    lines = cache.read_text().split("\n")
    new = [x for x in lines if x and x not in old]
    assert all(x in lines for x in old) and len(new) == 8
    assert not any(x.endswith(" 13") for x in new)
