"""FP64 batches whose scenes take different steps (rt_split.cuh's within their
bounds, the general one past them): every scene takes the step it takes alone,
also after an update."""
import numpy as np
import pytest

from paper_1012_5107_gb300 import inputs

pytestmark = pytest.mark.gpu
COUNTS = ("rays", "steps", "evals", "newton", "events", "status")


def scene(rt, torch, p):
    sc = rt.Scene(p)
    rgb = torch.zeros(sc.shape, dtype=torch.float32, device="cuda")
    sc.render(rgb)
    st = sc.stats()
    return sc, rgb.cpu().numpy(), [np.array(st[k]) for k in COUNTS]


def params(integrator, spp=4):
    base = dict(precision=1, integrator=integrator, rtol=1e-7, atol=1e-7, spp=spp, seed=3)
    inside = [inputs.base_scene(width=40, height=28, **base),
              inputs.base_scene(width=33, height=20, A=0.02, azim_deg=20.0, **base),
              inputs.base_scene(width=24, height=31, A=0.03, elev_deg=50.0, **base)]
    past = [dict(p, A=0.05 + 0.02 * q) for q, p in enumerate(inside)]       # kA 0.31 ... 0.57
    air = [inputs.three_renders(inside[0])[k] for k in ("bare", "mirror")]
    return inside, past, air


# The solves of W0 that a scene's step counts differ between the two steps, so
# equal sums say that each scene took the step it takes alone.
@pytest.mark.parametrize("integrator", [0, 1])
@pytest.mark.parametrize("spp", [1, 4])
def test_every_scene_takes_its_own_step(integrator, spp):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    inside, past, air = params(integrator, spp)
    sets = [inside + air, [past[0], inside[1], past[2]] + air, [inside[0], past[1], inside[2]] + air, past + air]
    alone = [[scene(rt, torch, p) for p in ps] for ps in sets]
    scenes = [sc for sc, _, _ in alone[1]]
    img = [torch.zeros(sc.shape, dtype=torch.float32, device="cuda") for sc in scenes]
    b = rt.Batch(scenes)
    for k in (1, 0, 2, 3, 1, 3, 0):
        b.update(sets[k])
        for t in img:
            t.fill_(-1.0)
        b.render(img)
        st = b.stats()
        for t, (_, r, _) in zip(img, alone[k]):
            assert np.array_equal(t.cpu().numpy(), r)
        for q, name in enumerate(COUNTS):
            assert np.array_equal(np.array(st[name]), sum(c[q] for _, _, c in alone[k])), name
        assert st["sched_timeouts"] == 0
    b.close()
