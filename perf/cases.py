"""The work a user has this renderer do, as cases that can be timed and checked.

listed() names the cases, draw() gives others of the same ranges, prepare() makes
what a program has in hand before a call (scenes, batches, a server, images on the
GPU), run() is one pass through the public entry points of rt.py, work() the bytes
and operations a pass cannot do without, and exact() the result in 64 bits from
torch alone, where it has one.

The sizes are the synthetic workloads of inputs.py (64 x 64 pixel centres, 512 x
512 x 4, 1920 x 1080 x 16 with the Dormand-Prince integrator, the 64 uneven scenes,
the serving mix, the Gaussian bump, Table 1's referenced cloak with Fresnel
weights) and what lies around them.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1012_5107_gb300 import inputs, rt

FOVS = (10.0, 25.0, 50.0)      # Table 1's horizontal fields of view, beside the centre line (0)
HFOV = 50.0
RK4T = 2                       # RT_RK4T: RK4 on Eq. 11 in physical time
REFERENCED, PLATE, FRESNEL = 1, 2, 4


def listed() -> list[dict]:
    return [
        # the smallest call: one frame of a viewer while the camera moves (single precision, pixel centres)
        dict(name="preview_f32_64", kind="render", precision=0, integrator=0, mirror="cloak", width=64, height=64,
             spp=1, E=8.0, H=2.0, A=0.04, elev=30.0, records=False),
        # the plain method in double precision with every ray's exit record: a parity or convergence study
        dict(name="exits_f64_64", kind="render", precision=1, integrator=0, mirror="cloak", width=64, height=64,
             spp=1, E=8.0, H=2.0, A=0.04, elev=30.0, records=True),
        # the workload of Fig. 3 and Table 1: three renders, their centre lines and C(0,0) at 0/10/25/50 degrees
        dict(name="step_f32_512", kind="step", precision=0, side=512, spp=4, A=0.04, elev=30.0),
        # the double precision frame that the single precision one is held against
        dict(name="cloak_f64_512x4", kind="render", precision=1, integrator=0, mirror="cloak", width=512, height=512,
             spp=4, E=8.0, H=2.0, A=0.04, elev=30.0, records=False),
        # a production frame: 1920 x 1080 x 16, Dormand-Prince, textured background
        dict(name="hd_f32_dp45", kind="render", precision=0, integrator=1, mirror="cloak", width=1920, height=1080,
             spp=16, E=8.0, H=2.0, A=0.04, elev=30.0, records=False, texture=2048),
        # the same frame's double precision check on a pixel subset, with exit records
        dict(name="hd_f64_pixels", kind="pixels", integrator=1, width=1920, height=1080, spp=16, E=8.0, A=0.04,
             npix=2500, texture=2048),
        # Table 1, lower half: the referenced cloak and the mirror under a plate, Fresnel weights, and their C
        dict(name="table1_f32_256", kind="table1", side=256, spp=4, H=1.1),
        # Fig. 4(c): the Gaussian bump's cloak, ragged size
        dict(name="gauss_f32_499x511", kind="render", precision=0, integrator=0, mirror="gauss", width=511,
             height=499, spp=4, E=8.0, H=1.1, A=0.13, elev=30.0, records=False),
        # many scenes of uneven size in one launch
        dict(name="batch_f32_64", kind="batch", count=64),
        # a burst of requests to the render server, until the last one is done
        dict(name="serve_f32_12", kind="serve", count=12, max_side=512, max_spp=16),
        # scoring one frame pair: C(0,0) per field of view, full frames and centre lines
        dict(name="score_512", kind="score", height=512, width=512, channels=3),
        # the correlation function over shifts and its peak
        dict(name="map_512", kind="map", height=512, width=512, channels=3, pairs=1, max_di=32, max_dj=32),
    ]


def _logint(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["render32", "render32", "render64", "render64", "gauss", "step", "pixels", "table1", "batch",
                       "serve", "score", "score", "map"])
    A, elev = round(rng.uniform(0.01, 0.04), 4), round(rng.uniform(10.0, 60.0), 2)
    E = rng.choice([2.0, 4.0, 8.0, 16.0, 32.0])
    if kind in ("render32", "render64"):
        f64 = kind == "render64"
        # rays of the two precisions cost about a hundredfold; double precision frames go up to 160 x 160 x 4
        side = _logint(rng, 24, 160 if f64 else 640)
        return dict(kind="render", precision=int(f64), integrator=rng.choice([0, 0, 0, 1, RK4T]),
                    mirror=rng.choice(["cloak", "cloak", "cloak", "bare", "flat"]), width=side,
                    height=max(16, int(side * rng.uniform(0.5, 1.0))), spp=rng.choice([1, 2, 4] if f64 else [1, 3, 4, 16]),
                    E=E, H=rng.choice([2.0, 2.0, 1.1, 0.55]), A=A, elev=elev, records=bool(f64),
                    texture=rng.choice([0, 512]))
    if kind == "gauss":
        side = _logint(rng, 48, 512)
        return dict(kind="render", precision=0, integrator=rng.choice([0, 0, 1]), mirror="gauss", width=side,
                    height=max(32, int(side * rng.uniform(0.5, 1.0))), spp=rng.choice([1, 4]), E=8.0, H=1.1, A=0.13,
                    elev=elev, records=False)
    if kind == "step":
        return dict(kind="step", precision=0, side=_logint(rng, 64, 512), spp=rng.choice([1, 4]), A=A, elev=elev)
    if kind == "pixels":
        return dict(kind="pixels", integrator=rng.choice([0, 1]), width=rng.choice([512, 960, 1920]), height=540,
                    spp=rng.choice([1, 4, 16]), E=E, A=A, npix=_logint(rng, 64, 2500), texture=rng.choice([0, 512]))
    if kind == "table1":
        return dict(kind="table1", side=_logint(rng, 32, 256), spp=rng.choice([1, 4]), H=rng.choice([1.1, 0.55, 0.41]))
    if kind == "batch":
        return dict(kind="batch", count=_logint(rng, 2, 40))
    if kind == "serve":
        return dict(kind="serve", count=rng.randint(1, 24), max_side=rng.choice([256, 512]), max_spp=rng.choice([4, 16]))
    if kind == "score":
        return dict(kind="score", height=_logint(rng, 32, 1440), width=_logint(rng, 32, 2560),
                    channels=rng.choice([1, 3, 3]))
    return dict(kind="map", height=_logint(rng, 48, 512), width=_logint(rng, 48, 512), channels=rng.choice([1, 3]),
                pairs=rng.choice([1, 2]), max_di=rng.randint(0, 40), max_dj=rng.randint(1, 40))


# ---------------------------------------------------------------------------
# What a program has before the call.
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _noise(size: int) -> np.ndarray:
    return inputs.value_noise(size, seed=3, base_period=min(256, size // 2))


def _texture(size: int, seed: int) -> np.ndarray | None:
    """The periodic value noise, moved by a seeded shift (another photograph)."""
    if not size:
        return None
    rng = np.random.default_rng([seed, 0x7E])
    return np.roll(_noise(size), tuple(int(v) for v in rng.integers(0, size, 2)), (0, 1))


def _params(case: dict, seed: int, **over) -> dict:
    """Scene parameters of a case: its geometry, with the seed's sample jitter, colours and a camera azimuth
    within two degrees."""
    rng = np.random.default_rng([seed, 0xCA5E])
    f32 = case.get("precision", 0) == 0
    mirror = case.get("mirror", "cloak")
    rtol = 1e-5 if f32 else 1e-7
    p = dict(width=case.get("width", 64), height=case.get("height", 64), spp=case.get("spp", 1), seed=seed,
             precision=case.get("precision", 0), integrator=case.get("integrator", 0), E=case.get("E", 8.0),
             H=case.get("H", 2.0), A=case.get("A", 0.04), elev_deg=case.get("elev", 30.0),
             azim_deg=float(rng.uniform(-2.0, 2.0)), rtol=rtol, atol=rtol)
    if case.get("texture"):
        p.update(background=inputs.TEXTURE, tex_size=case["texture"])
    p.update(over)
    if mirror == "gauss":
        return inputs.gauss_scene(**p)
    q = inputs.base_scene(**p)
    if mirror == "flat":
        q.update(mirror=inputs.FLAT, cloak=0)
    elif mirror == "bare":
        q.update(cloak=0)
    return q


def _seeded(p: dict, seed: int) -> dict:
    """One of the uneven scenes with the seed's jitter, colours and a camera azimuth within two degrees."""
    c0, c1 = inputs.checker_colours(p["seed"] + seed)
    azim = p["azim_deg"] + float(np.random.default_rng([p["seed"], seed]).uniform(-2.0, 2.0))
    return dict(p, seed=p["seed"] + seed, colour0=c0, colour1=c1, azim_deg=azim)


def _image(sc) -> torch.Tensor:
    return torch.empty(sc.shape, dtype=torch.float32, device="cuda")


def _frames(h: int, w: int, c: int, seed: int, n: int = 1) -> list[tuple[torch.Tensor, torch.Tensor]]:
    """Pairs of frames as renders give them: two colours in tilted cells, anti-aliased in quarters, and the same
    cells seen through a wavy medium."""
    out = []
    for q in range(n):
        gen = torch.Generator(device="cuda").manual_seed(int(seed) * 64 + q)
        col = torch.rand((2, c), generator=gen, device="cuda")
        ph = torch.rand(6, generator=gen, device="cuda").tolist()
        y = torch.arange(h, device="cuda", dtype=torch.float32)[:, None] / 37.0
        x = torch.arange(w, device="cuda", dtype=torch.float32)[None, :] / 31.0

        def cells(wave: float):
            acc = torch.zeros((h, w), device="cuda")
            for k in range(4):
                xx = x + 0.008 * (k % 2) + wave * torch.sin(9.0 * x + 6.0 * ph[2] + 0.5 * y)
                yy = y + 0.007 * (k // 2) + wave * torch.sin(5.0 * x + 6.0 * ph[3])
                par = torch.floor(xx + 0.11 * yy + ph[0]) + torch.floor(yy - 0.07 * xx + ph[1])
                acc += torch.remainder(par, 2.0)
            t = (acc * 0.25)[..., None]
            return (t * col[0] + (1.0 - t) * col[1]).contiguous()

        out.append((cells(0.0), cells(0.12)))
    return out


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    st: dict = {"case": case, "kind": kind}
    if kind == "render":
        p = _params(case, seed)
        sc = rt.Scene(p, _texture(case.get("texture", 0), seed))
        st.update(scene=sc, rgb=_image(sc))
        if case["records"]:
            st["rec"] = torch.zeros(sc.height * sc.wout * sc.spp * 80, dtype=torch.uint8, device="cuda")
        else:
            st["rgb8"] = torch.empty(sc.shape, dtype=torch.uint8, device="cuda")
    elif kind == "pixels":
        p = _params(dict(case, precision=1), seed)
        pix = inputs.pixel_subset(p["height"], p["width"], case["npix"], seed)
        st.update(scene=rt.Scene(p, _texture(case.get("texture", 0), seed)), pix=torch.from_numpy(pix).cuda(),
                  rgb=torch.empty((len(pix), 3), dtype=torch.float32, device="cuda"),
                  rec=torch.zeros(len(pix) * p["spp"] * 80, dtype=torch.uint8, device="cuda"))
    elif kind == "step":
        p = _params(dict(case, width=case["side"], height=case["side"]), seed)
        scenes = {}
        for name, q in inputs.three_renders(p).items():
            scenes[name] = rt.Scene(q)
            scenes[name + "_line"] = rt.Scene(dict(q, centre_line=1))
        st.update(scenes=scenes, img={k: _image(s) for k, s in scenes.items()}, batch=rt.Batch(list(scenes.values())))
    elif kind == "table1":
        # A = 3 / (16 pi): n / n_min in [1, 2.2]
        base = dict(width=case["side"], height=case["side"], A=3.0 / (16.0 * math.pi))
        cloak = _params(dict(case, **base), seed, flags=REFERENCED | FRESNEL)
        plate = dict(cloak, mirror=inputs.FLAT, cloak=0, flags=PLATE | FRESNEL)
        st["scenes"] = [rt.Scene(cloak), rt.Scene(plate)]
        st["img"] = [_image(s) for s in st["scenes"]]
    elif kind == "batch":
        st["scenes"] = [rt.Scene(_seeded(p, seed)) for p in inputs.batch_scenes(case["count"])]
        st["img"] = [_image(s) for s in st["scenes"]]
        st["batch"] = rt.Batch(st["scenes"])
    elif kind == "serve":
        # the mix of the serving workload, its largest requests left out; all at once
        reqs = inputs.serving_requests(case["count"], max_side=case["max_side"], min_side=64, max_spp=case["max_spp"])
        st["reqs"] = [_seeded(p, seed) for _, p in reqs]
        st["img"] = [torch.empty((p["height"], p["width"], 3), dtype=torch.float32, device="cuda") for p in st["reqs"]]
        st["server"] = rt.Server(1 << 30, max_inflight=2)
    elif kind == "score":
        (f, g), = _frames(case["height"], case["width"], case["channels"], seed)
        mid = case["width"] // 2
        st.update(f=f, g=g, fl=f[:, mid:mid + 1].contiguous(), gl=g[:, mid:mid + 1].contiguous())
    elif kind == "map":
        st["pairs"] = _frames(case["height"], case["width"], case["channels"], seed, case["pairs"])
    return st


def _records(rec: torch.Tensor) -> dict:
    """Exit records as their fields (rt_ray_record, 80 bytes)."""
    r = rec.view(-1, 80)
    return {"exit": r[:, :48].contiguous().view(torch.float64), "rgb": r[:, 48:60].contiguous().view(torch.float32),
            "counts": r[:, 60:72].contiguous().view(torch.int32), "steps": r[:, 72:80].contiguous().view(torch.int64)}


def run(st: dict):
    kind, case = st["kind"], st["case"]
    if kind == "render":
        st["scene"].render(st["rgb"], rgb8=st.get("rgb8"), rec=st.get("rec"))
        if case["records"]:
            return {"image": st["rgb"], "records": _records(st["rec"])}
        return {"image": st["rgb"], "image8": st["rgb8"]}
    if kind == "pixels":
        st["scene"].render_pixels(st["pix"], st["rgb"], rec=st["rec"])
        return {"pixels": st["rgb"], "records": _records(st["rec"])}
    if kind == "step":
        img = st["img"]
        st["batch"].render(list(img.values()))
        c = {}
        for g in ("bare", "cloak"):
            c[g] = rt.xcorr(img["mirror"], img[g], FOVS, HFOV)
            c[g + "_line"] = rt.xcorr(img["mirror_line"], img[g + "_line"], (0.0,), HFOV)
        return {"images": img, "c": c}
    if kind == "table1":
        for s, t in zip(st["scenes"], st["img"]):
            s.render(t)
        return {"cloak": st["img"][0], "plate": st["img"][1], "c": rt.xcorr(st["img"][1], st["img"][0], FOVS, HFOV)}
    if kind == "batch":
        st["batch"].render(st["img"])
        return st["img"]
    if kind == "serve":
        tickets = [st["server"].submit(p, t) for p, t in zip(st["reqs"], st["img"])]
        for t in tickets:
            while st["server"].poll(t, 1_000_000) is None:
                pass
        return st["img"]
    if kind == "score":
        return {"full": rt.xcorr(st["f"], st["g"], FOVS, HFOV), "line": rt.xcorr(st["fl"], st["gl"], (0.0,), HFOV)}
    cm, peak = rt.xcorr_map(st["pairs"], HFOV, HFOV, case["max_di"], case["max_dj"])
    return {"map": cm, "peak": peak}


# ---------------------------------------------------------------------------
# What a pass cannot do without.
# ---------------------------------------------------------------------------
# Integrator steps a camera sample takes on average at box extent E (rt_scene_stats of the synthetic workloads).
_RK4_STEPS = {2.0: 30, 4.0: 120, 8.0: 475, 16.0: 930, 32.0: 1100}
_DP45_STEPS = {2.0: 4, 4.0: 16, 8.0: 63, 16.0: 121, 32.0: 144}
_RK4_FLOP = 385                # per RK4 step: 2 Newton steps on W0, 5 evaluations, the state update
_DP45_FLOP = 700               # per Dormand-Prince attempt: 6 evaluations with their Newton steps


def _render_flops(samples: float, integrator: int, mirror: str, E: float) -> float:
    if mirror in ("bare", "flat"):
        return samples * 600.0
    steps, flop = (_DP45_STEPS, _DP45_FLOP) if integrator == 1 else (_RK4_STEPS, _RK4_FLOP)
    per = steps.get(E, 475) * flop
    if mirror == "gauss":
        per = (253 if integrator != 1 else 40) * (_RK4_FLOP + 400)
    return samples * per


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("render", "pixels"):
        npix = case["npix"] if kind == "pixels" else case["width"] * case["height"]
        samples = npix * case["spp"]
        recs = samples * 80 if kind == "pixels" or case["records"] else 0
        out = npix * (20 if kind == "pixels" else 12 if case["records"] else 15)
        tex = 4 * case.get("texture", 0) ** 2
        return {"bytes": out + recs + min(tex, 64 * samples),
                "flops": _render_flops(samples, case["integrator"], case.get("mirror", "cloak"), case["E"])}
    if kind == "step":
        n = case["side"] ** 2
        samples = (n + case["side"]) * case["spp"]
        return {"bytes": 36 * (n + case["side"]) + 48 * n, "flops": samples * (475 * _RK4_FLOP + 1200.0)}
    if kind == "table1":
        n = case["side"] ** 2
        return {"bytes": 48 * n, "flops": n * case["spp"] * 260.0 * _RK4_FLOP}
    if kind == "batch":
        samples = pixels = 0
        for p in inputs.batch_scenes(case["count"]):
            pixels += p["width"] * p["height"]
            samples += p["width"] * p["height"] * p["spp"]
        return {"bytes": 12 * pixels, "flops": samples * 450.0 * _RK4_FLOP}
    if kind == "serve":
        samples = pixels = 0
        for _, p in inputs.serving_requests(case["count"], max_side=case["max_side"], min_side=64,
                                            max_spp=case["max_spp"]):
            pixels += p["width"] * p["height"]
            samples += p["width"] * p["height"] * p["spp"]
        return {"bytes": 12 * pixels, "flops": samples * 450.0 * _RK4_FLOP}
    values = case["height"] * case["width"] * case["channels"]
    if kind == "score":
        return {"bytes": 8 * (values + case["height"] * case["channels"]) + 128, "flops": 6.0 * values}
    shifts = (2 * case["max_di"] + 1) * (2 * case["max_dj"] + 1)
    return {"bytes": 8 * values * case["pairs"] + 8 * shifts * (case["channels"] + 1),
            "flops": 2.0 * values * case["pairs"] * shifts}


# ---------------------------------------------------------------------------
# The results in 64 bits.  Renders have none here: an independent tracer of
# the cloak's rays takes minutes.
# ---------------------------------------------------------------------------
def _window(w: int, fov: float) -> slice:
    """Columns whose pixel centre lies within the field of view (a width-1 image has its column at angle 0)."""
    px = 2.0 * (np.arange(w) + 0.5) / w - 1.0
    alpha = np.degrees(np.arctan(np.abs(px) * math.tan(math.radians(0.5 * HFOV))))
    j = np.nonzero(alpha <= 0.5 * fov + 1e-9)[0]
    return slice(int(j[0]), int(j[-1]) + 1) if len(j) else slice(0, 0)


def _c00(f: torch.Tensor, g: torch.Tensor, fovs) -> torch.Tensor:
    rows = []
    for fov in fovs:
        s = _window(f.shape[1], fov)
        a, b = f[:, s].double(), g[:, s].double()
        a, b = a - a.mean((0, 1)), b - b.mean((0, 1))
        num, den = (a * b).sum((0, 1)), (a * a).sum((0, 1))
        rows.append(torch.cat([num / den, (num.sum() / den.sum())[None]]))
    return torch.stack(rows)


def exact(case: dict, seed: int):
    if case["kind"] == "score":
        st = prepare(case, seed)
        return {"full": _c00(st["f"], st["g"], FOVS), "line": _c00(st["fl"], st["gl"], (0.0,))}
    if case["kind"] == "map":
        di, dj = case["max_di"], case["max_dj"]
        total = 0.0
        for f, g in _frames(case["height"], case["width"], case["channels"], seed, case["pairs"]):
            a, b = f.double().permute(2, 0, 1), g.double().permute(2, 0, 1)
            a, b = a - a.mean((1, 2), keepdim=True), b - b.mean((1, 2), keepdim=True)
            size = (a.shape[1] + di + 1, a.shape[2] + dj + 1)
            cc = torch.fft.irfft2(torch.fft.rfft2(a, size).conj() * torch.fft.rfft2(b, size), size)
            rows = torch.arange(-di, di + 1, device="cuda") % size[0]
            cols = torch.arange(-dj, dj + 1, device="cuda") % size[1]
            num, den = cc[:, rows][:, :, cols], (a * a).sum((1, 2))
            m = torch.cat([num / den[:, None, None], (num.sum(0) / den.sum())[None]])
            total = total + m.permute(1, 2, 0)
        cm = (total / case["pairs"]).contiguous()
        # the peak's place is not a rounded quantity: its value and shift come from the map
        at = int(torch.argmax(cm[..., -1]))
        v = cm[..., -1].reshape(-1)[at]
        peak = torch.stack([v, torch.tensor(float(at // (2 * dj + 1) - di), dtype=torch.float64, device="cuda"),
                            torch.tensor(float(at % (2 * dj + 1) - dj), dtype=torch.float64, device="cuda")])
        return {"map": cm, "peak": peak}
    return None
