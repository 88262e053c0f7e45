"""rt_xcorr over the ranges its three-float sums take and past them (where a
block sums in FP64), and its column tiles, against Eqs. 14-15 in FP64."""
import math
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def columns(W, hfov, fov):
    px = 2.0 * (np.arange(W) + 0.5) / W - 1.0
    a = np.degrees(np.arctan(np.abs(px) * math.tan(math.radians(0.5 * hfov))))
    return np.nonzero(a <= 0.5 * fov + 1e-9)[0]


def c00(f, g, cols):
    f, g = f[:, cols].astype(np.float64), g[:, cols].astype(np.float64)
    f, g = f - f.mean((0, 1)), g - g.mean((0, 1))
    num, den = (f * g).sum((0, 1)), (f * f).sum((0, 1))
    return np.append(num / den, num.sum() / den.sum())


# FP64 moments of N values lose about N^(1/2) 1e-16 times the ratio of the
# mean square to the variance (at most 1e2 here): 1e-11 covers the largest.
@pytest.mark.parametrize("H,W,C,scale", [
    (512, 512, 3, 1.0), (7, 9721, 3, 1.0), (1, 9999, 4, 1.0), (2000, 22, 3, 1.0), (1030, 65, 1, 1.0),
    (33, 9729, 1, 1.0),                                  # one column past kXcorrBlocks tiles of 32
    (96, 70, 2, 2.0 ** -39), (96, 70, 2, 2.0 ** 59),     # the edges of the three-float range
    (96, 70, 2, 1e-30), (96, 70, 2, 1e25),               # products past FP32's range: FP64
])
def test_xcorr_ranges(H, W, C, scale):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    rng = np.random.default_rng([H, W, C])
    f = (np.round(4.0 * rng.random((H, W, C))) * 0.25 + 0.1 * rng.random((H, W, C))).astype(np.float32)
    g = (0.7 * f + 0.3 * rng.random((H, W, C))).astype(np.float32)
    f[0, 0, 0] = 0.0
    f, g = (f * np.float32(scale)).astype(np.float32), (g * np.float32(scale)).astype(np.float32)
    fovs = [0.0, 10.0, 25.0, 50.0]
    tf, tg = torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()
    out = rt.xcorr(tf, tg, fovs, 50.0).cpu().numpy()
    again = rt.xcorr(tf, tg, fovs, 50.0).cpu().numpy()
    assert np.array_equal(out, again, equal_nan=True)
    for q, fov in enumerate(fovs):
        cols = columns(W, 50.0, fov)
        if H * len(cols) > 1:                            # one pixel has no variance: 0/0
            assert np.abs(out[q] - c00(f, g, cols)).max() < 1e-11
        else:
            assert np.isnan(out[q]).all()


def test_xcorr_infinities_and_nan():
    """A value that is not finite spoils its own windows and channel only, as FP64 sums do."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    rng = np.random.default_rng(3)
    f, g = (rng.random((64, 96, 3)).astype(np.float32) for _ in range(2))
    g[5, 0, 1] = np.inf                                 # outside the inner window
    f[9, 95, 2] = np.nan
    out = rt.xcorr(torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda(), [10.0, 50.0], 50.0).cpu().numpy()
    assert np.isfinite(out[0]).all()
    assert np.isfinite(out[1, 0]) and not np.isfinite(out[1, 1]) and np.isnan(out[1, 2]) and not np.isfinite(out[1, 3])


CAPTURE = """
import sys
import torch
from paper_1012_5107_gb300 import rt
torch.manual_seed(3)
f = torch.rand(200, 180, 3, device="cuda")
g = torch.rand(200, 180, 3, device="cuda")
out = torch.empty((3, 4) if sys.argv[1] == "xcorr" else (13, 13, 4), dtype=torch.float64, device="cuda")
peak = torch.empty(3, dtype=torch.float64, device="cuda")
def call(stream):
    if sys.argv[1] == "xcorr":
        rt.xcorr(f, g, [10.0, 25.0, 50.0], 50.0, out=out, stream=stream)
    else:
        rt.xcorr_map([(f, g)], 40.0, 50.0, 6, 6, out=out, peak=peak, stream=stream)
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, capture_error_mode=sys.argv[2]):
    call(torch.cuda.current_stream().cuda_stream)
out.zero_()
graph.replay()
graph.replay()
torch.cuda.synchronize()
replayed = out.clone()
call(None)
torch.cuda.synchronize()
assert bool(replayed.ne(0).any()) and torch.equal(replayed, out)
"""


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("what", ["xcorr", "map"])
def test_first_call_under_capture(what, mode):
    """The process's first correlation may be one that a stream capture records."""
    pytest.importorskip("torch")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", CAPTURE, what, mode], cwd=root, capture_output=True, text=True,
                         timeout=300)
    assert run.returncode == 0, run.stderr[-2000:]


# The largest values whose products FP32 holds, over chunks of more rows than
# FP32 holds sums of (2^128 / 2^120 = 256), and the edge of the three-float
# range.  The tolerance is test_xcorr_ranges'.
@pytest.mark.parametrize("H,W,C,scale", [
    (1200, 9729, 1, 2.0 ** 59.9),                        # one chunk of all rows (W C >= 9728)
    (2160, 3840, 3, 2.0 ** 59.9), (1080, 1920, 3, 2.0 ** 48), (700, 9728, 1, 2.0 ** 47.9),
    (4096, 70, 1, 2.0 ** 59.9),
])
def test_xcorr_tall_chunks_of_large_values(H, W, C, scale):
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    rng = np.random.default_rng([H, W, C, 1])
    f = (0.5 + 0.5 * rng.random((H, W, C))).astype(np.float32)
    g = (0.7 * f + 0.3 * rng.random((H, W, C))).astype(np.float32)
    f, g = (f * np.float32(scale)).astype(np.float32), (g * np.float32(scale)).astype(np.float32)
    tf, tg = torch.from_numpy(f).cuda(), torch.from_numpy(g).cuda()
    ref = [c00(f, g, columns(W, 50.0, fov)) for fov in (25.0, 50.0)]
    for call in (rt.xcorr, rt.xcorr_noalloc):
        out = call(tf, tg, [25.0, 50.0], 50.0).cpu().numpy()
        assert np.abs(out - np.array(ref)).max() < 1e-11


def test_maps_of_two_threads_at_once():
    """Calls of one tile kernel whose plans need 92 KB and 13 KB of shared memory,
    on two threads and streams, give what they give alone."""
    torch = pytest.importorskip("torch")
    import threading

    from paper_1012_5107_gb300 import rt
    torch.manual_seed(5)
    sizes = [(96, 96, 3, 64, 1), (200, 300, 1, 1, 40)]
    pairs = [(torch.rand(H, W, C, device="cuda"), torch.rand(H, W, C, device="cuda")) for H, W, C, _, _ in sizes]
    alone = [rt.xcorr_map([p], 50.0, 50.0, di, dj)[0].cpu() for p, (_, _, _, di, dj) in zip(pairs, sizes)]
    errors = []

    def work(q):
        try:
            stream = torch.cuda.Stream()
            out = torch.empty_like(alone[q], device="cuda")
            peak = torch.empty(3, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            for _ in range(4000):
                rt.xcorr_map([pairs[q]], 50.0, 50.0, sizes[q][3], sizes[q][4], out=out, peak=peak, stream=stream)
            stream.synchronize()
            assert torch.equal(alone[q], out.cpu())
        except Exception as e:                           # noqa: BLE001 (reported by the test's own thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(q,)) for q in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


def test_scratch_is_given_back():
    """The memory that the correlation calls keep goes back on request, and the
    next calls are as before."""
    torch = pytest.importorskip("torch")
    from paper_1012_5107_gb300 import rt
    torch.manual_seed(6)
    f, g = torch.rand(600, 640, 3, device="cuda"), torch.rand(600, 640, 3, device="cuda")
    out, peak = rt.xcorr_map([(f, g)], 50.0, 50.0, 20, 20)
    first = out.clone()
    torch.cuda.synchronize()
    rt.trim_scratch()
    free = torch.cuda.mem_get_info()[0]
    rt.xcorr_map([(f, g)], 50.0, 50.0, 20, 20, out=out, peak=peak)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] > 1 << 20            # some 10 MB are kept
    rt.trim_scratch()
    assert free - torch.cuda.mem_get_info()[0] < 1 << 20
    rt.xcorr_map([(f, g)], 50.0, 50.0, 20, 20, out=out, peak=peak)
    rt.trim_scratch()                                               # with the call in flight
    torch.cuda.synchronize()
    assert torch.equal(out, first)
