"""Rounding of the steps in two and three floats (rt_split.cuh, compiled for the
host) over the range they are used in, against the same methods in 113 bits and in
double: they may be no less accurate than double."""
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1012_5107_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    out = str(tmp_path_factory.mktemp("split") / "split_accuracy")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-x", "c++", "-o", out,
                    os.path.join(HERE, "split_accuracy.cpp")], check=True)
    return out


def errors(program, *args):
    run = subprocess.run([program, *map(str, args)], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.returncode
    e = np.array([[float(x) for x in line.split()] for line in run.stdout.splitlines()])
    assert np.isfinite(e).all()
    return e


def summary(e):
    return np.array([*np.quantile(e, [0.5, 0.9], axis=0), np.sqrt((e ** 2).mean(0))])


# kh 0: the range's edge, the least accurate step it takes; 2 pi / 200 is the
# benchmark's step (in range up to kA = 0.27)
@pytest.mark.parametrize("kA,kh", [(0.003, 0), (0.02, 0), (0.0999, 0), (0.101, 0), (0.2, 0), (0.2513274, 0), (0.2999, 0),
                                   (0.2513274, 0.0314159265), (0.15, 0.0314159265), (0.2999, 0.01)])
def test_rk4_step(program, kA, kh):
    s = summary(errors(program, "rk4", kA, kh, 60, 250))
    assert (s[:, 1] <= s[:, 0]).all(), s


# The stages' W0 in 48 bits adds to the FP64 step's own roundings, 1.6e-16 of
# about ten operations a stage: a quarter more is the most it may come to.
@pytest.mark.parametrize("kA,tol", [(0.02, 1e-6), (0.1, 1e-6), (0.2513274, 1e-6), (0.2799, 1e-6), (0.2513274, 1e-9)])
def test_dormand_prince_step(program, kA, tol):
    s = summary(errors(program, "dp45", kA, 0, 200, 80, tol))
    assert (s[:, 1] <= 1.25 * s[:, 0]).all(), s


def test_range(program):
    """Steps past the range are told."""
    for args in (("rk4", 0.301, 0.001), ("rk4", 0.2997, 0.034), ("rk4", 0.101, 0.0487), ("rk4", 0.1, 0.0563),
                 ("rk4", 0.01, 0.0622), ("dp45", 0.2513, 0.45), ("dp45", 0.281, 0.3)):
        assert subprocess.run([program, *map(str, args), "1", "1"]).returncode == 3
