"""The FP64 reciprocal, root and quotient of the kernels against CUDA's own, over
random mantissas and exponents and at the edges of the range."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TINY, HUGE = np.finfo(float).tiny, np.finfo(float).max
EDGES = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 1e-310, TINY, -TINY, 2 * TINY, 2.0**1021,
                  2.0**1022, 2.0**1022 * 1.5, -(2.0**1023), HUGE, -HUGE, 1.0, -1.0, 3.0])


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2112_01349_gb300 import _build

    exe = str(tmp_path_factory.mktemp("math") / "device_math_check")
    cmd = [_build._nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-I", _build.CSRC, "-I",
           os.path.dirname(_build.HEADER), os.path.join(ROOT, "tests", "device_math_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def call(what, a, b):
        data = np.int32(len(a)).tobytes() + np.stack([a, b], 1).tobytes()
        r = subprocess.run([exe, what], input=data, capture_output=True)
        assert r.returncode == 0, r.stderr
        return np.frombuffer(r.stdout).reshape(-1, 2).T

    return call


def _random(n, low, high, seed):
    rng = np.random.default_rng(seed)
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(low, high, n)) * rng.choice([-1.0, 1.0], n)


def _units(got, ref):
    """Distance in units in the last place (same sign, finite)."""
    return np.abs(got.view(np.int64) - ref.view(np.int64))


def test_quotient_is_the_divide(run):
    a, b = _random(1 << 20, -300, 300, 1), np.abs(_random(1 << 20, -300, 300, 2))
    got, ref = run("quotient", a, b)
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("what", ["rcp", "sqrt"])
def test_reciprocal_and_root(run, what):
    """Within one unit in the last place (40- and 80-bit Newton iterates, rounded
    once more), and CUDA's own result at the edges."""
    x = _random(1 << 20, -1021, 1021, 3)
    if what == "sqrt":
        x = np.abs(x)
    got, ref = run(what, x, x)
    assert _units(got, ref).max() <= 1
    got, ref = run(what, EDGES, EDGES)
    exact = ~np.isin(np.abs(EDGES), [1.0, 3.0, TINY, 2 * TINY, 2.0**1021, 2.0**1022, 1.5 * 2.0**1022, 2.0**1023, HUGE])
    np.testing.assert_array_equal(got[exact], ref[exact])
    same = np.isfinite(ref)
    assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(got[~same], ref[~same], equal_nan=True)
    assert _units(got[same], ref[same]).max() <= 1
