"""FP64 arithmetic of the kernels against CUDA's own."""
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


def test_quotient_is_the_divide(run):
    a, b = _random(1 << 20, -300, 300, 1), np.abs(_random(1 << 20, -300, 300, 2))
    got, ref = run("quotient", a, b)
    np.testing.assert_array_equal(got, ref)
