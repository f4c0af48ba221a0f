"""The fixed-point transforms of the complex128 form (wp_fx.h) as the passes take their lines
through them, at every length of a pass, and as the resident lines do, at every length of
those (tests/fx_pass_host.cpp): against numpy's extended-precision FFT (eq. (ft), Sec. 2.1 of
arXiv:1306.3247). Lines whose parts all lie just below a power of two have the largest line
sum that the 32-bit sums must hold. Bound: 2e-16 relative in 2-norm for a transform (three
units of 2^-61 S for the last stage, S at most 1.6 sqrt(n / 2) times the 2-norm of a line of
noise, a tenth more for the stages before, and the rounding to double), and twice that for a
transform and back with the line stored in between."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fxp") / "fx_pass_host")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_1306_3247_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "fx_pass_host.cpp"), "-o", exe],
                   check=True)

    def run(cmd, x):
        inp = struct.pack("ii", cmd, int(np.log2(len(x)))) + np.ascontiguousarray(x, np.complex128).tobytes()
        return np.frombuffer(subprocess.run([exe], input=inp, capture_output=True, check=True).stdout, np.complex128)

    return run


def lines(n, rng):
    below = 1.0 - 2.0 ** -53
    sign = rng.choice([-1.0, 1.0], n) + 1j * rng.choice([-1.0, 1.0], n)
    for name, c in (("1 - 2^-53", below), ("0.9999999", 0.9999999), ("1", 1.0), ("2^-900", 2.0 ** -900 * below)):
        yield name, np.full(n, c * (1 + 1j))
        yield name + ", negative", np.full(n, -c * (1 + 1j))
        yield name + ", signs", c * sign
    yield "noise", rng.standard_normal(n) + 1j * rng.standard_normal(n)
    yield "impulse", np.where(np.arange(n) == n // 3, 1.0 - 0.5j, 0.0)


def rel(got, ref):
    s = np.max(np.abs(ref))
    return float(np.linalg.norm((got - ref) / s) / np.linalg.norm(ref / s))


@pytest.mark.parametrize("logn", range(5, 12))
def test_passes(fx, logn):
    n = 1 << logn
    for name, x in lines(n, np.random.default_rng(logn)):
        assert rel(fx(0, x), np.fft.fft(x.astype(np.clongdouble))) < 2e-16, name
        assert rel(fx(1, x), n * x.astype(np.clongdouble)) < 4e-16, name


@pytest.mark.parametrize("logn", range(8, 14))
def test_resident_lines(fx, logn):
    for name, x in lines(1 << logn, np.random.default_rng(logn)):
        assert rel(fx(2, x), np.fft.fft(x.astype(np.clongdouble))) < 2e-16, name


@pytest.mark.parametrize("logn", range(5, 12))
def test_stored_points(fx, logn):
    """A stored point keeps 57 bits of its own size (half the range of the six code bits of a
    number with its leading bit at 62), whatever its neighbours', above the 62 bits of the
    line; 2^-53 for the doubles it is read back as."""
    n, rng = 1 << logn, np.random.default_rng(logn)
    x = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 2.0 ** rng.uniform(-40, 0, n)
    err = np.abs(fx(3, x).astype(np.clongdouble) - x)
    assert np.all(err < 2.0 ** -52 * np.abs(x) + 2.0 ** -61 * np.max(np.abs(x)))
