"""The fixed-point arithmetic of the complex128 transforms (wp_fx.h), compiled for the host
and driven as the device passes drive it (tests/fx_host.cpp): transforms of every length
the passes and the resident lines take against numpy's extended-precision FFT (the DFT
behind the Fourier transforms of eq. (ft), Sec. 2.1), products with unit factors, and the
stored fixed-point form. Bounds, relative in 2-norm: the transform's own rounding is a few
units of 2^-62 min(q M, S) per stage, at most 1e-16 for any line of these lengths, plus the
rounding of the result to double (2^-53 / sqrt(3) for the mean, 6.5e-17)."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1306_3247_gb300", "csrc")


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fx") / "fx_host")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "fx_host.cpp"), "-o", exe], check=True)

    def run(cmd, n, *arrays):
        inp = struct.pack("ii", cmd, n) + b"".join(np.ascontiguousarray(a, np.complex128).tobytes() for a in arrays)
        out = subprocess.run([exe], input=inp, capture_output=True, check=True).stdout
        return np.frombuffer(out, dtype=np.complex128)

    return run


def lines(n, rng):
    x = np.arange(n)
    u = (x - 0.4 * n) / (0.05 * n)
    yield "packet", np.exp(-u * u + 1j * 0.9 * x)
    yield "noise", rng.standard_normal(n) + 1j * rng.standard_normal(n)
    yield "impulse", np.where(x == n // 3, 1.0 - 0.5j, 0.0)
    yield "plane wave", np.exp(2j * np.pi * 5 * x / n)
    yield "many magnitudes", (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 10.0 ** rng.uniform(-300, 0, n)
    yield "small", 1e-290 * (rng.standard_normal(n) + 1j * rng.standard_normal(n))
    yield "large", 1e290 * (rng.standard_normal(n) + 1j * rng.standard_normal(n))


@pytest.mark.parametrize("logn", range(6, 14))
def test_transform(fx, logn):
    n = 1 << logn
    for name, x in lines(n, np.random.default_rng(logn)):
        ref = np.fft.fft(x.astype(np.clongdouble))
        got = fx(0, logn, x)
        scale = np.max(np.abs(ref))
        err = np.linalg.norm((got - ref) / scale) / np.linalg.norm(ref / scale)
        assert err < 1.65e-16, (name, float(err))


def test_unit_factors(fx):
    rng = np.random.default_rng(3)
    n = 4096
    th = np.concatenate([rng.uniform(-np.pi, np.pi, n - 8), np.arange(8) * np.pi / 4])
    w = np.cos(th) + 1j * np.sin(th)
    v = rng.standard_normal(n) + 1j * rng.standard_normal(n)
    got, ref = fx(1, n, w, v), v.astype(np.clongdouble) * w.astype(np.clongdouble)
    # nine units of 2^-60 of the largest input, and the rounding to double
    assert np.max(np.abs(got - ref)) < 9 * 2.0 ** -60 * np.max(np.abs(v)) * 2 + 2.0 ** -52 * np.max(np.abs(ref))


def test_stored_form(fx):
    rng = np.random.default_rng(4)
    n = 4096
    v = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 10.0 ** rng.uniform(-12, 0, n)
    got = fx(2, n, v)
    # half the range of the six code bits of a number that uses 61 bits, and the rounding
    assert np.max(np.abs(got - v)) < 2.0 ** -54 * np.max(np.abs(v)) + 2.0 ** -53 * np.max(np.abs(v))
    assert abs(np.mean(np.real(got - v))) < 2.0 ** -57 * np.max(np.abs(v))
