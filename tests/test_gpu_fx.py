"""The fixed-point kernels of the complex128 form: transforms of every line length on both
kinds of axis against numpy (unnormalised, eq. (ft) of Sec. 2.1), with values near the ends
of a double's range, empty lines and lines that are not finite; short runs in both orders
against the oracle, which take every pass kind (the state stays in fixed point between the
passes of a step); resident 1-D lines of every length. Transforms agree with numpy's FP64
ones to the sum of both roundings, 2^-53 sqrt(2 log2 N) relative in 2-norm for numpy's
radix-2 count and 2e-16 per axis here; runs of at most 30 steps to 1e-13."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1306_3247_gb300 import wavepacket as WPK

pytestmark = pytest.mark.gpu


def rel_l2(a, b):
    s = np.max(np.abs(b))
    return float(np.linalg.norm(np.ravel(a / s - b / s)) / np.linalg.norm(np.ravel(b / s)))


def problem(n, order="vkv", dt=0.01):
    nd = len(n)
    return {"ndim": nd, "n": list(n), "xmin": [-5.0, -6.0, -4.0][:nd], "L": [10.0, 12.0, 8.0][:nd], "mass": 0.9,
            "hbar": 1.1, "dt": dt, "t0": 0.3, "order": order}


SHAPES = [(64, 1024), (1024, 64), (128, 512), (512, 128), (256, 256), (64, 128, 64), (64, 64, 256)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("scale", [1.0, 1e-292, 1e285])
def test_transform(shape, scale):
    rng = np.random.default_rng(sum(shape))
    x = (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) * scale
    x[3] = 0.0  # empty lines
    x[5] *= 1e-13
    tol = 2.0 ** -53 * np.sqrt(2 * np.log2(x.size)) + 2e-16 * len(shape)
    with WPK.Propagator(problem(shape), [], "c128") as P:
        for sign, ref in ((-1, np.fft.fftn(x)), (1, np.fft.ifftn(x) * x.size)):
            P.set_state(x)
            P.fft(sign)
            assert rel_l2(P.get_state(), ref) < tol
        P.set_state(np.zeros(shape, complex))
        P.fft(-1)
        assert not np.any(P.get_state())
        x.flat[x.size // 3] = np.inf
        P.set_state(x)
        P.fft(-1)
        assert np.all(np.isnan(P.get_state()))


TERMS = {
    "additive": lambda nd: [{"shape": "quad", "a": [1.0, 0.7, 1.3][:nd], "coef": {"A0": 1.0}},
                            {"shape": "linear", "a": [0.4, 0.2, 0.0][:nd], "coef": {"A": 1.0, "omega": 1.7}}],
    "gauss": lambda nd: [{"shape": "gauss", "a": [1.0, 1.5, 1.2][:nd], "c0": [0.5, -0.2, 0.1][:nd],
                          "coef": {"A0": 1.5, "A": 0.4, "omega": 2.0}}],
    "both": lambda nd: [{"shape": "quad", "a": [0.5] * nd, "coef": {"A0": 1.0}},
                        {"shape": "gauss", "a": [0.8] + [0.0] * (nd - 1), "v": [0.7, 0.0, 0.0][:nd], "coef": {"A0": 2.0}},
                        {"shape": "gauss", "a": [0.0] * (nd - 1) + [1.1], "coef": {"A0": -0.7}}],
}


@pytest.mark.parametrize("order", ["vkv", "kvk"])
@pytest.mark.parametrize("pot", list(TERMS))
@pytest.mark.parametrize("shape", [(64, 1024), (512, 128), (64, 128, 64), (256,), (512,), (1024,), (2048,), (4096,), (8192,)])
def test_runs(shape, pot, order):
    nd = len(shape)
    pb, terms = problem(shape, order), TERMS[pot](nd)
    psi0 = O.gaussian(pb, [0.3, -0.4, 0.2][:nd], [1.0, -0.5, 0.3][:nd], [1.0, 0.8, 0.9][:nd])
    ref, ref_obs = O.run(pb, terms, psi0, 30, 15)
    with WPK.Propagator(pb, terms, "c128", autocorr=True) as P:
        P.set_state(psi0)
        obs = WPK.obs_matrix(P.run(30, 15))
        assert rel_l2(P.get_state(), ref) < 1e-13
        P.set_state(psi0)
        P.step_index = 0
        P.step(30)  # without records
        assert rel_l2(P.get_state(), ref) < 1e-13
    scale = np.maximum(np.max(np.abs(ref_obs), axis=0), 1.0)
    assert np.max(np.abs(obs[:, :14] - ref_obs[:, :14]) / scale[:14]) < 1e-12


@pytest.mark.parametrize("shape", [(1024,), (64, 128), (64, 64, 64)])
def test_not_finite(shape):
    # a factor that is not finite (the well's exponential overflows on part of the grid)
    nd = len(shape)
    pb = problem(shape)
    terms = [{"shape": "morse", "a": [1.0, 300.0, 0.0], "coef": {"A0": 1.0}}]
    with WPK.Propagator(pb, terms, "c128") as P:
        P.init_gaussian([0.0] * nd, [0.0] * nd, [1.0] * nd)
        with pytest.raises(WPK.WavepacketError) as e:
            P.run(4, 4)
        assert e.value.status == WPK.WP_ENONFINITE
    # a state that is not finite
    with WPK.Propagator(pb, [], "c128") as P:
        x = np.ones(shape, complex)
        x.flat[7] = np.nan
        P.set_state(x)
        with pytest.raises(WPK.WavepacketError):
            P.run(4, 4)
        assert np.all(np.isnan(P.get_state()))


@pytest.mark.parametrize("prec,tol", [("c128", 1e-13), ("c64", 1e-5), ("c128f", 1e-11)])
@pytest.mark.parametrize("shape", [(32, 64), (64, 32), (32, 2048), (2048, 64), (2048, 4), (4, 2048), (32, 64, 64),
                                   (128, 32, 64), (64, 64, 32)])
def test_axes_of_32_and_2048(shape, prec, tol):
    """The shortest and longest compile-time lines: transforms, and runs with records (formed
    by the run-time kernels at these lengths) and without."""
    nd = len(shape)
    rng = np.random.default_rng(sum(shape))
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    pb, terms = problem(shape), TERMS["both"](nd)
    psi0 = O.gaussian(pb, [0.3, -0.4, 0.2][:nd], [1.0, -0.5, 0.3][:nd], [1.0, 0.8, 0.9][:nd])
    ref, ref_obs = O.run(pb, terms, psi0, 30, 15)
    with WPK.Propagator(pb, terms, prec) as P:
        P.set_state(x)
        P.fft(-1)
        assert rel_l2(P.get_state(), np.fft.fftn(x)) < (1e-15 if prec == "c128" else tol)
        P.set_state(psi0)
        obs = WPK.obs_matrix(P.run(30, 15))
        assert rel_l2(P.get_state(), ref) < tol
        P.set_state(psi0)
        P.step_index = 0
        P.step(30)
        alone = P.get_state()
        assert rel_l2(alone, ref) < tol
    scale = np.maximum(np.max(np.abs(ref_obs), axis=0), 1.0)
    assert np.max(np.abs(obs[:, :14] - ref_obs[:, :14]) / scale[:14]) < 10 * tol
    if nd == 2:
        with WPK.Batch(prec) as B:
            B.add(pb, terms)
            B.set_state(0, psi0)
            B.step(30)
            assert np.array_equal(alone, B.get_state(0))
