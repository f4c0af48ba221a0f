"""complex128 states whose parts all lie just below a power of two, uniform or with random
signs: the largest line sums that the fixed-point passes must hold, on 2048-point axes of
both kinds. Transforms against numpy (2^-53 sqrt(2 log2 N) relative in 2-norm for numpy's
rounding and 2e-16 per axis), and runs without and with a potential of value zero, whose
factors are exactly 1, against the free propagation over their time in one step, its phases
reduced in extended precision (30 steps to 1e-13; the oracle's FP64 phases of up to 1800
radians a step are good to a few 1e-12 on these states' full spectrum); the same instance in a
batch bit by bit."""
import numpy as np
import pytest

from paper_1306_3247_gb300 import wavepacket as WPK

pytestmark = pytest.mark.gpu

SHAPES = [(4, 2048), (2048, 64), (64, 2048)]
TERMS = {"free": [], "zero": [{"shape": "const", "coef": {"A0": 0.0}}],
         "pulse over": [{"shape": "linear", "a": [1.0, 0.5],
                         "coef": {"A": 2.0, "omega": 1.3, "env": "sin2", "t0": 50.0, "tau": 10.0}}]}


def states(shape):
    rng = np.random.default_rng(shape[0])
    below = 1.0 - 2.0 ** -53
    signs = rng.choice([-1.0, 1.0], shape) + 1j * rng.choice([-1.0, 1.0], shape)
    return {"1": np.full(shape, 1.0 + 1.0j), "-1": np.full(shape, -1.0 - 1.0j),
            "below 1": np.full(shape, below * (1 + 1j)), "below -1": np.full(shape, -below * (1 + 1j)),
            "signs": below * signs}


def problem(n, order="vkv"):
    return {"ndim": 2, "n": list(n), "xmin": [-5.0, -6.0], "L": [10.0, 12.0], "mass": 0.9, "hbar": 1.1, "dt": 0.01,
            "t0": 0.3, "order": order}


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b)))


def free(pb, x, t):
    th = np.longdouble(0)
    for d, n in enumerate(pb["n"]):
        j = np.arange(n).astype(np.longdouble)
        k = 8 * np.arctan(np.longdouble(1)) / np.longdouble(pb["L"][d]) * np.where(j < n // 2, j, j - n)
        th = th + (k * k).reshape([-1 if e == d else 1 for e in range(2)])
    th = th * np.longdouble(t) * np.longdouble(pb["hbar"]) / (2 * np.longdouble(pb["mass"]))
    return np.fft.ifftn(np.fft.fftn(x) * (np.cos(th) - 1j * np.sin(th)).astype(complex))


@pytest.mark.parametrize("shape", SHAPES)
def test_transform(shape):
    tol = 2.0 ** -53 * np.sqrt(2 * np.log2(np.prod(shape))) + 4e-16
    with WPK.Propagator(problem(shape), [], "c128") as P:
        for name, x in states(shape).items():
            for sign, ref in ((-1, np.fft.fftn(x)), (1, np.fft.ifftn(x) * x.size)):
                P.set_state(x)
                P.fft(sign)
                assert rel_l2(P.get_state(), ref) < tol, (name, sign)


@pytest.mark.parametrize("order", ["vkv", "kvk"])
@pytest.mark.parametrize("pot", list(TERMS))
@pytest.mark.parametrize("shape", SHAPES)
def test_runs(shape, pot, order):
    pb = problem(shape, order)
    with WPK.Propagator(pb, TERMS[pot], "c128") as P, WPK.Batch("c128") as B:
        B.add(pb, TERMS[pot])
        for name, x in states(shape).items():
            ref = free(pb, x, 30 * np.longdouble(pb["dt"]))
            norm = np.linalg.norm(x) * np.sqrt(np.prod(pb["L"]) / x.size)
            P.set_state(x)
            P.step_index = 0
            obs = WPK.obs_matrix(P.run(30, 15))
            assert rel_l2(P.get_state(), ref) < 1e-13, name
            assert np.allclose(obs[:, 1], norm, rtol=1e-13, atol=0.0), name
            P.set_state(x)
            P.step_index = 0
            P.step(30)
            alone = P.get_state()
            assert rel_l2(alone, ref) < 1e-13, name
            B.set_state(0, x)
            WPK.wp_set_step_index(B.handle(0), 0)
            B.step(30)
            assert np.array_equal(B.get_state(0), alone), name
