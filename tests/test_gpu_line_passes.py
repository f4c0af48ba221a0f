"""Passes over lines of 512 to 2048 points held in registers (complex64, float-float): equal to
the batched kernels of the same instance bit for bit (other tiles, the same stages and factors),
and to the oracle within the forms' bounds (20 steps: complex64 1e-5, float-float 1e-11
relative in 2-norm), for every potential kind, both orders and transforms alone, down to
the fewest columns a block takes."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1306_3247_gb300 import wavepacket as WPK

pytestmark = pytest.mark.gpu

TOL = {"c64": 1e-5, "c128f": 1e-11}
QUAD = {"shape": "quad", "a": [1.0, 0.7, 0.4], "coef": {"A0": 1.0}}
DRIVE = {"shape": "linear", "a": [0.4, 0.2, 0.1], "coef": {"A": 1.0, "omega": 1.7}}
BUMP = {"shape": "gauss", "a": [1.0, 1.5, 1.2], "v": [0.6, 0.0, 0.0], "coef": {"A0": 1.5, "A": 0.4, "omega": 2.0}}
WALL = {"shape": "gauss", "a": [0.0, 1.1, 0.0], "coef": {"A0": -0.7}}


def rel_l2(a, b):
    return float(np.linalg.norm(np.ravel(a - b)) / np.linalg.norm(np.ravel(b)))


def problem(n, order):
    nd = len(n)
    return {"ndim": nd, "n": list(n), "xmin": [-8.0, -7.0, -6.0][:nd], "L": [16.0, 14.0, 12.0][:nd], "mass": 0.9,
            "hbar": 1.1, "dt": 0.01, "t0": 0.3, "order": order}


def cut(terms, nd):
    return [dict(t, **{k: t[k][:nd] for k in ("a", "v") if k in t}) for t in terms]


@pytest.mark.parametrize("prec", ["c64", "c128f"])
@pytest.mark.parametrize("order", ["vkv", "kvk"])
@pytest.mark.parametrize("shape,terms", [((512, 1024), [QUAD, DRIVE]), ((1024, 512), [BUMP]),
                                         ((1024, 64), [QUAD, BUMP]), ((64, 512), [BUMP, WALL]),
                                         ((512, 512), [QUAD, BUMP, WALL]), ((1024, 4), [QUAD]),
                                         ((2048, 64), [QUAD, BUMP, WALL]), ((64, 2048), [BUMP]),
                                         ((2048, 4), [QUAD, DRIVE]), ((4, 2048), [QUAD])])
def test_alone_batched_and_oracle(shape, terms, order, prec):
    pb, terms = problem(shape, order), cut(terms, len(shape))
    psi0 = O.gaussian(pb, [0.5, -0.4], [1.0, -0.5], [1.3, 1.1])
    with WPK.Propagator(pb, terms, prec) as P:
        P.set_state(psi0)
        P.step(20)
        alone = P.get_state()
    with WPK.Batch(prec) as B:
        B.add(pb, terms)
        B.set_state(0, psi0)
        B.step(20)
        assert np.array_equal(alone, B.get_state(0))
    assert rel_l2(alone, O.propagate(pb, terms, psi0, 20)) < TOL[prec]


@pytest.mark.parametrize("prec", ["c64", "c128f"])
@pytest.mark.parametrize("shape", [(512, 32, 64), (32, 1024, 16), (16, 64, 512),
                                   (2048, 8, 16), (8, 2048, 16), (16, 4, 2048)])
def test_three_axes(shape, prec):
    pb, terms = problem(shape, "vkv"), [QUAD, BUMP]
    psi0 = O.gaussian(pb, [0.5, -0.4, 0.2], [1.0, -0.5, 0.0], [1.3, 1.1, 1.6])
    x = np.random.default_rng(3).standard_normal(shape) + 0.5j
    with WPK.Propagator(pb, terms, prec) as P:
        P.set_state(psi0)
        P.step(20)
        assert rel_l2(P.get_state(), O.propagate(pb, terms, psi0, 20)) < TOL[prec]
        P.set_state(x)
        P.fft(-1)
        assert rel_l2(P.get_state(), np.fft.fftn(x)) < TOL[prec]
        P.fft(1)
        assert rel_l2(P.get_state(), x * x.size) < TOL[prec]


@pytest.mark.parametrize("prec,shape", [("c64", (512, 128, 256)), ("c128f", (128, 512, 128))])
def test_states_beyond_64_mb(prec, shape):
    """The strided passes with two sectors of columns a block."""
    pb, terms = problem(shape, "vkv"), [QUAD, BUMP]
    psi0 = O.gaussian(pb, [0.5, -0.4, 0.2], [1.0, -0.5, 0.0], [1.3, 1.1, 1.6])
    with WPK.Propagator(pb, terms, prec) as P:
        P.set_state(psi0)
        P.step(2)
        assert rel_l2(P.get_state(), O.propagate(pb, terms, psi0, 2)) < TOL[prec]
        P.set_state(psi0)
        P.fft(-1)
        assert rel_l2(P.get_state(), np.fft.fftn(psi0)) < TOL[prec]
