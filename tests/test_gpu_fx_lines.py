"""The accuracy of the complex128 passes is that of each line by itself, as in FP64: lines far
smaller than their neighbours in a tile keep their digits, and a line that is all zero is only
as finite as its factors. The large lines here are constant, so that their transforms are one
point and exact zeros, and every other line of every pass holds small values only. Transforms
against numpy on the small part, 2^-53 sqrt(2 log2 N) relative in 2-norm for numpy's rounding
and 2e-16 per axis."""
import numpy as np
import pytest

from paper_1306_3247_gb300 import wavepacket as WPK

pytestmark = pytest.mark.gpu

SHAPES = [(32, 64), (64, 32), (128, 64), (64, 128), (256, 256), (512, 128), (128, 512), (1024, 64), (64, 1024),
          (2048, 32), (32, 2048), (64, 128, 64), (32, 64, 128)]


def problem(n):
    return {"ndim": len(n), "n": list(n), "xmin": [-5.0] * len(n), "L": [10.0] * len(n), "dt": 0.01}


@pytest.mark.parametrize("small", [1e-25, 1e-250])
@pytest.mark.parametrize("shape", SHAPES)
def test_small_lines_beside_large_ones(shape, small):
    rng = np.random.default_rng(sum(shape))
    x = small * (rng.standard_normal(shape) + 1j * rng.standard_normal(shape))
    rows = [3, 4, shape[0] // 2]
    x[rows] = 0.0
    tol = 2.0 ** -53 * np.sqrt(2 * np.log2(x.size)) + 2e-16 * len(shape)
    rest = np.ones(shape, bool)  # away from the lines that the constant reaches
    rest[(slice(None),) + (0,) * (len(shape) - 1)] = False
    with WPK.Propagator(problem(shape), [], "c128") as P:
        for sign, ref in ((-1, np.fft.fftn(x / small)), (1, np.fft.ifftn(x / small) * x.size)):
            y = x.copy()
            y[rows] = 1.0 + 0.5j
            P.set_state(y)
            P.fft(sign)
            got = P.get_state()[rest] / small
            assert np.linalg.norm(got - ref[rest]) < tol * np.linalg.norm(ref[rest]), sign


@pytest.mark.parametrize("shape", [(512,), (64, 128), (64, 64, 64)])
def test_zero_state_and_a_factor_that_is_not_finite(shape):
    terms = [{"shape": "morse", "a": [1.0, 300.0, 0.0], "coef": {"A0": 1.0}}]
    with WPK.Propagator(problem(shape), terms, "c128") as P:
        P.set_state(np.zeros(shape, complex))
        P.step(2)
        assert np.all(np.isnan(P.get_state()))
