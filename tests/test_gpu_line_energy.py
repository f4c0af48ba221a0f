"""The potential energy of a 1-D record on boxes far from the origin, with the centres of the
potential's terms near the packet: formed point by point, V(x_i) |psi_i|^2 (Tab. 3 of
arXiv:1306.3247), it is as exact as near the origin. Grid points, centres and the packet's
place are multiples of 1/256 below 2^21, so that x_i - c is exact. Tolerance 1e-13 of the mean
of |V|, FP64 sums of up to 8192 terms; the sums of x |psi|^2 and |psi|^2 cancel to about
2^20 2^-53 = 1e-10."""
import numpy as np
import pytest

from paper_1306_3247_gb300 import wavepacket as WPK

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["c128", "c128f"])
@pytest.mark.parametrize("n", [256, 1024, 2048, 8192])
@pytest.mark.parametrize("origin", [0.0, 2.0 ** 20, -(2.0 ** 20)])
def test_potential_energy(n, origin, prec):
    L, c = 32.0, origin + 1.0
    pb = {"ndim": 1, "n": [n], "xmin": [origin - L / 2], "L": [L], "dt": 0.01, "t0": 0.5}
    terms = [{"shape": "linear", "a": [0.7], "c0": [c], "coef": {"A0": 1.5}},
             {"shape": "linear", "a": [-0.2], "c0": [c - 2.0], "v": [4.0], "coef": {"A0": 1.0}},
             {"shape": "const", "coef": {"A0": 0.25}},
             {"shape": "quad", "a": [0.5], "c0": [c], "coef": {"A0": 1.0}}]
    with WPK.Propagator(pb, terms, prec) as P:
        P.init_gaussian([c + 1.0], [0.5], [1.2])
        psi, epot = P.get_state(), P.observe()["epot"]
    u = origin - L / 2 + np.arange(n) * (L / n) - c
    V = 1.5 * 0.7 * u - 0.2 * u + 0.25 + 0.25 * u * u  # the second centre is at c when t = 0.5
    rho = np.abs(psi) ** 2 * (L / n)
    assert abs(float(epot) - np.sum(V * rho)) < 1e-13 * np.sum(np.abs(V) * rho)
