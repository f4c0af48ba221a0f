"""A bounded device wait that ran out (WP_ETIMEOUT) is reported by the next call on the handle
that returns host data, whatever was launched in between, and then once only. No wait is made
to run out: the error is written into the handle's control block as a kernel would."""
import ctypes

import numpy as np
import pytest

from paper_1306_3247_gb300 import wavepacket as WPK

pytestmark = pytest.mark.gpu

SHAPES = [(64,), (1024,), (4096,), (64, 128), (32, 32, 32)]


def raise_error(h):
    f = WPK.load_library()._ZN2wp16handle_lose_waitEP9wp_handle
    f.argtypes, f.restype = [ctypes.c_void_p], ctypes.c_int
    assert f(h) == WPK.WP_OK


def problem(n):
    return {"ndim": len(n), "n": list(n), "xmin": [-8.0] * len(n), "L": [16.0] * len(n), "dt": 0.01}


def propagator(n, prec="c128"):
    P = WPK.Propagator(problem(n), [], prec)
    P.init_gaussian([0.0] * len(n), [0.5] * len(n), [1.0] * len(n))
    return P


def timed_out(call):
    with pytest.raises(WPK.WavepacketError) as e:
        call()
    return e.value.status == WPK.WP_ETIMEOUT


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("read", ["observe", "get_state", "run", "expect"])
def test_reported_after_more_steps(n, read):
    with propagator(n) as P:
        call = {"observe": P.observe, "get_state": P.get_state, "run": lambda: P.run(2, 1),
                "expect": lambda: P.expect_grid(np.ones(n))}[read]
        P.step(3)
        raise_error(P.h)
        P.step(3)
        assert timed_out(call)
        call()  # reported once


def test_reported_by_a_callback_run():
    with propagator((4096,)) as P:
        seen = []

        def record(prop, rec):
            seen.append(1)
            if len(seen) == 2:
                raise_error(P.h)
            return False

        assert timed_out(lambda: P.run_with_callback(6, 2, record))
        assert len(seen) == 2


@pytest.mark.parametrize("read", ["observe", "get_state"])
@pytest.mark.parametrize("n", [(8192,), (64, 128)])
def test_reported_by_a_batch_instance(n, read):
    with WPK.Batch("c64") as B:
        B.add(problem(n), [])
        B.set_state(0, np.ones(n))
        B.step(2)
        raise_error(B.handle(0))
        B.step(2)
        call = (lambda: WPK.wp_observe(B.handle(0))) if read == "observe" else (lambda: B.get_state(0))
        assert timed_out(call)
        call()


def test_outranks_a_norm_that_is_not_finite():
    x = np.ones((64, 128), complex)
    x[1, 2] = np.nan
    with propagator((64, 128)) as P:
        P.set_state(x)
        raise_error(P.h)
        assert timed_out(lambda: P.run(2, 1))
        with pytest.raises(WPK.WavepacketError) as e:
            P.run(2, 1)
        assert e.value.status == WPK.WP_ENONFINITE
        assert np.all(np.isnan(P.get_state()))  # a norm's error does not keep the state back
