"""GPU: inputs at the far ends of what the entry points accept, against the FP64 oracle.

Tolerances as for every parity test: FP64 1e-10 of the change plus 1e-13 of the magnitude (summation order only),
FP32-split 2e-5 of the change plus 2e-7 of the magnitude (rounding of 32-bit deviations).
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_03479_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    from paper_2605_03479_gb300 import build, hbugks
    build.build()
    return hbugks


def compare(hb, case, state, iters, change, size):
    s = hb.Solver(case)
    s.set_state(0, *state)
    s.iterate(iters)
    got = s.get_state(0)
    ref = tuple(x.copy() for x in state)
    O.iterate(O.Problem(case), *ref, iters)
    for g, r, init in zip(got, ref, state):
        assert np.all(np.isfinite(r)) and np.all(np.isfinite(g))
        assert np.max(np.abs(g - r)) <= change * np.max(np.abs(r - init)) + size * np.max(np.abs(r))


@pytest.mark.parametrize("w_vss", [0.0, 1.0, 2.0])
def test_negative_temperature_with_a_whole_viscosity_exponent(hb, w_vss):
    # one cell of one level starts below zero internal energy: (T/T0)^w is defined for a whole exponent w, so the
    # iteration goes on, as in the oracle
    c = I.make_case("neg", 5, 8, kn=0.3, st=1.0, nh=1, pr=2 / 3, drive="thermal", amp=0.3)
    c.w_vss = w_vss
    W, h, b = I.initial_state(c, seed=3)
    W[1, 7, 3] = -0.2
    compare(hb, c, (W, h, b), 1, 1e-10, 1e-13)
