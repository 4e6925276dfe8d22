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


@pytest.mark.parametrize("half_width", [7.8, 7.84, 7.88])
def test_wide_velocity_grid_in_hot_gas(hb, half_width):
    # gas at 3.8 T0 with a large heat flux on a grid so wide that H/H_ref reaches 1e37 in its corners, where H_ref lies
    # below the smallest 32-bit value: H (1 + Shakhov factor) is finite there though (H/H_ref)(1 + factor) is not
    c = I.make_case("hot", 6, 24, kn=10.0, st=1.0, nh=1, pr=0.3, drive="thermal", amp=0.3, precision=1,
                    half_width=half_width)
    for w in c.walls:
        w[2] = 3.8
    x, y = (0.5 * (n[1:] + n[:-1]) for n in (c.xnodes, c.ynodes))
    X, Y = (a.ravel() for a in np.meshgrid(x, y))
    u, v = np.tile(c.u, c.nv), np.repeat(c.v, c.nu)
    skew = 1.0 + 0.9 * np.tanh((u + v) ** 3 / 40.0 - (u + v))
    W, h = np.zeros((c.nt, c.nc, 4)), np.zeros((c.nt, c.nc, c.nvel))
    b = np.zeros_like(h)
    for n in range(c.nt):
        T = 3.8 + 0.4 * np.cos(np.pi * X + 0.3 * n) * np.cos(np.pi * Y)
        rho, U, V = 1.0 + 0.1 * np.sin(2 * X + n) * Y, 0.1 * np.sin(3 * Y + n), 0.1 * np.cos(2 * X)
        H = (rho / (np.pi * T))[:, None] * np.exp(-((u - U[:, None]) ** 2 + (v - V[:, None]) ** 2) / T[:, None])
        h[n], b[n] = H * skew, H * skew * 0.5 * T[:, None]
        W[n] = np.stack([rho, rho * U, rho * V, 0.5 * rho * (U ** 2 + V ** 2) + 0.75 * rho * T], 1)
    compare(hb, c, (W, h, b), 1, 2e-5, 2e-7)


@pytest.mark.parametrize("node", [1e-18, 1e-24, 1e-30])
@pytest.mark.parametrize("precision", [0, 1])
def test_velocity_node_close_to_zero(hb, node, precision):
    # a node whose square lies below the smallest 32-bit value still moves into the walls on its side
    c = I.make_case("tiny", 5, 9, kn=0.3, st=1.0, nh=1, pr=2 / 3, drive="thermal", amp=0.3, precision=precision)
    c.u, c.v = c.u.copy(), c.v.copy()
    c.u[4], c.v[4] = node, -node
    compare(hb, c, I.initial_state(c, seed=3), 2, *((1e-10, 1e-13) if precision == 0 else (2e-5, 2e-7)))
