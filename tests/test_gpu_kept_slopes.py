"""GPU: the FP64 micro update with the slopes the face sums have kept, against forming them itself.

A handle keeps them while they take at most 8 GiB, so a small case next to one of more than that runs the other route;
both read the same neighbours in the same order, so the iterates must be bitwise equal.  Sizes: one column, strips that
overlap, a row left over after a segment, zero velocity nodes, walls on every side of partial strips.
"""
import numpy as np
import pytest

from paper_2605_03479_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_kept_slopes_give_the_same_iterate():
    from paper_2605_03479_gb300 import build, hbugks as hb
    build.build()
    sizes = [(1, 5, 8, 8, 1), (5, 33, 8, 10, 1), (7, 9, 9, 11, 2), (9, 6, 16, 8, 3)]
    small = [I.make_case("s", nx, nu, kn=0.2, st=2.0, nh=nh, pr=2 / 3, drive="thermal", amp=0.3, ncell_y=ny, nvel_y=nv)
             for nx, ny, nu, nv, nh in sizes]
    large = I.make_case("large", 96, 64, kn=0.2, st=1.0, nh=5, pr=2 / 3, drive="shear")
    assert 32 * large.updates_per_iteration() > 8 << 30
    states = [I.initial_state(c, seed=3 + k) for k, c in enumerate(small)]

    def run(cases):
        s = hb.Solver(cases)
        s.set_active([1] * len(small) + [0] * (len(cases) - len(small)))
        for k, st in enumerate(states):
            s.set_state(k, *st)
        s.iterate(3)
        return [s.get_state(k) for k in range(len(small))]

    for a, b in zip(run(small), run(small + [large])):
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
