"""GPU: the marching micro update at the edges of its strips, segments and velocity groups.

Sizes: fewer columns than a strip, strips that overlap by one to three columns, segments of 2, 8, 16 and 32 rows with
one row left over, one row, one level and fifteen, sign classes whose last velocity block goes alone, zero velocity
nodes, the spectral source at the new iterate.  Each against the FP64 oracle after three iterations (FP64: 1e-10 of the
change plus 1e-13 of the magnitude, summation order only; FP32-split: 2e-5 of the change plus 2e-7 of the magnitude, the
rounding of 32-bit deviations), and every variant the case can run bitwise equal to the others.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2605_03479_gb300 import inputs as I

pytestmark = pytest.mark.gpu

VARIANTS = [(4, 4, 1), (4, 2, 1), (2, 2, 1), (8, 4, 1), (4, 2, 2)]
# nx, ny, nu, nv, N_H, implicit
SIZES = [(1, 1, 8, 8, 1, 0), (2, 3, 10, 8, 0, 0), (3, 9, 9, 8, 2, 0), (4, 2, 12, 12, 1, 1), (5, 33, 8, 10, 1, 0),
         (6, 17, 16, 8, 3, 0), (7, 1, 8, 9, 7, 0), (9, 5, 8, 8, 5, 1), (11, 18, 24, 12, 2, 0)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny,nu,nv,nh,implicit", SIZES)
def test_edges_of_strips_and_segments(nx, ny, nu, nv, nh, implicit, precision):
    from paper_2605_03479_gb300 import build, hbugks as hb
    build.build()
    c = I.make_case("march", nx, nu, kn=0.2, st=2.0, nh=nh, pr=2 / 3, drive="thermal", amp=0.3, ncell_y=ny, nvel_y=nv,
                    precision=precision)
    c.spectral_implicit = implicit
    state = I.initial_state(c, seed=11)
    s = hb.Solver(c)
    results = []
    for v in VARIANTS:
        try:
            s.set_micro_variant(0, *v)
        except hb.HbugksError:
            continue
        s.set_state(0, *state)
        s.iterate(3)
        results.append(s.get_state(0))
    assert len(results) >= 2
    for other in results[1:]:
        for a, b in zip(results[0], other):
            assert np.array_equal(a, b)
    W, h, b = (x.copy() for x in state)
    O.iterate(O.Problem(c), W, h, b, 3)
    change, size = (1e-10, 1e-13) if precision == 0 else (2e-5, 2e-7)
    for got, ref, init in zip(results[0], (W, h, b), state):
        tol = change * np.max(np.abs(ref - init)) + size * np.max(np.abs(ref))
        assert np.max(np.abs(got - ref)) <= tol
