"""GPU: an FP64 handle in a workspace without room for the slopes it would keep between two kernels.

It forms them in both, with bitwise the same iterate; only less than that is refused.
"""
import ctypes as C

import numpy as np
import pytest

from paper_2605_03479_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    from paper_2605_03479_gb300 import build, hbugks
    build.build()
    return hbugks


def slope_bytes(c):
    # two pairs of doubles per cell, level and stored velocity; a sign class fills whole blocks of 32 velocities
    blocks = sum(-(-(np.sum(sx * c.u > 0) * np.sum(sy * c.v > 0)) // 32) for sx in (1, -1) for sy in (1, -1))
    return int(blocks) * 32 * c.nc * c.nt * 32


def create(hb, c, nbytes):
    """Status of hbugks_create in a workspace of nbytes, and the handle."""
    import torch
    args = hb._CaseArgs(c)
    ws = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda:0")
    h = C.c_void_p()
    rc = hb.lib().hbugks_create(1, C.byref(args.c), C.c_void_p((ws.data_ptr() + 255) // 256 * 256), nbytes,
                                C.c_void_p(torch.cuda.current_stream().cuda_stream), C.byref(h))
    if rc == hb.OK:
        hb.lib().hbugks_destroy(h)
    return rc


@pytest.mark.parametrize("size", [(1, 8, 0), (6, 10, 1), (33, 16, 3)])
def test_a_workspace_without_the_slopes_is_accepted(hb, size):
    n, nv, nh = size
    c = I.make_case("ws", n, nv, kn=0.2, st=1.0, nh=nh, pr=2 / 3, drive="thermal")
    full = hb.workspace_bytes([c])
    without = full - slope_bytes(c) + 256              # 256: arrays start on multiples of 256 bytes
    assert create(hb, c, full) == hb.OK
    assert create(hb, c, without) == hb.OK
    assert create(hb, c, without - 1024) == hb.ENOMEM


def test_solver_goes_without_the_slopes_where_memory_is_short(hb, monkeypatch):
    import torch
    c = I.make_case("ws", 12, 10, kn=0.2, st=1.0, nh=2, pr=2 / 3, drive="thermal", ncell_y=9)
    state = I.initial_state(c, seed=4)

    def run():
        s = hb.Solver(c)
        s.set_state(0, *state)
        s.iterate(4)
        return s.workspace_bytes, s.get_state(0)

    full, a = run()
    empty = torch.empty

    def scarce(n, *args, **kw):
        if isinstance(n, int) and n >= full:
            raise torch.OutOfMemoryError("short")
        return empty(n, *args, **kw)

    monkeypatch.setattr(torch, "empty", scarce)
    least, b = run()
    assert full - slope_bytes(c) - 256 <= least <= full - slope_bytes(c) + 256
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    c32 = I.make_case("ws", 6, 10, kn=0.2, st=1.0, nh=1, precision=1)
    full = 0                                           # nothing to go without in single precision
    with pytest.raises(torch.OutOfMemoryError):
        hb.Solver(c32)
