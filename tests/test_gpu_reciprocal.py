"""GPU: the FP64 reciprocal of the kernels against division, and their sign test against x > 0.

Bound: with a seed of relative error d, the cubic step leaves d^3 (2^-60 for the hardware's 2^-20) and three roundings, of
which only the last is of the size of half an ulp, so the result lies within 0.51 ulp of 1/x and within 1 ulp of the
correctly rounded quotient.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    import torch
    from paper_2605_03479_gb300 import build
    lib = str(tmp_path_factory.mktemp("rcp") / "libdevice_reciprocal.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "--expt-relaxed-constexpr", "-I", os.path.join(build.HERE, "csrc"), "-o", lib,
                           os.path.join(HERE, "device_reciprocal.cu")])
    fn = C.CDLL(lib).device_reciprocal
    fn.argtypes = [C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]

    def run(x):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        normal, anyx = torch.empty_like(t), torch.empty_like(t)
        positive = torch.empty(len(x), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        assert fn(t.data_ptr(), len(x), normal.data_ptr(), anyx.data_ptr(), positive.data_ptr()) == 0
        return normal.cpu().numpy(), anyx.cpu().numpy(), positive.cpu().numpy() != 0

    return run


@pytest.mark.parametrize("low,high", [(-1, 1), (-60, 60), (-1022, 1020)])
def test_reciprocal_is_within_one_ulp_of_the_quotient(evaluate, low, high):
    rng = np.random.default_rng(low + 2000)
    n = 1 << 20
    x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(low, high + 1, n)) * rng.choice([-1.0, 1.0], n)
    edges = np.concatenate([np.ldexp(m, np.arange(low, high + 1)) for m in (1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52)])
    x = np.concatenate([x, edges, -edges])
    normal, anyx, positive = evaluate(x)
    ref = 1.0 / x
    assert np.all(np.abs(normal - ref) <= np.spacing(np.abs(ref)))
    assert np.array_equal(normal, anyx)
    assert np.array_equal(positive, x > 0)


def test_zero_infinite_and_denormal_values(evaluate):
    tiny, denormal = np.finfo(float).tiny, 5e-324
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, denormal, -denormal, tiny, -tiny, 2.0 ** -1043, 2.0 ** -1042,
                  np.finfo(float).max])
    _, anyx, positive = evaluate(x)
    want = np.array([np.inf, -np.inf, 0.0, -0.0, np.nan, np.inf, -np.inf, 1 / tiny, -1 / tiny, np.inf, np.inf, 0.0])
    assert np.array_equal(anyx, want, equal_nan=True)
    assert np.array_equal(np.signbit(anyx[:4]), np.signbit(want[:4]))
    assert np.array_equal(positive, x > 0)


def test_temperature_of_a_cold_beam_is_zero():
    # one velocity node and b = 0: no internal energy, so 1/(2 R T) is infinite and T and p are zero
    import torch
    from paper_2605_03479_gb300 import build, hbugks as hb
    build.build()
    one = torch.ones(1, dtype=torch.float64, device="cuda")
    h, b = torch.full((1, 4, 1), 2.0, dtype=torch.float64, device="cuda"), torch.zeros(1, 4, 1, dtype=torch.float64, device="cuda")
    re, im = (torch.empty(8, 4, dtype=torch.float64, device="cuda") for _ in range(2))
    assert hb.harmonic_noalloc(2, 2, 1, 1, one, one, one, one, 1, h, b, 0, re, im) == hb.OK
    torch.cuda.synchronize()
    want = np.array([2.0, 1.0, 1.0, 0.0, 0.0, 0.0, 0.0, 0.0])
    assert np.array_equal(re.cpu().numpy(), np.repeat(want[:, None], 4, axis=1))
