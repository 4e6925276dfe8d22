"""GPU: the FP64 reciprocal of the kernels against division, their sign test against x > 0, and their power of a
temperature ratio against 128-bit arithmetic.

Bound: with a seed of relative error d, the cubic step leaves d^3 (2^-60 for the hardware's 2^-20) and three roundings, of
which only the last is of the size of half an ulp, so the result lies within 0.51 ulp of 1/x and within 1 ulp of the
correctly rounded quotient.  The power: exp and log are within 1 ulp each, so exp(y) of a y = -w log x with |y| <= 1/4 is
within 1 ulp plus |y| times the 1.5 ulp of y, below 2 ulp; beyond, pow within 2 ulp plus w <= 1 times the reciprocal's
ulp (twice as many of the result's where its mantissa is small), below 4 ulp.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    from paper_2605_03479_gb300 import build
    lib = str(tmp_path_factory.mktemp("rcp") / "libdevice_reciprocal.so")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "--expt-relaxed-constexpr", "-I", os.path.join(build.HERE, "csrc"), "-o", lib,
                           os.path.join(HERE, "device_reciprocal.cu")])
    lib = C.CDLL(lib)
    lib.device_reciprocal.argtypes = [C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
    lib.device_power.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_void_p]
    return lib


@pytest.fixture(scope="module")
def evaluate(library):
    import torch

    def run(x):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        normal, anyx = torch.empty_like(t), torch.empty_like(t)
        positive = torch.empty(len(x), dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        assert library.device_reciprocal(t.data_ptr(), len(x), normal.data_ptr(), anyx.data_ptr(), positive.data_ptr()) == 0
        return normal.cpu().numpy(), anyx.cpu().numpy(), positive.cpu().numpy() != 0

    return run


def power(library, x, w):
    import torch
    t, e = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, w))
    here, ref = torch.empty_like(t), torch.empty_like(t)
    torch.cuda.synchronize()
    assert library.device_power(t.data_ptr(), e.data_ptr(), len(x), here.data_ptr(), ref.data_ptr()) == 0
    return here.cpu().numpy(), ref.cpu().numpy()


@pytest.mark.parametrize("spread", [1e-3, 0.3, 3.0])
def test_temperature_power(library, spread):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no wider floating point on this host")
    rng = np.random.default_rng(7)
    n = 1 << 18
    x, w = np.exp(rng.uniform(-spread, spread, n)), rng.uniform(0.5, 1.0, n)
    here, ref = power(library, x, w)
    exact = np.power(x.astype(np.longdouble), -w.astype(np.longdouble))
    ulp = np.spacing(exact.astype(np.float64)).astype(np.longdouble)
    err, err_pow = np.abs(here - exact) / ulp, np.abs(ref - exact) / ulp
    print(f"spread {spread}: {float(err.max()):.3f} ulp, pow of the quotient {float(err_pow.max()):.3f} ulp")
    near = np.abs(w * np.log(x)) < 0.25
    assert np.all(err[near] <= 2.0) and np.all(err <= 4.0)


def test_temperature_power_below_zero(library):
    x = np.repeat([-0.25, -1.0, -3.0], 4)
    w = np.tile([0.0, 1.0, 2.0, 0.81], 3)
    here, _ = power(library, x, w)
    with np.errstate(invalid="ignore"):
        want = np.power(1.0 / x, w)
    assert np.allclose(here, want, rtol=1e-15, atol=0.0, equal_nan=True)


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
