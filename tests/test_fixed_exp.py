"""Tests of fixed_exp.h (square root, reciprocal root, quotient and e^-x in integer arithmetic) on the CPU and on
the GPU: the first three bit for bit against IEEE arithmetic, e^-x within the header's bounds, at random
arguments, next to rounding boundaries, and at the ends of the ranges they are used on."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2410_09819_gb300", "csrc")
SRC = os.path.join(HERE, "fixed_exp_harness.cu")


def _compile(cmd, out):
    r = subprocess.run([*cmd, "-I", CSRC, SRC, "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)
    lib.apply_all.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int, ctypes.c_void_p]
    table = np.empty(1024, dtype=np.uint64)
    lib.fill_table(table.ctypes.data_as(ctypes.c_void_p))
    return lib, table


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    out = str(tmp_path_factory.mktemp("fx") / "fx_host.so")
    lib, table = _compile(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off", "-x", "c++"], out)

    def run(op, x, y):
        x, y = np.ascontiguousarray(x), np.ascontiguousarray(y)
        z = np.empty_like(x)
        assert lib.apply_all(op, x.ctypes.data, y.ctypes.data, z.ctypes.data, x.size, table.ctypes.data) == 0
        return z
    return run


@pytest.fixture(scope="module")
def device(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    out = str(tmp_path_factory.mktemp("fx") / "fx_device.so")
    lib, table = _compile([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-cudart", "shared"], out)
    tab = torch.from_numpy(table.view(np.int64)).cuda()

    def run(op, x, y):
        xd, yd = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (x, y))
        zd = torch.empty_like(xd)
        torch.cuda.synchronize()
        assert lib.apply_all(op, xd.data_ptr(), yd.data_ptr(), zd.data_ptr(), xd.numel(), tab.data_ptr()) == 0
        return zd.cpu().numpy()
    return run


def _shift(x, ulps):
    return (x.view(np.int64) + ulps).view(np.float64)


def _mantissas(rng, n):
    """In [1, 2): random, few leading bits, all ones but few, and the neighbours of 1 and 2."""
    w = rng.integers(0, 1 << 52, n, dtype=np.int64)
    w[: n // 8] &= ~np.int64((1 << 40) - 1)
    w[n // 8: n // 4] |= np.int64(((1 << 52) - 1) ^ 0xFFFF)
    w[:16] = [0, 1, 2, 3, (1 << 52) - 1, (1 << 52) - 2, (1 << 52) - 3, 1 << 51] * 2
    return (w | (np.int64(1023) << 52)).view(np.float64)


def _root_arguments(rng, n):
    """Normal numbers over POTRF's range of exponents; half of them next to a square whose root is exact or lies
    half way between two numbers (the only places where the rounding of a root is close)."""
    e = rng.integers(-920, 921, n)
    e[:4] = [-922, -921, 921, 922]
    x = np.ldexp(_mantissas(rng, n), e)
    h = _mantissas(rng, n // 2)
    h[: n // 4] = _mantissas(rng, n // 4).astype(np.float32)                       # exact squares
    sq = np.ldexp(h, 0).astype(np.longdouble)
    sq[n // 4:] += np.longdouble(2.0) ** -53                                       # boundaries of the root
    x[n // 2:] = np.ldexp(_shift((sq * sq).astype(np.float64), rng.integers(-2, 3, n // 2)), 2 * rng.integers(-200, 200, n // 2))
    return x


def _check_roots(run):
    x = _root_arguments(np.random.default_rng(1), 400000)
    r = np.sqrt(x)
    assert np.array_equal(run(0, x, x), r)
    assert np.array_equal(run(1, x, x), r)
    assert np.array_equal(run(2, x, x), 1.0 / r)


def _check_quotients(run):
    rng = np.random.default_rng(2)
    n = 400000
    y = np.ldexp(_mantissas(rng, n), rng.integers(-332, 333, n))                   # the divisors' range in use: 1e-100 .. 1e100
    x = np.ldexp(_mantissas(rng, n), rng.integers(-250, 251, n))
    # next to a quotient that is exact or half way between two numbers
    q = _mantissas(rng, n // 2).astype(np.longdouble)
    q[n // 4:] += np.longdouble(2.0) ** -53
    x[n // 2:] = _shift((q * y[n // 2:]).astype(np.float64), rng.integers(-2, 3, n // 2))
    assert np.array_equal(run(3, x, y), x / y)


def _check_exponentials(run):
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.random(200000) * 700, rng.random(200000) * 40, rng.random(100000),
                        np.ldexp(_mantissas(rng, 100000), rng.integers(-320, 5, 100000)),
                        np.nextafter([700.0, 40.0, 1.0], 0), np.arange(1, 1000) * np.log(2.0) / 1024, np.arange(1.0, 700.0)])
    exact = np.exp(-x.astype(np.longdouble))
    ulp = np.spacing(exact.astype(np.float64))
    ulp[exact < exact.astype(np.float64)] = np.spacing(np.nextafter(exact.astype(np.float64), 0))[exact < exact.astype(np.float64)]
    err = np.abs(run(4, x, x).astype(np.longdouble) - exact) / ulp
    assert err[x < 40].max() <= 0.52 and err.max() <= 0.62, (err[x < 40].max(), err.max())


CHECKS = [_check_roots, _check_quotients, _check_exponentials]


@pytest.mark.parametrize("check", CHECKS)
def test_on_the_host(host, check):
    check(host)


@pytest.mark.gpu
@pytest.mark.parametrize("check", CHECKS)
def test_on_the_device(device, check):
    check(device)
