"""mu |d|^-3 (and mu |d|^-2, mu |d|^-1) on the integer pipes (csrc/inv_cube.h), built with g++ through
tests/inv_cube_shim.cpp and checked on the CPU against 80-bit arithmetic.

Bound, in units in the last place (2^53 times a relative error at most):
half for the rounding; 0.14 for |d|^2 (three units of at least 2^58, times
3/2); 0.07 for the series (35/16 e^3 with |e| < 2^-19.2); 0.05 for the
truncations of the 60- to 64-bit products: 0.77 in all (the other powers
have less of each).  The seed is given
every error the FP32 instruction may have (2^-22.4 relative, documented
2 ulp).  Inputs: all magnitudes the path takes, components that are equal,
zero, tiny beside another or a power of two, masses likewise; what it leaves
to the FP64 series (zero, subnormal, infinite and NaN differences, masses
beyond its range) it must say so.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2112_15079_gb300", "csrc")
BOUND_ULP = 0.77


@pytest.fixture(scope="module")
def ic(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("ic") / "libic.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "inv_cube_shim.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)

    def factors(d, mu, off, power=3):
        d, mu, off = (np.ascontiguousarray(t, dtype=np.float64) for t in (d, mu, off))
        n = mu.shape[0]
        res, taken = np.empty(n), np.empty(n, dtype=np.int32)
        P = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        lib.ic_factors(ctypes.c_int64(n), ctypes.c_int32(power), P(d[0]), P(d[1]), P(d[2]), P(mu), P(off), P(res), P(taken))
        return res, taken
    return factors


def _draws(kind, n, rng):
    d = rng.uniform(-1.0, 1.0, (3, n)) * np.exp2(rng.uniform(-60, 60, n))
    mu = rng.uniform(1.0, 2.0, n) * np.exp2(rng.integers(-100, 100, n))
    if kind == "small components":
        d *= np.exp2(-rng.uniform(0, 80, (3, n)))
    elif kind == "zero components":
        d *= rng.integers(0, 2, (3, n))
        d[0] += np.where(np.any(d, axis=0), 0.0, 1.0)
    elif kind == "equal components":
        d[1] = d[0]
        d[2] = -d[0]
    elif kind == "powers of two":
        e = np.exp2(rng.integers(-190, 190, n).astype(float))
        d[:] = 0.0
        d[rng.integers(0, 3, n), np.arange(n)] = np.where(rng.integers(0, 2, n) == 1, e, np.nextafter(e, 0.0))
        mu = np.exp2(rng.integers(-390, 390, n).astype(float))
    return d, mu


@pytest.mark.parametrize("kind", ["any", "small components", "zero components", "equal components", "powers of two"])
@pytest.mark.parametrize("power", [3, 2, 1])
def test_within_the_bound(ic, kind, power):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision here")
    rng = np.random.default_rng(5)
    n = 400_000
    d, mu = _draws(kind, n, rng)
    if power < 3 and kind == "powers of two":
        mu = np.exp2(np.clip(np.log2(mu), -350, 350))  # (so that the result is a normal number)
    got, taken = ic(d, mu, rng.uniform(-1, 1, n) * 2.0**-22.4, power)
    assert np.all(taken == 1)
    q = d.astype(np.longdouble)
    r2 = q[0] * q[0] + q[1] * q[1] + q[2] * q[2]
    want = mu.astype(np.longdouble) / {3: r2 * np.sqrt(r2), 2: r2, 1: np.sqrt(r2)}[power]
    ulp = np.spacing(np.abs(want.astype(np.float64)))
    err = (got.astype(np.longdouble) - want).astype(np.float64) / ulp
    assert np.abs(err).max() <= BOUND_ULP
    if kind == "any":
        assert abs(err.mean()) < 0.01  # no bias


def test_massless_gives_zero(ic):
    got, taken = ic(np.array([[3.0], [0.0], [-1.0]]), np.array([0.0]), np.zeros(1))
    assert taken[0] == 1 and got[0] == 0.0


@pytest.mark.parametrize("d, mu", [(0.0, 1.0), (5e-324, 1.0), (2.0**-201, 1.0), (2.0**201, 1.0), (np.inf, 1.0),
                                   (np.nan, 1.0), (1.0, 2.0**-401), (1.0, 2.0**402), (1.0, 5e-324)])
def test_left_to_the_series(ic, d, mu):
    _, taken = ic(np.array([[0.0], [d], [0.0]]), np.array([mu]), np.zeros(1))
    assert taken[0] == 0
