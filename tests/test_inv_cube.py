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

    def differences(xi, xj, E):
        xi, xj, E = np.ascontiguousarray(xi), np.ascontiguousarray(xj), np.ascontiguousarray(E, dtype=np.int32)
        n = E.shape[0]
        d, cube, taken = np.zeros((3, n)), np.zeros(n), np.zeros(n, dtype=np.int32)
        P = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        lib.ic_differences(ctypes.c_int64(n), P(xi), P(xj), P(E), P(d), P(cube), P(taken))
        return d, cube, taken == 1

    def factors(d, mu, off, power=3):
        d, mu, off = (np.ascontiguousarray(t, dtype=np.float64) for t in (d, mu, off))
        n = mu.shape[0]
        res, taken = np.empty(n), np.empty(n, dtype=np.int32)
        P = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
        lib.ic_factors(ctypes.c_int64(n), ctypes.c_int32(power), P(d[0]), P(d[1]), P(d[2]), P(mu), P(off), P(res), P(taken))
        return res, taken
    factors.differences = differences
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


@pytest.mark.parametrize("kind", ["any", "near the origin", "pairs far from it", "flat", "another body sets the scale"])
def test_fixed_point_differences(ic, kind):
    """96-bit integers hold a coordinate exactly down to 2^-40 of the largest
    and to 2^-92 of it below, so a component (at least 2^-37 of the scale,
    where it is taken) is exact to 2^-55 and then rounds to FP64: 0.63 units in
    the last place of the component itself.  |d|^-3 is off by 3 x sqrt(3) 2^-61
    from the 62-bit alignment, plus its own 0.77 units in the last place."""
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision here")
    rng = np.random.default_rng(9)
    n = 300_000
    scale = np.exp2(rng.integers(-150, 150, n).astype(float))
    xi, xj = rng.uniform(-1, 1, (3, n)) * scale, rng.uniform(-1, 1, (3, n)) * scale
    if kind == "near the origin":
        xi *= np.exp2(-rng.uniform(0, 30, (3, n)))
    elif kind == "pairs far from it":
        xj = xi + xj * np.exp2(-rng.uniform(0, 12, n))
    elif kind == "flat":
        xi[2] = xj[2] = 0.0
    # the field of the largest coordinate, or of a further body's
    E = np.frexp(np.abs(np.concatenate([xi, xj])).max(0))[1] + 1022
    if kind == "another body sets the scale":
        E = E + rng.integers(0, 7, n)
    got, cube, ok = ic.differences(xi, xj, E)
    if kind == "flat":
        assert not ok.any()  # a component below 2^-30 of the largest: left to FP64
        return
    assert ok.mean() > (0.2 if kind in ("pairs far from it", "another body sets the scale") else 0.9)
    want = xj.astype(np.longdouble) - xi.astype(np.longdouble)
    ulp = np.spacing(np.abs(want.astype(np.float64)))
    assert (np.abs(got.astype(np.longdouble) - want) / ulp)[:, ok].max() <= 0.63
    r2 = (want * want).sum(0)
    ref = (1 / (r2 * np.sqrt(r2)))[ok]
    err = np.abs((cube[ok] - ref) / ref).astype(float)
    assert err.max() <= 3 * np.sqrt(3) * 2.0**-61 + 0.77 * 2.0**-52


def test_fixed_point_leaves_close_pairs(ic):
    one, E = np.ones((3, 1)), np.array([1023])
    near = one * (1 + 2.0**-9)   # closer than 2^-7 of the scale
    far = one * np.array([[-1.0], [0.5], [0.25]])
    assert not ic.differences(one, near, E)[2][0]
    assert ic.differences(one, far, E)[2][0]
    assert not ic.differences(one, far, np.array([1023 - 195]))[2][0]  # a scale beyond the range
    assert not ic.differences(one, one, E)[2][0]
