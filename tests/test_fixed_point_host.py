"""The fixed-point constraint solve (csrc/fixed.cuh, solve_fx.cuh) compiled for the host: its
exponential and conversions against long doubles, its solve against the 13 constraints and the
FP64 iteration, and the cells it must give up.

Tolerances: the exponential rounds to 53 bits (0.5 ulp) a value whose parts are rounded to 2^-55
(table, second part of the product: 1/16 and 1/8 ulp) with float errors below 2^-55 (1/8 ulp) in
the product: 1 ulp.  A solve ends with max|G| below tol/100 = 1e-14 or after a polishing step; G is
read from truncations of 39 values to 2^-58 times at most 27: 1.1e-14 covers both."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LD = np.longdouble


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fx") / "fixed_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-shared", "-fPIC",
                    os.path.join(HERE, "fixed_host.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.fx_solve.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                           ctypes.c_int, ctypes.c_double, ctypes.c_int, ctypes.c_void_p]
    return L


def p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def ints(a):
    """Exact integers of a long-double array as Python ints."""
    return [int(x) for x in a]


def test_exponential(lib):
    rng = np.random.default_rng(0)
    edge = [(n << 55) + (j << 45) + d for n in (-124, -20, -1, 0, 3) for j in (0, 1, 511, 1023)
            for d in (0, 1, (1 << 44) - 1, 1 << 44, (1 << 45) - 1)]
    X = np.concatenate([np.array(edge, np.int64),
                        rng.integers(-(60 << 55), 4 << 55, 100_000, dtype=np.int64)])
    y = np.empty(len(X))
    lib.fx_exp2(p(X), p(y), ctypes.c_longlong(len(X)))
    n = X >> 55
    frac = (X - (n << 55)).astype(LD) / LD(2) ** 55      # in [0, 1), exact
    exact = np.exp2(frac)                                 # in [1, 2): the long double's own error is below 2^-62
    err = (np.ldexp(y.astype(LD), -n.astype(np.int32)) - exact) * LD(2) ** 52
    assert np.abs(err).max() <= 1.0
    assert abs(err.mean()) <= 0.05


def test_conversions(lib):
    rng = np.random.default_rng(1)
    n = 20_000
    F = np.exp2(-rng.uniform(0.42, 70.0, n))
    F[:3] = 0.75 - 2.0**-53, 2.0**-58, 2.0**-126
    v = rng.uniform(-32, 32, n) * np.exp2(-rng.uniform(0, 50, n))
    v[:4] = 0.0, 1.0, -31.999, 2.0**-60
    l = rng.uniform(-100, 100, n) * np.exp2(-rng.uniform(0, 60, n))
    l[:2] = 0.0, -0.0
    u58, s58 = np.empty(n, np.uint64), np.empty(n, np.int64)
    L, back = np.empty(n, np.int64), np.empty(n)
    lib.fx_convert(p(F), p(u58), p(v), p(s58), p(l), p(L), p(back), ctypes.c_longlong(n))
    assert ints(u58) == ints(np.floor(F * 2.0**58))
    assert ints(s58) == ints(np.trunc(v * 2.0**58))
    log2e = LD(1) / np.log(LD(2))
    d = l.astype(LD) * log2e * LD(2) ** 55 - L.astype(LD)
    assert (np.abs(d) <= 0.5 + 2.0**-6 + np.abs(l) * 2.0**-6).all()  # the long double's own rounding
    assert (np.abs(back - l) <= 2.0**-56 + np.abs(l) * 2.0**-52).all()


def basis(lib):
    v = np.empty((39, 3), np.int32)
    lib.velocities(p(v))
    v = v.astype(float)
    c2 = (v * v).sum(1)
    x, y, z = v.T
    return np.stack([np.ones(39), x, y, z, x * x, y * y, z * z, x * y, x * z, y * z, x * c2,
                     y * c2, z * c2])


def targets(u, T):
    x, y, z = u
    h = u @ u + 5 * T
    return np.array([1, x, y, z, x * x + T, y * y + T, z * z + T, x * y, x * z, y * z, x * h,
                     y * h, z * h])


def solve(lib, phi, lam, m, cached, refine, d2, fixed, maxit=200, tol=1e-12):
    ws = np.concatenate([np.exp(lam @ phi), lam, m])
    out = np.zeros(3, np.int32)
    ok = lib.fx_solve(p(ws), refine, d2, fixed, cached, tol, maxit, p(out))
    return ok, ws[:39].copy(), ws[39:52].copy(), int(out[0]), int(out[1])


def gaussian(phi, u, T):
    lam = np.zeros(13)
    lam[1:4] = u / T
    lam[4:7] = -0.5 / T
    lam[0] = -np.log(np.exp(lam @ phi).sum())
    return lam


@pytest.mark.parametrize("refine", [1, 0])
@pytest.mark.parametrize("d2", [0, 1])
def test_solve_meets_the_constraints_as_the_fp64_iteration(lib, refine, d2):
    phi = basis(lib)
    rng = np.random.default_rng(2)
    updates = np.zeros(2, int)
    for k in range(60):
        u = rng.uniform(-0.6, 0.6, 3) if k else np.zeros(3)
        if k % 7 == 1:
            u *= 1.1 / max(np.linalg.norm(u), 1e-3)       # fast
        if d2:
            u[2] = 0.0
        T = float(rng.uniform(0.42, 0.75))
        cold = solve(lib, phi, gaussian(phi, u, T), targets(u, T), 0, 1, 0, 1)
        if not cold[0]:      # outside the ranges from the cold start: nothing to warm-start from
            continue
        lam = cold[2]
        if d2:
            lam[[3, 8, 9, 12]] = 0.0
        du = rng.normal(0, 0.02, 3) * (1, 1, 0 if d2 else 1)
        m = targets(u + du, T * 1.01)
        a = solve(lib, phi, lam, m, 1, refine, d2, 1)
        b = solve(lib, phi, lam, m, 1, refine, d2, 0)
        assert a[0] and b[0] and a[4] == 0 and b[4] == 0
        G = (a[1].astype(LD) * phi.astype(LD)).sum(1) - m
        assert np.abs(G).max() <= 1.1e-14
        assert np.abs(a[1] - b[1]).max() <= 1e-13
        assert abs(a[3] - b[3]) <= 1
        updates += a[3], b[3]
    assert updates[1] > 100 and abs(updates[0] - updates[1]) <= 0.02 * updates[1]


def test_solve_gives_up_what_it_cannot_represent(lib):
    phi = basis(lib)
    u, T = np.array([0.3, -0.2, 0.1]), 0.5
    lam, m = gaussian(phi, u, T), targets(u, T)
    assert solve(lib, phi, lam, m, 0, 1, 0, 1)[0] == 1
    for k, big in ((0, 50.0), (1, 12.0), (4, 3.0), (10, 0.8)):   # beyond 64, 16, 4, 1 times ln 2
        bad = lam.copy()
        bad[k] = -big
        assert solve(lib, phi, bad, m, 0, 1, 0, 1)[0] == 0
    for k in (0, 4, 12):
        for v in (16.5, np.nan, np.inf):
            bad = m.copy()
            bad[k] = v
            assert solve(lib, phi, lam, bad, 0, 1, 0, 1)[0] == 0
    hot = lam.copy()
    hot[0] += 3.0                                                # sum F_i = 20
    assert solve(lib, phi, hot, m, 1, 1, 0, 1)[0] == 0


def test_no_update_leaves_the_multipliers_alone(lib):
    phi = basis(lib)
    u, T = np.array([0.25, 0.1, -0.3]), 0.55
    first = solve(lib, phi, gaussian(phi, u, T), targets(u, T), 0, 1, 0, 1)
    ws = np.concatenate([first[1], first[2], targets(u, T)])
    out = np.zeros(3, np.int32)
    assert lib.fx_solve(p(ws), 1, 0, 1, 1, 1e-12, 30, p(out)) == 1
    assert out[0] == 0 and out[1] == 0 and out[2] == 0
    assert np.array_equal(ws[:39], first[1]) and np.array_equal(ws[39:52], first[2])
