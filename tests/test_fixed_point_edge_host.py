"""The fixed-point solve where it fails or gives up (csrc/solve_fx.cuh, compiled for the host): a line
search that ends without a lower residual, a spent budget, the edge of the moment cone in both
constraint systems, and the Gaussian start.  Tolerances: as in test_fixed_point_host (1.1e-14 on the
constraints); the multipliers are rounded to 2^-55, times sums |phi_k| of at most 27 in an exponent
and a factor 4 for the 13 of them: F = exp(Phi lam) within 27 * 4 * 2^-55 + 2^-52 < 4e-15; the
normalising sum of the Gaussian start is 39 values within 1 ulp each, its logarithm within 4e-16 and
the rounding of a result below 8 (4.5e-16): 1e-15."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from test_fixed_point_host import LD, basis, gaussian, p, solve, targets

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("edge") / "units_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-shared", "-fPIC",
                    os.path.join(HERE, "units_host.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.fx_solve.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int, ctypes.c_int,
                           ctypes.c_int, ctypes.c_double, ctypes.c_int, ctypes.c_void_p]
    L.fx_gaussian.argtypes = [ctypes.c_void_p, ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p]
    return L


def residual(F, phi, m):
    return float(np.abs((F.astype(LD) * phi.astype(LD)).sum(1) - m).max())


def test_failed_line_search_returns_to_the_last_accepted_point(lib):
    """A tolerance below the resolution: at round-off no halved step lowers the residual."""
    phi = basis(lib)
    rng = np.random.default_rng(5)
    failed = 0
    for _ in range(60):
        u, T = rng.uniform(-0.6, 0.6, 3), float(rng.uniform(0.42, 0.7))
        m = targets(u, T)
        ok, F, lam, n, fail = solve(lib, phi, gaussian(phi, u, T), m, 0, 1, 0, 1, maxit=60, tol=1e-17)
        if not ok:
            continue
        failed += fail
        assert 3 <= n < 60 and fail == 1
        assert residual(F, phi, m) <= 1.1e-14
        assert np.abs(np.exp(lam @ phi) / F - 1).max() <= 4e-15
    assert failed > 40


@pytest.mark.parametrize("budget", [0, 1, 2])
def test_a_spent_budget_fails_as_the_fp64_iteration(lib, budget):
    phi = basis(lib)
    u, T = np.array([0.5, -0.3, 0.2]), 0.5
    lam, m = gaussian(phi, np.zeros(3), 0.6), targets(u, T)
    a = solve(lib, phi, lam, m, 0, 1, 0, 1, maxit=budget)
    b = solve(lib, phi, lam, m, 0, 1, 0, 0, maxit=budget)
    assert a[0] == b[0] == 1 and a[4] == b[4] == 1 and a[3] == b[3] == budget
    assert np.abs(a[1] - b[1]).max() <= 1e-9      # the same iterates: directions to 1e-11


def test_both_systems_give_up_the_same_cells_at_the_edge_of_the_cone(lib):
    phi = basis(lib)
    rng = np.random.default_rng(1)
    kept = left = 0
    for k in range(500):
        u = rng.uniform(-1, 1, 3) * (1, 1, 0)
        u *= rng.uniform(0.3, 1.7) / np.linalg.norm(u)
        T = float(rng.uniform(0.3, 0.6))
        lam, m = gaussian(phi, u, T), targets(u, T)
        a = solve(lib, phi, lam, m, 0, 1, 0, 1, maxit=30)
        b = solve(lib, phi, lam, m, 0, 1, 1, 1, maxit=30)
        assert a[0] == b[0]
        if a[0]:
            kept += 1
            assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2]) and a[3:] == b[3:]
        else:
            left += 1
    assert kept > 200 and left > 50


def test_gaussian_start(lib):
    rng = np.random.default_rng(9)
    x, y = np.empty(13), np.empty(13)
    for k in range(300):
        u, T = rng.uniform(-1, 1, 3), float(rng.uniform(0.3, 1.2))
        assert lib.fx_gaussian(p(u), T, p(x), p(y)) == 1
        assert np.array_equal(x[1:], y[1:]) and abs(x[0] - y[0]) <= 1e-15
    assert lib.fx_gaussian(p(np.array([0.1, 0.0, 0.0])), 0.05, p(x), p(y)) == 0  # 1/T = 20
