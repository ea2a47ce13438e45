"""The subspace eigensolver of the Davidson iteration on the host: couplings
far below the leading element of their column (1e-7 to 1e-12 of it), weakly
coupled blocks, degenerate and diagonal matrices; the residual at rounding
level and numpy's lowest eigenvalue."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_08154_gb300", "csrc")


@pytest.fixture(scope="module")
def solve(tmp_path_factory):
    d = tmp_path_factory.mktemp("eig")
    src, so = d / "shim.cpp", d / "shim.so"
    src.write_text('#include <vector>\n#include "lowest_eigenpair.h"\n'
                   'extern "C" double solve(int m, const double* a, double* y) {\n'
                   "  return qp::lowest_eigenpair(m, std::vector<double>(a, a + m * m), y);\n}\n")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(so)])
    lib = ctypes.CDLL(str(so))
    lib.solve.restype = ctypes.c_double
    P = ctypes.POINTER(ctypes.c_double)
    lib.solve.argtypes = [ctypes.c_int, P, P]

    def run(a):
        a = np.ascontiguousarray(a, dtype=np.float64)
        y = np.zeros(len(a))
        return lib.solve(len(a), a.ctypes.data_as(P), y.ctypes.data_as(P)), y

    return run


def _check(solve, a):
    """A backward stable reduction of order m leaves a residual of a few m ulp
    of the norm."""
    m, norm = len(a), np.abs(a).sum(axis=1).max()
    theta, y = solve(a)
    tol = 8 * m * np.finfo(float).eps * norm
    assert abs(np.linalg.norm(y) - 1.0) < 1e-14
    assert np.linalg.norm(a @ y - theta * y) <= tol
    assert abs(theta - np.linalg.eigvalsh(a)[0]) <= tol


@pytest.mark.parametrize("eps", [0.0, 1e-7, 2e-8, 1e-8, 5e-9, 1e-9, 1e-10, 1e-12])
@pytest.mark.parametrize("m", [3, 5, 17, 32])
def test_weak_couplings(solve, m, eps):
    rng = np.random.default_rng(m)
    # an arrow: one strong coupling in the first column, weak ones beyond it
    a = np.diag(-30.0 + 0.1 * np.arange(m))
    a[1, 1] = -28.0
    a[0, 1] = a[1, 0] = 1.0
    a[0, 2:] = a[2:, 0] = eps * (1.0 + rng.random(m - 2))
    _check(solve, a)
    # weakly coupled blocks with the same lowest element
    b = np.diag(np.where(np.arange(m) % 3 == 0, -30.0, -27.0 + 0.01 * np.arange(m)))
    w = rng.standard_normal((m, m)) * eps
    b += np.tril(w, -2) + np.tril(w, -2).T
    for i in range(0, m - 1, 3):
        b[i, i + 1] = b[i + 1, i] = 0.7
    _check(solve, b)


@pytest.mark.parametrize("m", [1, 2, 3, 8, 32])
def test_dense_degenerate_and_scaled(solve, m):
    rng = np.random.default_rng(100 + m)
    a = rng.standard_normal((m, m))
    a = a + a.T
    _check(solve, a)
    _check(solve, 1e-150 * a)
    _check(solve, np.zeros((m, m)))
    _check(solve, -2.0 * np.eye(m))
    q, _ = np.linalg.qr(rng.standard_normal((m, m)))
    e = np.linspace(0.0, 1.0, m)
    e[: min(m, 3)] = -5.0
    d = (q * e) @ q.T
    _check(solve, 0.5 * (d + d.T))
