"""The rational square root of the Lanczos control kernel, on the host copy of its
elimination: T^{1/2} e1 against the eigen-decomposition over the orders and spectra
that take it, and its refusal of spectra outside its window."""
import ctypes

import numpy as np
import pytest

import paper_1709_06946_gb300 as pkg


@pytest.fixture(scope='module')
def lib():
    pkg.build()
    return pkg.load()


def _lanczos_matrix(lam, n, rng):
    """Tridiagonal T (order n) of n exact Lanczos steps on diag(lam)."""
    v = rng.standard_normal(len(lam))
    V, al, be = [v / np.linalg.norm(v)], [], []
    for _ in range(n):
        w = lam * V[-1]
        al.append(V[-1] @ w)
        for _ in range(2):
            for q in V:
                w = w - (q @ w) * q
        be.append(np.linalg.norm(w))
        V.append(w / be[-1])
    return np.array(al), np.array(be[:n])


def _run(lib, al, be):
    c = np.zeros(len(al))
    p = [a.ctypes.data_as(ctypes.c_void_p) for a in (al, be, c)]
    return lib.pse_internal_rational_sqrt_e1(len(al), *p), c


# n = 64 is the longest recurrence the kernel keeps in shared memory; a condition
# number of 1e5 leaves the smallest Ritz value ten times above the window's edge.
# Quadrature error of the 31 nodes 1e-15, rounding of the eliminations and of the
# oracle's eigenvectors a few n eps: 1e-13 of |c|.
@pytest.mark.parametrize('n', [1, 2, 3, 31, 32, 33, 64])
@pytest.mark.parametrize('cond', [1.5, 100.0, 1e5])
def test_rational_square_root(lib, n, cond):
    rng = np.random.default_rng(n)
    al, be = _lanczos_matrix(np.geomspace(1.0 / cond, 1.0, 200) * 0.37, n, rng)
    rc, c = _run(lib, al, be)
    assert rc == 0
    w, Q = np.linalg.eigh(np.diag(al) + np.diag(be[:n - 1], 1) + np.diag(be[:n - 1], -1))
    ref = Q @ (np.sqrt(w) * Q[0])
    assert np.linalg.norm(c - ref) <= 1e-13 * np.linalg.norm(ref)


@pytest.mark.parametrize('low', [1e-8, 0.0, -1e-3])
def test_spectrum_outside_the_window_is_refused(lib, low):
    # T = [[a, b], [b, a]] with eigenvalues low and 1
    a, b = 0.5 * (1.0 + low), 0.5 * (1.0 - low)
    rc, _ = _run(lib, np.array([a, a]), np.array([b, 0.0]))
    assert rc == 1
