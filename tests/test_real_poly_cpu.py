"""The FP32 fit of the real-space functions beyond contact (host copy of the pair sum's
evaluation) against the functions themselves, and the rule that refuses it."""
import ctypes
import math

import numpy as np
import pytest

import paper_1709_06946_gb300 as pkg

FIT_TOL = 1.5e-6


@pytest.fixture(scope='module')
def lib():
    pkg.build()
    lb = pkg.load()
    lb.pse_internal_real_poly.restype = ctypes.c_double
    return lb


def _both(lib, xi, rcut, r):
    p = [ctypes.c_double(v) for v in (1.0, 1.0, xi)]
    out = np.zeros((len(r), 7), np.float32)
    err = lib.pse_internal_real_poly(*p, ctypes.c_double(rcut), len(r), r.ctypes.data_as(ctypes.c_void_p),
                                     out.ctypes.data_as(ctypes.c_void_p))
    f = np.zeros((len(r), 7))
    r64 = r.astype(np.float64)
    lib.pse_internal_real_functions(*p, len(r), r64.ctypes.data_as(ctypes.c_void_p), f.ctypes.data_as(ctypes.c_void_p), None)
    f[:, 1] -= f[:, 0]
    return err, np.abs(out - f).max(0) / np.abs(f).max(0)


# Fit error at most FIT_TOL of the maximum, plus the rounding of eight FP32 steps
# (8 x 6e-8) and of a Gaussian whose exponent reaches ln(10/tol) (12 x 6e-8), twice over.
@pytest.mark.parametrize('xi,tol', [(0.4, 1e-3), (0.45, 1e-4), (0.5, 1e-3), (0.5, 1e-6), (0.6, 1e-3), (1.0, 1e-3), (2.0, 1e-4)])
def test_fit_beyond_contact(lib, xi, tol):
    rcut = 1.0 + math.sqrt(math.log(10.0 / tol)) / xi
    r = np.linspace(2.00001, rcut, 4001).astype(np.float32)
    err, off = _both(lib, xi, rcut, r)
    assert err <= 1.0   # at least as close as the table
    assert off.max() <= FIT_TOL + 2 * 20 * 6e-8


@pytest.mark.parametrize('xi,rcut', [(0.2, 16.0), (0.5, 2.0), (0.5, 1.5)])
def test_fit_is_refused(lib, xi, rcut):
    err, _ = _both(lib, xi, rcut, np.array([2.1], np.float32))
    assert not err <= 1.0
