"""GPU tests of the graph step's guarded outputs: a step that fails (a position or a force
that is not finite) leaves the caller's positions and stresslets as they were, and a step
whose neighbour lists overflow in the captured graph writes both from its rerun; device
and host arrays."""
import ctypes

import numpy as np
import pytest

import pse_inputs

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module')
def pkg():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import paper_1709_06946_gb300 as p
    p.build()
    p.load()
    return p


def _arr(a, device, dtype=None):
    """A copy on the device or on the host."""
    a = np.array(a, dtype=dtype, order='C')
    return torch.tensor(a, device='cuda') if device else a


def _np(a):
    return a.cpu().numpy() if isinstance(a, torch.Tensor) else a.copy()


def _addr(a):
    return None if a is None else (a.data_ptr() if isinstance(a, torch.Tensor) else a.ctypes.data)


def _step(pkg, h, x, S, FP=None, step=0):
    """pse_constrained_step into the caller's own stresslets; the status."""
    from paper_1709_06946_gb300 import binding
    st = binding.Stats()
    rc = pkg.load().pse_constrained_step(h._h, _addr(x), _addr(FP), 1e-3, 11, step, _addr(S), ctypes.byref(st),
                                         torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return rc


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
@pytest.mark.parametrize('device', [True, False])
@pytest.mark.parametrize('what', ['position', 'force'])
@pytest.mark.parametrize('bad', [np.nan, np.inf])
def test_failed_step_writes_nothing(pkg, prec, device, what, bad):
    N, dt = 300, np.float64 if prec == 'fp64' else np.float32
    pos, L = pse_inputs.rsa_positions(N, 0.1, seed=161)
    F = pse_inputs.moments(N, seed=162)[0]
    h = pkg.PSE(N, L, xi=0.5, tol=1e-3, precision=prec, use_graph=1)
    mark = np.random.default_rng(1).standard_normal((N, 5)).astype(dt)
    x, S, FP = _arr(pos, device), _arr(mark, device), _arr(F, device, dt)
    assert _step(pkg, h, x, S, FP) == 0 and h.graph_ready()[0]
    good = _np(x)
    assert not np.array_equal(_np(S), mark)
    bx, bF = good.copy(), F.copy()
    (bx if what == 'position' else bF)[N // 2, 1] = bad
    x, S = _arr(bx, device), _arr(mark, device)
    assert _step(pkg, h, x, S, _arr(bF, device, dt), step=1) == 5
    assert np.array_equal(_np(x), bx, equal_nan=True) and np.array_equal(_np(S), mark)
    # the handle goes on: the same step with finite inputs
    x, S = _arr(good, device), _arr(mark, device)
    assert _step(pkg, h, x, S, FP, step=1) == 0
    assert not np.array_equal(_np(x), good) and not np.array_equal(_np(S), mark) and np.isfinite(_np(S)).all()
    h.close()


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
@pytest.mark.parametrize('device', [True, False])
def test_overflowing_lists_are_rerun(pkg, prec, device):
    """Captured on a dilute configuration, then a cluster of 343 touching spheres, of which each has more
    neighbours than a dilute system's slots; against a host-launched handle."""
    N, dt = 400, np.float64 if prec == 'fp64' else np.float32
    dilute, L = pse_inputs.rsa_positions(N, 0.005, seed=171)
    g = 2.1 * np.stack(np.meshgrid(*[np.arange(7)] * 3, indexing='ij'), -1).reshape(-1, 3) + 0.3 * L
    far = dilute[(np.abs(dilute - (0.3 * L + 6.3)) > 12.0).any(1)][:N - 343]
    assert len(far) == N - 343
    pos = np.concatenate([g, far])
    hg = pkg.PSE(N, L, xi=0.5, tol=1e-3, precision=prec, use_graph=1)
    hh = pkg.PSE(N, L, xi=0.5, tol=1e-3, precision=prec)
    x = _arr(dilute, device)
    assert _step(pkg, hg, x, _arr(np.zeros((N, 5), dt), device)) == 0 and hg.graph_ready()[0]
    for k in (1, 2):   # the overflow and its rerun, then the recaptured graph
        xg, xh = _arr(pos, device), _arr(pos, True)
        Sg, Sh = _arr(np.full((N, 5), 7.0, dt), device), _arr(np.zeros((N, 5), dt), True)
        assert _step(pkg, hg, xg, Sg, step=k) == 0 and _step(pkg, hh, xh, Sh, step=k) == 0
        a, b = _np(xg) - pos, _np(xh) - pos
        a, b = a - L * np.rint(a / L), b - L * np.rint(b / L)
        tol = 1e-10 if prec == 'fp64' else 1e-5
        assert np.linalg.norm(a - b) < tol * np.linalg.norm(b)
        assert np.linalg.norm(_np(Sg) - _np(Sh)) < tol * np.linalg.norm(_np(Sh))
    hg.close()
    hh.close()
