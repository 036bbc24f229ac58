"""GPU tests of the Krylov control arithmetic: the Newton reciprocal and square root
against FP64's own, the tridiagonal square root of the Lanczos kernel on either side of
its two lines (orders above 64 and spectra outside the rational form's window go to the
serial eigensolver), and whole samples on both sides of order 64."""
import ctypes

import numpy as np
import pytest

import pse_inputs

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope='module')
def pkg():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import paper_1709_06946_gb300 as p
    p.build()
    p.load()
    return p


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_reciprocal_and_root(pkg):
    """Two units in the last place (a rounded Newton step and the final correction, each half a unit and
    the rounding of its residual), over the FP64 range and at both ends of the FP32-seeded one."""
    r = np.random.default_rng(3)
    edge = np.array([1e-30, 1e30])[:, None] * (1.0 + np.array([-1e-6, -6e-8, -1e-12, 0.0, 1e-12, 6e-8, 1e-6]))
    x = np.concatenate([10.0 ** r.uniform(-300, 300, 20000), 10.0 ** r.uniform(-31, 31, 20000), edge.ravel(),
                        2.0 ** np.arange(-1000, 1000, 7), [1.0, 4.0, 1.0 - EPS / 2, 1.0 + EPS]])
    x = np.concatenate([x, -x, [0.0, -0.0, np.inf, -np.inf, np.nan, 1e-320]])
    rec, rt = np.empty_like(x), np.empty_like(x)
    assert pkg.load().pse_internal_device_scalars(len(x), _ptr(x), _ptr(rec), _ptr(rt)) == 0
    with np.errstate(all='ignore'):
        for got, ref in ((rec, 1.0 / x), (rt, np.sqrt(x))):
            fin = np.isfinite(ref) & (ref != 0)
            assert np.max(np.abs(got[fin] - ref[fin]) / np.abs(ref[fin])) <= 2 * EPS
            assert np.array_equal(got[~fin], ref[~fin], equal_nan=True)


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


def _sqrt_e1(pkg, al, be):
    c = np.zeros(len(al))
    be = np.append(be[:len(al) - 1], 0.0)
    assert pkg.load().pse_internal_device_sqrt_e1(len(al), _ptr(al), _ptr(be), _ptr(c)) == 0
    w, Q = np.linalg.eigh(np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1))
    ref = Q @ (np.sqrt(np.maximum(w, 0.0)) * Q[0])
    return np.linalg.norm(c - ref) / np.linalg.norm(ref)


# as on the host: quadrature 1e-15, eliminations and the oracle's eigenvectors a few n eps
@pytest.mark.parametrize('n', [1, 2, 3, 31, 32, 33, 63, 64, 65, 80, 120])
@pytest.mark.parametrize('cond', [1.5, 100.0, 1e5])
def test_square_root_of_the_tridiagonal(pkg, n, cond):
    al, be = _lanczos_matrix(np.geomspace(1.0 / cond, 1.0, 200) * 0.37, n, np.random.default_rng(n))
    assert _sqrt_e1(pkg, al, be) <= 1e-13 * max(1.0, n / 64)


# a smallest eigenvalue w is known to n eps of the largest, its root to n eps / (2 sqrt(w)), at most sqrt(n eps)
@pytest.mark.parametrize('n', [2, 40, 64, 65])
@pytest.mark.parametrize('low', [1e-8, 0.0, -1e-3])
def test_spectrum_outside_the_window(pkg, n, low):
    if n == 2:
        al, be = np.full(2, 0.5 * (1.0 + low)), np.array([0.5 * (1.0 - low), 0.0])
    else:
        lam = np.append(np.linspace(0.1, 1.0, 199), low)
        al, be = _lanczos_matrix(lam, n, np.random.default_rng(n))
    tol = 1e-13 + 4 * n * EPS / (2 * np.sqrt(max(low, n * EPS)))
    assert _sqrt_e1(pkg, al, be) <= tol


@pytest.mark.parametrize('m', [63, 64, 65, 80])
def test_samples_around_order_64(pkg, m):
    """Fixed Lanczos lengths on both sides of the warp's order against the oracle's Lanczos (FP64)."""
    from oracle import params, pse as opse
    N, phi, xi, tol, dt = 200, 0.2, 0.6, 1e-3, 1e-3
    pos, L = pse_inputs.rsa_positions(N, phi, seed=29)
    h = pkg.PSE(N, L, xi=xi, tol=tol, precision='fp64', lanczos_tol=0.0, lanczos_maxiter=m)
    inf = h.info
    p = params.choose(N, L, 1.0, 1.0, 1.0, xi, tol, Ng=inf['Ng'], P=inf['P'], rcut=inf['rcut'])
    w1 = pse_inputs.lanczos_noise(N, seed=30)
    w2 = pse_inputs.wave_noise(p.Ng, seed=31)
    U, E, st = h.brownian(torch.tensor(pos, device='cuda'), dt, w1=torch.tensor(w1, device='cuda'),
                          w2=torch.tensor(w2, device='cuda'))
    B, sto = opse.brownian_sample(pos, dt, w1, w2, p, lanczos_tol=0.0, lanczos_maxiter=m)
    h.close()
    assert st['lanczos_iters'] == m and sto['lanczos_iters'] == m
    got = np.concatenate([U.cpu().numpy(), E.cpu().numpy()], 1)
    assert np.linalg.norm(got - B) < 1e-10 * np.linalg.norm(B)


def test_batch_stopping_on_both_sides_of_order_64(pkg):
    """Suspensions of one handle that stop at orders below and above 64 give their own handles' samples."""
    Ns, Ls, pos = [], [], []
    for n, phi, ideal in ((150, 0.05, False), (500, 1.5, True), (250, 0.25, False)):
        L = (4.0 * np.pi * n / (3.0 * phi)) ** (1.0 / 3.0)
        x = np.random.default_rng(n).uniform(0, L, (n, 3)) if ideal else pse_inputs.rsa_positions(n, phi, seed=n)[0]
        Ns.append(n)
        Ls.append(L)
        pos.append(x)
    opts = dict(xi=0.9, tol=1e-3, precision='fp64', lanczos_tol=1e-10, lanczos_maxiter=120)
    w1 = [pse_inputs.lanczos_noise(n, seed=n) for n in Ns]
    hb = pkg.PSE(Ns, Ls, **opts)
    w2 = [pse_inputs.wave_noise(hb.system_info(q)['Ng'], seed=q) for q in range(3)]

    def dev(a):
        return torch.tensor(np.ascontiguousarray(a), device='cuda')
    U, E, _ = hb.brownian(dev(np.concatenate(pos)), 1e-3, w1=dev(np.concatenate(w1)),
                          w2=dev(np.concatenate([w.reshape(-1) for w in w2])))
    its = [hb.system_stats(q)['lanczos_iters'] for q in range(3)]
    hb.close()
    assert min(its) <= 64 < max(its) < 120, its
    got = np.concatenate([U.cpu().numpy(), E.cpu().numpy()], 1)
    at = 0
    for q, n in enumerate(Ns):
        h = pkg.PSE(n, Ls[q], **opts)
        Us, Es, st = h.brownian(dev(pos[q]), 1e-3, w1=dev(w1[q]), w2=dev(w2[q]))
        h.close()
        assert st['lanczos_iters'] == its[q]
        ref = np.concatenate([Us.cpu().numpy(), Es.cpu().numpy()], 1)
        assert np.linalg.norm(got[at:at + n] - ref) < 1e-10 * np.linalg.norm(ref)
        at += n
