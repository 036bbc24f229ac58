"""GPU tests of the neighbour search of dilute systems (one thread per particle, taken
from about 91000 cells on): particles around a corner of the box, so that runs wrap on
either side of every axis, cells of many particles, more neighbours than slots, sheared
cells, several suspensions, and the largest numbers of cells below which the other form
is taken.  The real-space product sums over exactly the pairs of the list, so it is
compared with the oracle's (tolerances of the parity tests: relative L2 1e-10 in FP64,
2e-5 in FP32)."""
import numpy as np
import pytest

import pse_inputs

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu
TOL = {'fp64': 1e-10, 'mixed': 2e-5}
RC = 1.0 + np.sqrt(np.log(1e4)) / 0.7   # r_cut at xi = 0.7, tol = 1e-3


@pytest.fixture(scope='module')
def pkg():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import paper_1709_06946_gb300 as p
    p.build()
    p.load()
    return p


def _blob(n, seed):
    """n points of a jittered lattice of spacing 1.4 (neighbour counts far above a dilute system's)."""
    k = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing='ij'), -1).reshape(-1, 3)[:n]
    return 1.4 * g + np.random.default_rng(seed).uniform(-0.1, 0.1, (n, 3))


def _corner(n, L, seed):
    """Half of the particles around the corner of the box, the others spread over it."""
    r = np.random.default_rng(seed)
    b = _blob(n // 2, seed)
    b -= b.mean(0) if len(b) else 0.0
    return np.concatenate([b, r.uniform(0.0, L, (n - n // 2, 3))])


def _check(pkg, pos, Ls, prec, A=None):
    from oracle import params, pse as opse
    X = np.concatenate(pos)
    F, S = pse_inputs.moments(len(X), seed=7)
    if prec == 'mixed':
        F, S = F.astype(np.float32), S.astype(np.float32)
    kw = {} if A is None else {'deform': A}
    Ns = [len(x) for x in pos]
    h = pkg.PSE(*((Ns, Ls) if len(Ns) > 1 else (Ns[0], Ls[0])), xi=0.7, tol=1e-3, precision=prec, **kw)
    U, E = h.mobility(torch.tensor(X, device='cuda'), torch.tensor(F, device='cuda'), torch.tensor(S, device='cuda'),
                      parts='real')
    got = np.concatenate([U.double().cpu().numpy(), E.double().cpu().numpy()], 1)
    cells, at = 0, 0
    for q, (x, L) in enumerate(zip(pos, Ls)):
        inf = h.system_info(q)
        p = params.choose(len(x), L, 1.0, 1.0, 1.0, 0.7, 1e-3, Ng=inf['Ng'], P=inf['P'], rcut=inf['rcut'],
                          **({} if A is None else {'A': A}))
        b = slice(at, at + len(x))
        ref = np.concatenate(opse.mobility_apply(x, F[b].astype(np.float64), S[b].astype(np.float64), p,
                                                 parts=('real',)), 1)
        assert np.linalg.norm(got[b] - ref) < TOL[prec] * np.linalg.norm(ref)
        at += len(x)
        cells += inf['cells_per_side'] ** 3
    h.close()
    return cells


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
@pytest.mark.parametrize('nc,n', [(44, 500), (45, 61), (46, 500), (47, 2), (48, 900)])
def test_dilute_cells(pkg, prec, nc, n):
    L = 0.5 * RC * (nc + 0.01)
    assert _check(pkg, [_corner(n, L, nc + n)], [L], prec) == nc ** 3


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
def test_dilute_sheared_cells(pkg, prec):
    A = np.array([[1.0, 0.3, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    L = 0.5 * RC * 58.0
    assert _check(pkg, [_corner(400, L, 5) @ A.T], [L], prec, A) >= 91200


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
def test_dilute_suspensions(pkg, prec):
    Ls = [0.5 * RC * (nc + 0.01) for nc in (40, 5, 36)]
    pos = [_corner(n, L, n) for n, L in zip((300, 1, 173), Ls)]
    assert _check(pkg, pos, Ls, prec) >= 91200


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
def test_few_cells_beside_dilute_suspensions(pkg, prec):
    """Four cells per side (every cell once, nearest image by rounding) and five in the same launch."""
    Ls = [0.5 * RC * (nc + 0.01) for nc in (46, 4, 5)]
    pos = [_corner(260, Ls[0], 260)] + [pse_inputs.rsa_positions(n, 0.0, seed=n, L=L)[0] for n, L in zip((50, 60), Ls[1:])]
    assert _check(pkg, pos, Ls, prec) >= 91200
