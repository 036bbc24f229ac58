"""GPU tests of the neighbour search where its cell-wise warps can go wrong: four cells
per side (every cell visited, nearest image by rounding), five (each cell once, runs that
wrap), six and seven, cells with more particles than the warp tests at once, a single
particle, several suspensions, sheared cells.  The real-space product sums over exactly
the pairs of the list, so it is compared with the oracle's (tolerances of the parity
tests: relative L2 1e-10 in FP64, 2e-5 in FP32)."""
import numpy as np
import pytest

import pse_inputs

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu
TOL = {'fp64': 1e-10, 'mixed': 2e-5}


@pytest.fixture(scope='module')
def pkg():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import paper_1709_06946_gb300 as p
    p.build()
    p.load()
    return p


def _oracle(pos, F, S, L, inf, A=None):
    from oracle import params, pse as opse
    kw = {} if A is None else {'A': A}
    p = params.choose(len(pos), L, 1.0, 1.0, 1.0, 0.7, 1e-3, Ng=inf['Ng'], P=inf['P'], rcut=inf['rcut'], **kw)
    return np.concatenate(opse.mobility_apply(pos, F, S, p, parts=('real',)), 1)


def _run(pkg, pos, L, prec, A=None):
    N = len(pos)
    F, S = pse_inputs.moments(N, seed=7)
    if prec == 'mixed':
        F, S = F.astype(np.float32), S.astype(np.float32)
    h = pkg.PSE(N, L, xi=0.7, tol=1e-3, precision=prec, **({} if A is None else {'deform': A}))
    U, E = h.mobility(torch.tensor(pos, device='cuda'), torch.tensor(F, device='cuda'), torch.tensor(S, device='cuda'),
                      parts='real')
    got = np.concatenate([U.double().cpu().numpy(), E.double().cpu().numpy()], 1)
    ref = _oracle(pos, F.astype(np.float64), S.astype(np.float64), L, h.info, A)
    nc = h.info['cells_per_side']
    h.close()
    return np.linalg.norm(got - ref) / np.linalg.norm(ref), nc


def _blob(n, seed):
    """n points of a jittered lattice of spacing 1/2 (many particles in one cell)."""
    k = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing='ij'), -1).reshape(-1, 3)[:n]
    return 0.5 * g + np.random.default_rng(seed).uniform(-0.04, 0.04, (n, 3))


RC = 1.0 + np.sqrt(np.log(1e4)) / 0.7   # r_cut at xi = 0.7, tol = 1e-3


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
@pytest.mark.parametrize('nc', [4, 5, 6, 7])
def test_few_cells_per_side(pkg, prec, nc):
    L = 0.5 * RC * (nc + 0.01)
    pos = pse_inputs.rsa_positions(60, 0.0, seed=3 + nc, L=L)[0] + np.array([0.0, -0.3 * L, 5.0 * L])
    err, got = _run(pkg, pos, L, prec)
    assert got == nc and err < TOL[prec]


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
@pytest.mark.parametrize('n', [1, 2, 5, 33, 150])
def test_crowded_cells(pkg, prec, n):
    # a blob across the corner of the box: cells of up to about 100 particles, wrapped runs
    L = 0.5 * RC * 6.5
    pos = _blob(n, seed=n) - 0.4
    err, _ = _run(pkg, pos, L, prec)
    assert err < TOL[prec]


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
@pytest.mark.parametrize('strain', [0.3, 0.5])
def test_sheared_cells(pkg, prec, strain):
    A = np.array([[1.0, strain, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    L = 0.5 * RC * 8.2
    pos = pse_inputs.rsa_positions(90, 0.0, seed=9, L=L)[0] @ A.T
    err, _ = _run(pkg, pos, L, prec, A)
    assert err < TOL[prec]


@pytest.mark.parametrize('prec', ['fp64', 'mixed'])
def test_suspensions_share_the_search(pkg, prec):
    Ls = [0.5 * RC * (nc + 0.01) for nc in (4, 9, 5)]
    pos = [pse_inputs.rsa_positions(n, 0.0, seed=20 + n, L=L)[0] for n, L in zip((40, 300, 1), Ls)]
    X = np.concatenate(pos)
    F, S = pse_inputs.moments(len(X), seed=7)
    if prec == 'mixed':
        F, S = F.astype(np.float32), S.astype(np.float32)
    h = pkg.PSE([len(x) for x in pos], Ls, xi=0.7, tol=1e-3, precision=prec)
    U, E = h.mobility(torch.tensor(X, device='cuda'), torch.tensor(F, device='cuda'), torch.tensor(S, device='cuda'),
                      parts='real')
    got = np.concatenate([U.double().cpu().numpy(), E.double().cpu().numpy()], 1)
    at = 0
    for q, (x, L) in enumerate(zip(pos, Ls)):
        b = slice(at, at + len(x))
        ref = _oracle(x, F[b].astype(np.float64), S[b].astype(np.float64), L, h.system_info(q))
        assert np.linalg.norm(got[b] - ref) < TOL[prec] * np.linalg.norm(ref)
        at += len(x)
    h.close()
