"""GPU tests of the 16^3-tile spreading and interpolation kernels on grids that 16 does not
divide (as equal tiles as leave the last one a support), and of the 11-moment product on
them: the wave-space part against the FP64 form (general kernels, same grid and support),
for two, three and four tiles per side, equal and ragged, narrow last tiles, every support
with its own instance, the full and reduced products, batches, and the general kernels
(forced by a fixed tile).  Relative L2 2e-5, the mixed form's parity tolerance."""
import numpy as np
import pytest

import pse_inputs

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu
TOL = 2e-5


@pytest.fixture(scope='module')
def pkg():
    if not torch.cuda.is_available():
        pytest.skip('no CUDA device')
    import paper_1709_06946_gb300 as p
    p.build()
    p.load()
    return p


def _inputs(N, L, seed=3):
    pos = pse_inputs.random_positions(N, L, seed=seed)
    pos[:4] = [[0.0, 0.0, 0.0], [L - 1e-9, L / 2, 1e-12], [0.45 * L, L - 1e-7, L - 1e-7], [-0.2, L + 0.3, 2.5 * L]]
    rng = np.random.default_rng(seed + 1)
    return pos, rng.standard_normal((N, 3)), rng.standard_normal((N, 3)), rng.standard_normal((N, 5))


def _t(x, prec):
    return torch.tensor(x, device='cuda', dtype=torch.float64 if prec == 'fp64' else torch.float32)


def _wave(pkg, pos, F, S, prec, want, L, Ng, P, **kw):
    h = pkg.PSE(len(pos), L, xi=0.5, tol=1e-3, precision=prec, Ng=Ng, P=P, rcut=7.0, **kw)
    out = h.mobility(torch.tensor(pos, device='cuda'), None if F is None else _t(F, prec), _t(S, prec), parts='wave',
                     want=want)
    out = torch.cat([x.double() for x in out if x is not None], 1).cpu().numpy()
    info = h.info
    h.close()
    return out, info


# (N_g, P, tile expected): 18 = 9 + 9, 20, 26, 36 equal; 44, 50, 54, 100 ragged (grids whose
# smallest divisor of a support's size does not fit shared memory, 46 or 106, are refused
# in either form)
CASES = [(18, 6, 9), (20, 8, 10), (26, 5, 13), (36, 6, 12), (36, 10, 12), (44, 8, 15), (50, 6, 13), (54, 6, 14),
         (54, 10, 14), (100, 8, 15)]


@pytest.mark.parametrize('Ng,P,T', CASES)
def test_products(pkg, Ng, P, T):
    L, N = 0.9 * Ng, 700
    pos, F, _, S = _inputs(N, L)
    for f, want in ((F, ('U', 'E')), (None, ('E',)), (F, ('U',)), (None, ('U',))):
        ref, _ = _wave(pkg, pos, f, S, 'fp64', want, L, Ng, P)
        got, info = _wave(pkg, pos, f, S, 'mixed', want, L, Ng, P)
        assert info['tile_kernels'] == 1 and info['tile'] == (T, T, T)
        assert np.linalg.norm(got - ref) < TOL * np.linalg.norm(ref), want


# enough tiles for the ring of planes (8 components from two tiles per SM, 5 from four)
@pytest.mark.parametrize('Ng,P,T,N', [(112, 6, 16, 30000), (130, 5, 15, 30000), (130, 6, 15, 900), (130, 8, 15, 30000),
                                      (130, 10, 15, 5000)])
def test_ring_of_planes(pkg, Ng, P, T, N):
    L = 0.9 * Ng
    pos, F, _, S = _inputs(N, L)
    for f, want in ((F, ('U', 'E')), (None, ('E',))):
        ref, _ = _wave(pkg, pos, f, S, 'fp64', want, L, Ng, P)
        got, info = _wave(pkg, pos, f, S, 'mixed', want, L, Ng, P)
        assert info['tile_kernels'] == 1 and info['tile'] == (T, T, T)
        assert np.linalg.norm(got - ref) < TOL * np.linalg.norm(ref), want


@pytest.mark.parametrize('Ng,tile', [(36, (12, 12, 12)), (54, (9, 9, 9)), (32, (8, 16, 16))])
def test_fixed_tiles_take_the_general_kernels(pkg, Ng, tile):
    L = 0.9 * Ng
    pos, F, _, S = _inputs(400, L)
    ref, _ = _wave(pkg, pos, F, S, 'fp64', ('U', 'E'), L, Ng, 6)
    got, info = _wave(pkg, pos, F, S, 'mixed', ('U', 'E'), L, Ng, 6, tile=tile)
    assert info['tile_kernels'] == 0
    assert np.linalg.norm(got - ref) < TOL * np.linalg.norm(ref)


@pytest.mark.parametrize('Ng,P', [(18, 6), (32, 5), (36, 8), (48, 6), (54, 10)])
def test_eleven_moments(pkg, Ng, P):
    L = 0.9 * Ng
    pos, F, Lt, S = _inputs(500, L)
    out = {}
    for prec in ('fp64', 'mixed'):
        h = pkg.PSE(len(pos), L, xi=0.5, tol=1e-3, precision=prec, Ng=Ng, P=P, rcut=7.0, torque=1)
        out[prec] = [x.double().cpu().numpy() for x in
                     h.mobility11(torch.tensor(pos, device='cuda'), _t(F, prec), _t(Lt, prec), _t(S, prec), parts='wave')]
        if prec == 'mixed':
            assert h.info['tile_kernels'] == 1
        h.close()
    for a, b in zip(out['mixed'], out['fp64']):
        assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b)


def test_sheared_eleven_moments(pkg):
    A = np.array([[1.0, 0.4, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])
    Ng, L = 48, 40.0
    pos, F, Lt, S = _inputs(500, L)
    pos = pos @ A.T
    out = {}
    for prec in ('fp64', 'mixed'):
        h = pkg.PSE(len(pos), L, xi=0.5, tol=1e-3, precision=prec, Ng=Ng, P=10, rcut=7.0, torque=1, deform=A)
        out[prec] = [x.double().cpu().numpy() for x in
                     h.mobility11(torch.tensor(pos, device='cuda'), _t(F, prec), _t(Lt, prec), _t(S, prec), parts='wave')]
        h.close()
    for a, b in zip(out['mixed'], out['fp64']):
        assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b)


def test_lattice_handles_keep_the_divisor(pkg):
    # a handle for the deformed cell may be given a deformation that couples z later
    A = np.eye(3)
    A[0, 1] = 0.3
    h = pkg.PSE(300, 32.4, xi=0.5, tol=1e-3, precision='mixed', Ng=36, P=8, rcut=7.0, deform=A)
    assert h.info['tile_kernels'] == 0 and all(36 % t == 0 for t in h.info['tile'])
    A[0, 1], A[0, 2] = 0.2, 0.05   # within the eigenvalues the handle was made for
    h.set_deformation(A)
    h.close()


def test_batch_of_ragged_grids(pkg):
    Ns, Ls = [900, 400, 2500, 300], [26.0, 19.0, 41.0, 15.5]
    ins = [_inputs(n, L, seed=10 + n) for n, L in zip(Ns, Ls)]
    pos, F, S = (np.concatenate([i[k] for i in ins]) for k in (0, 1, 3))
    out = {}
    for prec in ('fp64', 'mixed'):
        h = pkg.PSE(Ns, Ls, xi=0.5, tol=1e-3, precision=prec)
        U, E = h.mobility(torch.tensor(pos, device='cuda'), _t(F, prec), _t(S, prec), parts='wave')
        out[prec] = torch.cat([U.double(), E.double()], 1).cpu().numpy()
        grids = [h.system_info(q)['Ng'] for q in range(4)]
        h.close()
    at = 0
    for n in Ns:
        a, b = out['mixed'][at:at + n], out['fp64'][at:at + n]
        assert np.linalg.norm(a - b) < TOL * np.linalg.norm(b), grids
        at += n
