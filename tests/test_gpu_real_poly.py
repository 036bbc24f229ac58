"""GPU tests of the pair sum's function sources: the polynomial fit beyond contact, with
the table below it, against the all-table form (option table_points set) and the FP64
form, over the products, lanes and contact distances (2a exactly, a rounding step to either
side, deep overlap, r_cut).  Tolerance of the mixed form's parity tests, 2e-5."""
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


def _positions(n, L, xi):
    """Pairs at chosen distances along x on a coarse lattice: overlaps, contact, the cutoff."""
    rc = 1.0 + np.sqrt(np.log(1e4)) / xi
    d = np.array([0.3, 1.0, 1.9, 2.0 - 1e-6, 2.0, 2.0 + 1e-6, 2.1, 3.0, rc - 1e-5, rc + 1e-5])
    base = pse_inputs.rsa_positions(n, 0.0, seed=5, L=L)[0]
    return np.concatenate([base, base + np.stack([d[np.arange(n) % len(d)], np.zeros(n), np.zeros(n)], 1)])


@pytest.mark.parametrize('xi', [0.5, 0.8])
@pytest.mark.parametrize('lanes', [0, 1, 4, 8, 16, 32])
@pytest.mark.parametrize('product', ['full', 'se', 'fsu', 'su'])
def test_fit_against_table_and_fp64(pkg, product, lanes, xi):
    L, n = 20.0, 150
    pos = torch.tensor(_positions(n, L, xi), device='cuda')
    F, S = pse_inputs.moments(2 * n, seed=6)
    kw = {'full': (True, True, ('U', 'E')), 'se': (False, True, ('E',)), 'fsu': (True, True, ('U',)),
          'su': (False, True, ('U',))}[product]

    def run(prec, **opts):
        dt = torch.float64 if prec == 'fp64' else torch.float32
        h = pkg.PSE(2 * n, L, xi=xi, tol=1e-3, precision=prec, real_lanes=lanes, **opts)
        out = h.mobility(pos, torch.tensor(F, device='cuda', dtype=dt) if kw[0] else None,
                         torch.tensor(S, device='cuda', dtype=dt), parts='real', want=kw[2])
        out = torch.cat([x.double() for x in out if x is not None], 1).cpu().numpy()
        h.close()
        return out
    ref, fit, table = run('fp64'), run('mixed'), run('mixed', table_points=1024)
    for x in (fit, table):
        assert np.linalg.norm(x - ref) < 2e-5 * np.linalg.norm(ref)
    # the fit is the closer of the two, or both are at the rounding level of FP32
    assert np.linalg.norm(fit - ref) <= max(np.linalg.norm(table - ref), 1e-6 * np.linalg.norm(ref))
