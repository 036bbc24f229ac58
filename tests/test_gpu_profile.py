"""GPU test of the stage profile: a stage's calls are the products that the Krylov
solves took, one per iteration, so that its time over its calls is a launch's time."""
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


@pytest.mark.parametrize('cap', [0, 3])
def test_profile_counts_the_iterations(pkg, cap):
    """One step without a force: Lanczos takes full products in real space alone, GMRES S -> E
    products, and the final velocity one S -> U product.  cap: both solves end at their
    iteration caps instead of their tolerances."""
    N = 2000
    pos, L = pse_inputs.rsa_positions(N, 0.2, seed=151)
    opts = {} if cap == 0 else {'lanczos_tol': 0.0, 'lanczos_maxiter': cap, 'krylov_tol': 0.0, 'krylov_maxiter': cap}
    h = pkg.PSE(N, L, xi=0.5, tol=1e-3, precision='mixed', **opts)
    x = torch.tensor(pos, device='cuda', dtype=torch.float64)
    h.set_profiling(True)
    _, st = h.step(x, 1e-3, seed=1, step=0)
    lz, gm = st['lanczos_iters'], st['krylov_iters']
    assert (lz, gm) == (cap, cap) if cap else min(lz, gm) >= 3
    calls = h.profile()['variant_calls']
    h.close()
    assert calls['real']['full'] == lz and calls['spread']['full'] == 0
    for stage in ('real', 'spread', 'scale', 'interp'):
        assert calls[stage]['se'] == gm, stage
    assert calls['real']['su'] == calls['spread']['su'] == calls['interp']['su'] == 1
