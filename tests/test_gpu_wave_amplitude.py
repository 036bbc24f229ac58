"""GPU test of the tile kernels' weights (mixed precision): the amplitude of the wave
part, its projection on the FP64 form's, against that of the general kernels (forced by
an explicit tile), whose exponentials are unbiased.  The transforms and the scaling are
the same and cancel.  Of the five exponentials in a particle's weights (two to spread,
three to interpolate) only the spreading's in x and y is the special-function unit's
2^x, low by 4.8e-8 on average; the roundings of the constants scatter by 1.2e-7 from
size to size, 3.5e-8 in the mean over twelve: 8.5e-8."""
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


def _wave(pkg, pos, L, F, Lt, S, prec, **opts):
    dt = torch.float64 if prec == 'fp64' else torch.float32
    h = pkg.PSE(len(pos), L, xi=0.5, tol=1e-3, precision=prec, torque=1, **opts)
    x = torch.tensor(pos, device='cuda')
    f, t, s = (torch.tensor(a, device='cuda').to(dt) for a in (F, Lt, S))
    out = [torch.cat([v.double().ravel() for v in r]) for r in (h.mobility(x, f, s, parts='wave'),
                                                               h.mobility11(x, f, t, s, parts='wave'))]
    inf = h.info
    h.close()
    return out, inf


def test_tile_kernels_keep_the_amplitude(pkg):
    diff = []
    for k, n in enumerate((1010, 1174, 2236, 3098, 3179, 4679, 4940, 5280, 7347, 13329, 19635, 20133)):
        phi = 0.09 + 0.017 * k
        pos, L = pse_inputs.rsa_positions(n, min(phi, 0.28), seed=200 + k)
        F, S = (a.astype(np.float32) for a in pse_inputs.moments(n, seed=300 + k))
        Lt = pse_inputs.moments(n, seed=400 + k)[0].astype(np.float32)
        ref, inf = _wave(pkg, pos, L, F, Lt, S, 'fp64')
        opts = {'Ng': inf['Ng'], 'P': inf['P']}
        tile, ti = _wave(pkg, pos, L, F, Lt, S, 'mixed', **opts)
        side = next(t for t in (8, 12, 9, 10) if inf['Ng'] % t == 0)
        gen, gi = _wave(pkg, pos, L, F, Lt, S, 'mixed', tile=(side,) * 3, **opts)
        assert ti['tile_kernels'] == 1 and gi['tile_kernels'] == 0
        diff.append([float((a - b) @ r / (r @ r)) for a, b, r in zip(tile, gen, ref)])
    mean = np.mean(diff, axis=0)
    assert np.abs(mean).max() < 8.5e-8, (mean, diff)
