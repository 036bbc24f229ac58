"""The captured step graph after an autotuning that failed half-way, on the host side
alone (a CUDA runtime without a device, tests/fake_cuda.c): the graph holds the tiles,
lanes and addresses that the tuner changes, so the next step has to capture it anew,
wherever the tuner stopped."""
import os
import subprocess
import sys

import pytest

import paper_1709_06946_gb300 as pkg
from paper_1709_06946_gb300 import builder

HERE = os.path.dirname(os.path.abspath(__file__))

CHILD = r'''
import ctypes, sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import paper_1709_06946_gb300 as pkg
fake = ctypes.CDLL(sys.argv[2])
h = pkg.PSE(500, 60.0, xi=0.5, tol=1e-3, precision=sys.argv[3], use_graph=1)
x = np.random.default_rng(1).uniform(0.0, 60.0, (500, 3))
h.step(x, 1e-3, seed=1, step=0)
h.step(x, 1e-3, seed=1, step=1)
assert fake.fake_captures() == 1, fake.fake_captures()
fake.fake_fail_malloc(int(sys.argv[4]))
try:
    h.autotune(x, reps=1)
except pkg.PSEError as e:
    assert e.code == 2, e
else:
    raise SystemExit('the autotuner did not fail')
h.step(x, 1e-3, seed=1, step=2)
assert fake.fake_captures() == 2, 'the graph of the old tiles ran again'
h.step(x, 1e-3, seed=1, step=3)
assert fake.fake_captures() == 2
h.autotune(x, reps=1)
h.step(x, 1e-3, seed=1, step=4)
assert fake.fake_captures() == 3
'''


@pytest.fixture(scope='module')
def fake(tmp_path_factory):
    pkg.build()
    out = str(tmp_path_factory.mktemp('fake') / 'libfake_cuda.so')
    subprocess.run(['gcc', '-shared', '-fPIC', '-O1', '-w', '-I' + os.path.join(builder.CUDA, 'include'),
                    os.path.join(HERE, 'fake_cuda.c'), '-o', out], check=True)
    return out


# the tuner's first allocations belong to its first larger tiling: counts, then tile starts
@pytest.mark.parametrize('prec', ['mixed', 'fp64'])
@pytest.mark.parametrize('failing', [1, 2])
def test_graph_is_captured_anew_after_a_failed_autotuning(fake, prec, failing):
    r = subprocess.run([sys.executable, '-c', CHILD, os.path.dirname(HERE), fake, prec, str(failing)],
                       env={**os.environ, 'LD_PRELOAD': fake}, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
