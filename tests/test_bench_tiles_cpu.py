"""bench.py names the kernels that a handle launched: the tile kernels also run on tiles
that are no 16^3 (ragged grids), and not on every 16^3 tiling; and it says that the pair
sum's rate counts the formulas' operations."""
import importlib.util
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope='module')
def bench():
    spec = importlib.util.spec_from_file_location('bench_under_test', os.path.join(ROOT, 'bench.py'))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


@pytest.mark.parametrize('tile,ran', [([16, 16, 16], 1), ([14, 14, 14], 1), ([12, 12, 12], 1), ([16, 16, 16], 0)])
def test_kernels_are_named_as_launched(bench, tile, ran):
    assert bench.uses_tile_kernels({'tile': tile, 'tile_kernels': ran}) == bool(ran)


def test_pair_sum_rate_names_its_operations(bench):
    v = ('full', 'se', 'fsu', 'su')
    st = ('spread', 'interp', 'scale', 'noise', 'real')
    prof = {'variant_ms': {s: {k: 0.0 for k in v} for s in st}, 'variant_calls': {s: {k: 0 for k in v} for s in st}}
    prof['variant_ms']['real']['se'], prof['variant_calls']['real']['se'] = 4.0, 10
    k, = bench.kernel_instances(prof, 1000, 54, 6, 1e5, True)
    assert 'no utilisation' in k['flops_note']
