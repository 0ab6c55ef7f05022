"""Bounded waits inside the passes that run out, and the grid after them.

The plane passes by tiles (forward variant 2, inverse variant 8) wait for tiles, the pencil
variants 2 and 4 for bulk copies.  OKMC_TILE_EXTRA makes the first wait for one tile more than
there is, OKMC_TMA_EXTRA_TX the second for more bytes than its copies bring: each CTA gives up
after 0.5 s, records the error and returns.  A second-kind tile of a plane waits for all tiles
of the first kind, so with the hook none of them runs, and every CTA gives up once.
"""
import time

import numpy as np
import pytest

import __graft_entry__
from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300.workload import scaled_population

pytestmark = pytest.mark.gpu


@pytest.fixture(scope='module', autouse=True)
def _lib():
    __graft_entry__.build()
    ok.load()


@pytest.mark.parametrize('which,variant,hook,value', [(0, 2, 'OKMC_TILE_EXTRA', '1'), (2, 8, 'OKMC_TILE_EXTRA', '1'),
                                                      (1, 2, 'OKMC_TMA_EXTRA_TX', '16'), (1, 4, 'OKMC_TMA_EXTRA_TX', '16')])
@pytest.mark.parametrize('n', [(32, 32, 32), (96, 96, 48)])
def test_a_wait_that_gives_up_leaves_a_grid_that_can_be_set_up_again(n, which, variant, hook, value, monkeypatch):
    """ETIMEOUT, again for the next call, and after okmc_set_defects on the same grid, with the
    same kernels, the tables, the stress and a trajectory of a fresh grid, bit for bit."""
    w = scaled_population(n, 8, seed=11, r111=(0.4, 1.0), r100=(0.4, 1.0))
    monkeypatch.setenv('OKMC_VARIANTS', '0,0,0')
    fresh = ok.Grid(w.n, w.voxel_nm, *w.C, seed=3)
    fresh.set_defects(w.defects)
    g = ok.Grid(w.n, w.voxel_nm, *w.C, seed=3)
    g.set_defects(w.defects)
    if not (g.variants()[1][which] >> variant) & 1:
        pytest.skip('no tensor maps on this device')
    monkeypatch.setenv(hook, value)
    g.set_variant(which, variant)  # reads the hook
    t0 = time.time()
    for _ in range(2):
        with pytest.raises(ok.OkmcError) as ei:
            g.solve_stress()
        assert ei.value.code == ok.OKMC_ETIMEOUT, ei.value
    assert 0.4 < time.time() - t0 < 30.0
    monkeypatch.delenv(hook)
    g.set_variant(which, variant)
    for _ in range(2):  # a count left behind by one pass would show in the next
        g.set_defects(w.defects)
        assert np.array_equal(g.self_terms(), fresh.self_terms())
        assert np.array_equal(g.solve_stress(), fresh.solve_stress())
    a, b = g.step(500.0, 4), fresh.step(500.0, 4)
    assert a['clock'] == b['clock'] and np.array_equal(g.get_positions(), fresh.get_positions())
    assert np.array_equal(g.solve_stress(), fresh.solve_stress())
    g.close()
    fresh.close()
