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


def test_a_rejected_probe_does_not_hide_an_earlier_error(monkeypatch):
    """A device-side probe off the lattice is reported once and cleared; a wait that gave up
    before it stays reported until okmc_set_defects."""
    torch = pytest.importorskip('torch')
    w = scaled_population((32, 32, 32), 8, seed=11, r111=(0.4, 1.0), r100=(0.4, 1.0))
    monkeypatch.setenv('OKMC_VARIANTS', '0,0,0')
    g = ok.Grid(w.n, w.voxel_nm, *w.C, seed=3)
    g.set_defects(w.defects)
    pos = torch.tensor([[1, 2, 2]], dtype=torch.int32, device='cuda')
    P = torch.ones((1, 6), dtype=torch.float64, device='cuda')
    E = torch.zeros(1, dtype=torch.float64, device='cuda')
    torch.cuda.synchronize()

    def probe():
        return g.lib.okmc_point_dipole_energies(g.h, pos.data_ptr(), P.data_ptr(), 1, E.data_ptr(), 1)
    assert probe() == ok.OKMC_EINVAL and bool(torch.isnan(E[0]))
    ref = g.solve_stress()  # cleared
    monkeypatch.setenv('OKMC_TILE_EXTRA', '1')
    g.set_variant(2, 8)
    assert probe() == ok.OKMC_ETIMEOUT
    monkeypatch.delenv('OKMC_TILE_EXTRA')
    g.set_variant(2, 8)
    with pytest.raises(ok.OkmcError) as ei:
        g.stats()
    assert ei.value.code == ok.OKMC_ETIMEOUT
    g.set_defects(w.defects)
    assert np.array_equal(g.solve_stress(), ref)
    g.close()
