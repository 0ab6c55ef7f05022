"""Plane passes by tiles (forward variant 2, inverse variant 8) and the pencil pass by steps
of the block (variants 3 and 4) against variant 0 where only some planes are transformed: a
few dirty planes, and the plane lists of a kinetic step.  Equality is exact: the variants
round alike (full passes: test_pass_variants_bitwise_equal)."""
import numpy as np
import pytest

import __graft_entry__
from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300.workload import FE_CUBIC, LOOP_111, ONE_D, SIA_CLUSTER, THREE_D, make_defects

pytestmark = pytest.mark.gpu
H = 0.2855


@pytest.fixture(scope='module', autouse=True)
def _lib():
    __graft_entry__.build()
    ok.load()


def _grid(monkeypatch, n, variants):
    monkeypatch.setenv('OKMC_VARIANTS', variants)
    g = ok.Grid(n, H, *FE_CUBIC, seed=7)
    # a loop across the periodic faces, a single atom, a loop in the middle
    pos = np.array([[0, 0, 2 * n[2] - 2], [9, 11, n[2] // 2 * 2 + 1], [n[0], n[1], n[2]]])
    pos[1] |= 1
    pos[2] &= ~1
    g.set_defects(make_defects([LOOP_111, SIA_CLUSTER, LOOP_111], pos, [0, 1, 2], [0.8, 0.0, 0.6], [0, 1, 0], [0.1] * 3,
                               [ONE_D, THREE_D, ONE_D]))
    got, avail = g.variants()
    want = [int(x) for x in variants.split(',')]
    if not (avail[1] >> 4) & 1 and want[1] == 4:
        want[1] = 0  # no tensor maps on this device
    assert got == want
    return g


@pytest.mark.parametrize('n', [(32, 32, 32), (48, 48, 64), (96, 96, 48), (160, 160, 96), (192, 192, 64), (256, 256, 160),
                               (320, 320, 48), (32, 32, 320)])
def test_partial_passes_equal_variant_0(n, monkeypatch):
    a = _grid(monkeypatch, n, '0,0,0')
    others = [_grid(monkeypatch, n, v) for v in ('2,3,8', '2,4,8')]
    for k in range(3):
        ref = a.solve_stress()
        p = a.get_positions()
        p[k] = np.mod(p[k] + np.array([1, -1, 1]), 2 * np.array(n))
        for g in others:
            assert np.array_equal(g.solve_stress(), ref), k
            g.set_positions(p)
        a.set_positions(p)
    st = a.step(500.0, 6)
    for g in others:
        sg = g.step(500.0, 6)
        assert sg['clock'] == st['clock']
        assert np.array_equal(g.get_positions(), a.get_positions())
        assert np.array_equal(g.interaction_energies(), a.interaction_energies())
    ref = a.solve_stress()
    for g in others:
        assert np.array_equal(g.solve_stress(), ref)
        g.close()
    a.close()
