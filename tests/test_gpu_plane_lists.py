"""Few defects in a tall box: the kinetic step reads and writes only the z-planes of the
defects' scan boxes (okmc_step, batches); everything else asks for the whole field."""
import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300.workload import FE_CUBIC, LOOP_111, ONE_D, SIA_CLUSTER, THREE_D, make_defects

pytestmark = pytest.mark.gpu
H = 0.2855
SEED = 311


@pytest.fixture(scope='module', autouse=True)
def _lib():
    __graft_entry__.build()
    ok.load()


def _defects(n, nd=2):
    """A loop across the periodic z face, a single atom elsewhere (and a second loop beside it)."""
    z = np.array([2 * n[2] - 2, n[2] // 2 * 2 + 1, n[2] // 2 * 2 + 14])
    pos = np.stack([np.array([n[0], n[0] // 2 * 2 + 1, 12]), np.array([n[1], 9, 20]), z], axis=1)
    pos[1] |= 1
    return make_defects([LOOP_111, SIA_CLUSTER, LOOP_111][:nd], pos[:nd], [0, 1, 2][:nd], [0.8, 0.0, 0.6][:nd], [0, 1, 0][:nd],
                        [0.1, 0.1, 0.1][:nd], [ONE_D, THREE_D, ONE_D][:nd])


def _line(n):
    return [(np.array([[0.2, 0.3, 0.6], [0.2, 0.3 + n[1] * H, 0.6]]), 0.5 * H * np.array([1.0, -1.0, 1.0]), False)]


@pytest.mark.parametrize('lines', [False, True])
@pytest.mark.parametrize('n,precision', [((64, 64, 64), ok.FP32_FIELDS), ((128, 128, 160), ok.FP32_FIELDS),
                                         ((48, 32, 80), ok.FP32_FIELDS), ((32, 48, 64), ok.FP64_FIELDS),
                                         ((32, 32, 512), ok.FP32_FIELDS), ((160, 160, 96), ok.FP32_FIELDS)])
def test_steps_take_the_decisions_of_the_whole_field(n, precision, lines):
    """Energies from whole-field solves and the oracle's event against okmc_step, event by
    event; the clock follows to 1e-12, so the step's energies are those of the whole field
    (an energy off by 1e-9 eV would move it by 1e-8)."""
    g = ok.Grid(n, H, *FE_CUBIC, precision=precision, seed=SEED)
    g.set_defects(_defects(n, 3))
    if lines:
        g.set_dislocations(_line(n))
    assert 1 <= g.nd <= 3
    d, clock = _defects(n, 3), 0.0
    for step in range(8):
        E, Ec = g.interaction_energies(), g.candidate_energies()[0]
        _, _, dt, _ = O.residence_step(d, E, Ec, 500.0, SEED, step, n)
        st = g.step(500.0, 1)
        assert np.array_equal(g.get_positions(), d['pos']), step
        clock += dt
        assert abs(st['clock'] - clock) <= 1e-12 * clock
    # a run of steps without whole-field solves between them, then the whole field again
    g.step(500.0, 5)
    g.step(500.0, 5, mode=ok.FIXED_DT)
    fresh = ok.Grid(n, H, *FE_CUBIC, precision=precision, seed=SEED)
    fresh.set_defects(g.get_defects())
    if lines:
        fresh.set_dislocations(_line(n))
    assert np.array_equal(g.solve_stress(), fresh.solve_stress())
    assert np.array_equal(g.candidate_energies()[0], fresh.candidate_energies()[0])
    g.close()
    fresh.close()


@pytest.mark.parametrize('mode', [ok.BATCH_KERNELS, ok.BATCH_GRAPHS])
def test_batches_of_few_and_many_defects_equal_alone(mode):
    """Replicas of one edge with and without plane lists, and one with dislocation lines."""
    boxes = [((64, 64, 64), 2, False), ((64, 64, 64), 3, True), ((128, 128, 64), 2, False)]
    dense = make_defects([SIA_CLUSTER] * 12, np.array([[10 * k + 3, 5, 9 * k + 1 | 1] for k in range(12)]) | 1, [0] * 12,
                         [0.0] * 12, [2] * 12, [0.2] * 12, [ONE_D] * 12)

    def make():
        out = []
        for n, nd, lines in boxes:
            g = ok.Grid(n, H, *FE_CUBIC, seed=SEED)
            g.set_defects(_defects(n, nd))
            if lines:
                g.set_dislocations(_line(n))
            out.append(g)
        g = ok.Grid((64, 64, 64), H, *FE_CUBIC, seed=SEED)
        g.set_defects(dense)
        return out + [g]
    alone, grids = make(), make()
    stats = [g.step(450.0, 7) for g in alone]
    b = ok.Batch(grids, mode=mode)
    b.step([450.0] * 4, 3)
    got = b.step([450.0] * 4, 4)
    assert b.mode() == mode
    for g, a, s, t in zip(grids, alone, got, stats):
        assert np.array_equal(g.get_positions(), a.get_positions())
        assert s['clock'] == t['clock'] and s['events'] == t['events']
        assert np.array_equal(g.solve_stress(), a.solve_stress())
    b.close()
    for g in grids + alone:
        g.close()


def test_fast_passes_keep_the_tuned_pencil_form_with_few_defects(monkeypatch):
    """The register-FFT passes take a list only in the inverse plane pass of a step: the pencil
    pass runs in the pinned variant (bulk copies that never complete time out, which no other
    form can), and a whole-field solve launches no list."""
    n = (256, 256, 192)  # above the size from which line passes list the planes of whole-field solves
    monkeypatch.setenv('OKMC_VARIANTS', '0,0,0')
    g = ok.Grid(n, H, *FE_CUBIC, seed=SEED)
    g.set_defects(_defects(n, 3))
    if not (g.variants()[1][1] >> 4) & 1:
        pytest.skip('no tensor maps on this device')
    ref = g.solve_stress()
    E = g.interaction_energies()
    g.set_variant(1, 4)
    g.set_profiling(True)
    g.reset_kernel_times()
    assert np.array_equal(g.solve_stress(), ref)
    assert 'plane_list' not in g.kernel_times()
    g.set_profiling(False)
    assert np.array_equal(g.interaction_energies(), E)
    monkeypatch.setenv('OKMC_TMA_EXTRA_TX', '16')
    for call in (lambda: g.solve_stress(), lambda: g.step(500.0, 1)):
        g.set_variant(1, 4)
        with pytest.raises(ok.OkmcError) as ei:
            call()
        assert ei.value.code == ok.OKMC_ETIMEOUT
        g.set_defects(_defects(n, 3))
    g.close()


def test_a_failed_set_up_leaves_the_field_that_the_solve_reads():
    """okmc_set_defects runs out of its budget before it has touched the field: a solve then gives
    the stress of the field as it stands, not of its part in the new defects' planes."""
    n = (240, 240, 240)  # line passes, whole-field solves by plane lists
    loop = make_defects([LOOP_111], np.array([[240, 240, 240]]), [0], [60 * H], [0], [0.1], [ONE_D])
    other = ok.Grid(n, H, *FE_CUBIC, hbm_budget=1 << 33)
    other.set_defects(_defects(n, 2))
    ref = other.solve_stress()
    g = ok.Grid(n, H, *FE_CUBIC, hbm_budget=other.device_bytes() + (100 << 10))
    other.close()
    g.set_defects(_defects(n, 2))
    with pytest.raises(ok.OkmcError) as ei:
        g.set_defects(loop)  # its stencils alone take 0.3 MB
    assert ei.value.code == ok.OKMC_ENOMEM
    assert np.array_equal(g.solve_stress(), ref)
    g.close()


@pytest.mark.parametrize('budget', [0, 1 << 36])
@pytest.mark.parametrize('n,precision', [((240, 240, 240), ok.FP32_FIELDS), ((160, 160, 480), ok.FP32_FIELDS),
                                         ((256, 144, 320), ok.FP64_FIELDS)])
def test_whole_field_solves_by_lists_equal_those_over_every_plane(n, precision, budget):
    """Line passes of few defects in a large box, with a second spectrum and in place: the same
    solves on a grid with a dislocation line far below the eigenstrain's quantum, which adds
    nothing to the field and leaves no plane out.  A defect jumps to planes never used before,
    so that the planes it has left are stale and outside the list."""
    grids = []
    for line in (False, True):
        g = ok.Grid(n, H, *FE_CUBIC, precision=precision, seed=SEED, hbm_budget=budget)
        g.set_defects(_defects(n, 3))
        if line:
            before = g.eigenstrain()
            g.set_dislocations([(p, 1e-30 * b, c) for p, b, c in _line(n)])
            assert np.array_equal(g.eigenstrain(), before)
        grids.append(g)
    a, b = grids
    p = a.get_positions()
    for k in range(4):
        a.set_profiling(True)
        a.reset_kernel_times()
        ref = b.solve_stress()
        assert np.array_equal(a.solve_stress(), ref), k
        assert 'plane_list' in a.kernel_times()
        a.set_profiling(False)
        assert np.array_equal(a.interaction_energies(), b.interaction_energies())
        p[k % 3, 2] = (p[k % 3, 2] + 2 * (n[2] // 3)) % (2 * n[2])
        for g in grids:
            g.set_positions(p)
            if k == 2:
                g.step(500.0, 3)
        assert np.array_equal(a.get_positions(), b.get_positions())
        p = a.get_positions()
    for g in grids:
        g.close()
