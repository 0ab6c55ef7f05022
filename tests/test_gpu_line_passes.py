"""The line passes (csrc/lines.cuh) against the CPU oracle: every line length of the grids
along each axis, alone in its box, in FP32 and FP64 fields."""
import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300.workload import FE_CUBIC, scaled_population

pytestmark = pytest.mark.gpu

EDGES = [16, 32, 48, 64, 80, 96, 128, 144, 160, 192, 240, 256, 288, 320, 384, 400, 432, 480, 512]
# relative L2: FP32 transforms of up to 2^27 points keep ~1e-6; FP64 ~1e-14
TOL = {ok.FP32_FIELDS: 1e-5, ok.FP64_FIELDS: 1e-10}


@pytest.fixture(scope='module', autouse=True)
def _lib():
    __graft_entry__.build()
    ok.load()


def _boxes(edge):
    for a in range(3):
        n = [16, 16, 16]
        n[a] = edge
        yield tuple(n)
        n[(a + 1) % 3] = 48
        yield tuple(n)


@pytest.mark.parametrize('precision', [ok.FP32_FIELDS, ok.FP64_FIELDS])
@pytest.mark.parametrize('edge', EDGES)
def test_every_line_length_along_every_axis(edge, precision):
    """One box per axis with the edge along it (and one with a second edge of 48): the
    stress against the oracle, then again after one defect has moved (with a second
    spectrum only its planes are transformed again)."""
    for n in _boxes(edge):
        w = scaled_population(n, 3, seed=sum(n), r111=(0.4, 0.9), r100=(0.4, 0.9))
        g = ok.Grid(n, w.voxel_nm, *FE_CUBIC, k0_mode=ok.MEAN_STRAIN_ZERO, precision=precision)
        g.set_defects(w.defects)
        for moved in (False, True):
            d = w.defects.copy()
            if moved:
                d['pos'][0] = np.mod(d['pos'][0] + [1, 1, -1], 2 * np.array(n))
                g.set_positions(d['pos'].astype(np.int32))
            sig = g.solve_stress()
            ref = O.solve_stress(O.eigenstrain_field(d, n, w.voxel_nm), O.stiffness_cubic(*FE_CUBIC), w.voxel_nm,
                                 O.MEAN_STRAIN_ZERO)
            ref = np.transpose(ref, (0, 3, 2, 1))
            rel = np.linalg.norm(sig.astype(np.float64) - ref) / np.linalg.norm(ref)
            assert rel <= TOL[precision], (n, moved, rel)
        g.close()


@pytest.mark.parametrize('precision', [ok.FP32_FIELDS, ok.FP64_FIELDS])
def test_second_spectrum_and_in_place_solves_agree(precision):
    """A memory bound keeps the grid to one spectrum (every plane transformed, in place); the
    stress, the energies and a trajectory are those of a grid with two, bit for bit."""
    n = (80, 48, 96)
    w = scaled_population(n, 6, seed=4, r111=(0.4, 1.0), r100=(0.4, 1.0))
    free = ok.Grid(n, w.voxel_nm, *FE_CUBIC, precision=precision, seed=2)
    tight = ok.Grid(n, w.voxel_nm, *FE_CUBIC, precision=precision, seed=2, hbm_budget=1 << 30)
    assert tight.device_bytes() < free.device_bytes()
    for g in (free, tight):
        g.set_defects(w.defects)
        g.step(400.0, 6)
    assert np.array_equal(free.get_positions(), tight.get_positions())
    assert np.array_equal(free.solve_stress(), tight.solve_stress())
    assert np.array_equal(free.candidate_energies()[0], tight.candidate_energies()[0])
    free.close()
    tight.close()


@pytest.mark.parametrize('n,precision', [((64, 64, 64), ok.FP32_FIELDS), ((48, 32, 80), ok.FP32_FIELDS),
                                         ((64, 64, 64), ok.FP64_FIELDS)])
def test_a_solve_is_timed_under_the_same_three_names_on_every_grid(n, precision):
    w = scaled_population(n, 12, seed=6, r111=(0.4, 0.9), r100=(0.4, 0.9))
    g = ok.Grid(n, w.voxel_nm, *FE_CUBIC, precision=precision)
    g.set_defects(w.defects)
    g.set_profiling(True)
    g.solve_stress(copy=False)
    assert {k: v[1] for k, v in g.kernel_times().items()} == {'plane_fwd': 1, 'pencil_green': 1, 'plane_inv': 1}
    g.reset_kernel_times()
    g.shift_energies(0, np.zeros((2, 3)))
    assert set(g.kernel_times()) == {'shift_eps_fwd', 'shift_eps_pencil', 'shift_fields', 'shift_w_fwd', 'shift_w_pencil',
                                     'shift_energies'}
    g.close()


@pytest.mark.parametrize('n,precision,width', [((16, 16, 16), ok.FP32_FIELDS, 8), ((48, 32, 240), ok.FP32_FIELDS, 8),
                                               ((16, 16, 256), ok.FP32_FIELDS, 8), ((16, 16, 288), ok.FP32_FIELDS, 4),
                                               ((16, 16, 512), ok.FP32_FIELDS, 4), ((64, 64, 64), ok.FP64_FIELDS, 4)])
def test_launch_shape_is_that_of_the_line_passes(n, precision, width):
    """No clusters; one CTA of the pencil pass per kx and `width` ky (as lines.cuh lays out
    its tiles: eight FP32 columns while two tiles fit an SM)."""
    w = scaled_population(n, 1, seed=6, r111=(0.4, 0.5), r100=(0.4, 0.5))
    g = ok.Grid(n, w.voxel_nm, *FE_CUBIC, precision=precision)
    assert list(g.launch_shape()) == [1, (n[0] // 2 + 1) * n[1] // width, 1]
    g.close()
