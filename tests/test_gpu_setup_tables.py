"""Self-term tables and stencils of okmc_set_defects at the edges of their kernels: box sizes of
the sums inside the pencil pass and of the line passes, batches of one to three shapes,
scan boxes as wide as the box allows, both zero-frequency modes."""
import numpy as np
import pytest

import __graft_entry__
import oracle as O
from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300.workload import FE_CUBIC, LOOP_100, LOOP_111, SIA_CLUSTER, make_defects

pytestmark = pytest.mark.gpu
H = 0.2855


@pytest.fixture(scope='module', autouse=True)
def _lib():
    __graft_entry__.build()
    ok.load()


def _defects(n, shapes):
    kinds, axes, radii, sizes = zip(*shapes)
    pos = np.array([[2 * i + 1, 4 * i + 1, 6 * i + 1] for i in range(len(shapes))]) % (2 * np.array(n)) | 1
    return make_defects(kinds, pos, axes, radii, sizes, [0.3] * len(shapes), [0] * len(shapes))


SHAPES = [(LOOP_111, 2, 0.9, 0), (SIA_CLUSTER, 0, 0.0, 1), (LOOP_100, 1, 0.7, 0), (SIA_CLUSTER, 0, 0.0, 9), (LOOP_111, 0, 0.5, 0)]


@pytest.mark.parametrize('k0', [ok.MEAN_STRESS_ZERO, ok.MEAN_STRAIN_ZERO])
@pytest.mark.parametrize('n,count,precision', [((32, 32, 32), 1, ok.FP32_FIELDS), ((48, 48, 96), 2, ok.FP32_FIELDS),
                                               ((32, 32, 320), 4, ok.FP32_FIELDS), ((96, 96, 32), 5, ok.FP32_FIELDS),
                                               ((32, 48, 64), 5, ok.FP32_FIELDS), ((16, 32, 48), 4, ok.FP64_FIELDS)])
def test_self_terms_match_oracle_over_shapes(n, count, precision, k0):
    """FP32 spectra: 5e-7 relative plus 1e-6 eV (the transform's rounding), FP64: 1e-9."""
    d = _defects(n, SHAPES[:count])
    g = ok.Grid(n, H, *FE_CUBIC, precision=precision, k0_mode=k0)
    g.set_defects(d)
    for again in range(2):  # a second set-up of the same grid starts from the first one's buffers
        W = g.self_terms()
        for i in range(count):
            Wo = O.self_term_table_fourier(d[i], n, H, O.stiffness_cubic(*FE_CUBIC), k0)
            tol = 1e-9 * max(1.0, np.abs(Wo).max()) if precision == ok.FP64_FIELDS else 5e-7 * np.abs(Wo).max() + 1e-6
            assert np.abs(W[i] - Wo).max() <= tol, (i, np.abs(W[i] - Wo).max())
        g.set_defects(d)
    eps = np.transpose(O.eigenstrain_field(d, n, H), (0, 3, 2, 1))
    assert np.abs(g.eigenstrain() - eps).max() < (1e-11 if precision == ok.FP64_FIELDS else 2e-7)
    g.close()


def test_stencils_of_extreme_shapes_bit_exact():
    """Radii at rounding edges of the slab and circle tests, the largest loop a 64^3 box takes
    and clusters on both sides of the one-voxel sphere and far above it."""
    n = (64, 64, 64)
    shapes = [(LOOP_111, 3, 8.0, 0), (LOOP_100, 2, 8.2, 0), (LOOP_100, 0, H, 0), (LOOP_111, 1, 0.5 * H, 0),
              (LOOP_111, 0, 2.0 * H * np.sqrt(3.0), 0)] + [(SIA_CLUSTER, 0, 0.0, s) for s in (1, 8, 9, 33, 1000, 60000)]
    d = _defects(n, shapes)
    g = ok.Grid(n, H, *FE_CUBIC)
    g.set_defects(d)
    for i in range(len(d)):
        for c in (0, 1):
            offs, cnt, alpha = g.stencil(i, c)
            o2, c2, a2 = O.stencil(d[i], c, H)
            assert np.array_equal(offs, o2) and np.array_equal(cnt, c2), (i, c)
            assert abs(alpha - a2) <= 1e-15 * a2
    g.close()
