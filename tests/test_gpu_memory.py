"""Device memory of a handle: what okmc_estimate_field_bytes says, and the line passes' second
spectrum, which gives way when an allocation would otherwise fail."""
import threading

import numpy as np
import pytest

import __graft_entry__
from paper_2403_09158_gb300 import okmc as ok
from paper_2403_09158_gb300.workload import FE_CUBIC, scaled_population

pytestmark = pytest.mark.gpu
H = 0.2855


@pytest.fixture(scope='module', autouse=True)
def _lib():
    __graft_entry__.build()
    ok.load()


@pytest.mark.parametrize('budget', [0, 1 << 33])
@pytest.mark.parametrize('n,precision', [((64, 64, 64), ok.FP32_FIELDS), ((96, 64, 160), ok.FP32_FIELDS),
                                         ((16, 16, 16), ok.FP32_FIELDS), ((48, 48, 48), ok.FP64_FIELDS),
                                         ((32, 80, 16), ok.FP64_FIELDS)])
def test_estimate_is_what_a_grid_allocates(n, precision, budget):
    g = ok.Grid(n, H, *FE_CUBIC, precision=precision, hbm_budget=budget)
    assert g.device_bytes() == ok.estimate_field_bytes(n, H, *FE_CUBIC, precision=precision, hbm_budget=budget)
    g.close()


N = (128, 128, 128)
NEED = 6 * 128 ** 3 * 8  # one FP64 field: what okmc_eigenstrain allocates for its copy


def _grid(w, **kw):
    g = ok.Grid(N, w.voxel_nm, *FE_CUBIC, precision=ok.FP64_FIELDS, seed=5, **kw)
    g.set_defects(w.defects)
    return g


def _script(g):
    """Every kernel that the tests below launch; ends on the stress of the state it leaves."""
    g.step(400.0, 3)
    g.eigenstrain()
    return g.solve_stress()


class _Full:
    """All device memory but about `leave` bytes, held by another allocator of the process."""

    def __init__(self, leave):
        torch = pytest.importorskip('torch')
        self.torch, self.hold = torch, []
        torch.cuda.empty_cache()
        for chunk in (1 << 32, 1 << 28, 1 << 24):
            while torch.cuda.mem_get_info()[0] > leave + chunk:
                self.hold.append(torch.empty(chunk, dtype=torch.uint8, device='cuda'))

    def close(self):
        self.hold.clear()
        self.torch.cuda.empty_cache()


def test_a_failing_allocation_takes_another_grids_second_spectrum():
    """Grid a has a second spectrum; grid b, without one, has no room left for a temporary
    field until a gives way.  Both go on with the same results, a under a graph captured
    before as well."""
    w = scaled_population(N, 6, seed=3, r111=(0.4, 1.0), r100=(0.4, 1.0))
    a, ref = _grid(w), _grid(w, hbm_budget=1 << 40)
    assert np.array_equal(_script(a), _script(ref))
    b = _grid(w, hbm_budget=1 << 40)
    assert np.array_equal(_script(b), ref.solve_stress())
    before, eps = a.device_bytes(), b.eigenstrain()
    assert b.device_bytes() < before
    full = _Full(NEED // 2)
    try:
        assert np.array_equal(b.eigenstrain(), eps)
        assert a.device_bytes() == before - 6 * 128 * 65 * 128 * 16
        st, want = a.step(400.0, 3), ref.step(400.0, 3)
        assert st['clock'] == want['clock']
        assert np.array_equal(a.solve_stress(), ref.solve_stress())
    finally:
        full.close()
    for g in (a, b, ref):
        g.close()


def test_a_grid_in_use_by_another_thread_gives_way_between_its_calls():
    """One thread steps grid a while this one's allocations take a's second spectrum (they wait
    for a call to end): a's trajectory is the one it follows alone."""
    w = scaled_population(N, 6, seed=3, r111=(0.4, 1.0), r100=(0.4, 1.0))
    a, ref, b = _grid(w), _grid(w), _grid(w, hbm_budget=1 << 40)
    for g in (a, ref, b):
        _script(g)
    before = a.device_bytes()
    ref.step(400.0, 40)
    want, stress = ref.stats(), ref.solve_stress()
    ref.close()
    full = _Full(NEED // 2)
    failed = []

    def work():
        try:
            for _ in range(40):
                a.step(400.0, 1)
        except ok.OkmcError as e:
            failed.append(e)
    t = threading.Thread(target=work)
    try:
        t.start()
        took = 0
        for _ in range(200):
            try:
                b.eigenstrain()
                took += 1
            except ok.OkmcError as e:  # a was inside a call for a second
                assert e.code == ok.OKMC_ENOMEM
            if not t.is_alive() and took:
                break
    finally:
        t.join()
        full.close()
    assert not failed and took
    assert a.device_bytes() < before
    assert a.stats()['clock'] == want['clock'] and np.array_equal(a.solve_stress(), stress)
    a.close()
    b.close()


def test_a_callers_capture_keeps_the_second_spectrum():
    """Work that a caller captures from the grid's stream is replayed with the addresses it
    had: the spectrum then stays, and the failing allocation fails."""
    torch = pytest.importorskip('torch')
    w = scaled_population(N, 6, seed=3, r111=(0.4, 1.0), r100=(0.4, 1.0))
    st = torch.cuda.Stream()
    a = ok.Grid(N, w.voxel_nm, *FE_CUBIC, precision=ok.FP64_FIELDS, seed=5, stream=st.cuda_stream)
    a.set_defects(w.defects)
    b = _grid(w, hbm_budget=1 << 40)
    E = torch.zeros(a.nd, dtype=torch.float64, device='cuda')
    p = torch.tensor(a.get_positions(), device='cuda')
    a.interaction_energies(E)
    b.eigenstrain()
    ref = b.interaction_energies()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        graph.capture_begin(capture_error_mode='thread_local')
        a.set_positions(p)
        a.interaction_energies(E)
        graph.capture_end()
    before = a.device_bytes()
    full = _Full(NEED // 2)
    try:
        with pytest.raises(ok.OkmcError) as ei:
            b.eigenstrain()
        assert ei.value.code == ok.OKMC_ENOMEM and a.device_bytes() == before
        E.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(E.cpu().numpy(), ref)
    finally:
        full.close()
    del graph
    a.close()
    b.close()
