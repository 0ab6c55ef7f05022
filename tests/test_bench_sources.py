"""bench.py reports a measured DRAM figure only while the sources of the kernel are those of the
capture: the list of a pass names every file that holds a form of it."""
import os
import re

import bench

CSRC = os.path.join(bench.ROOT, 'paper_2403_09158_gb300', 'csrc')
# the kernels a pass of a register-FFT grid can launch
FORMS = {'plane_fwd': r'k_plane_(fwd_n|tiles)\(', 'pencil_green': r'k_pencil_(fast|tma|reg|tma_reg)\(',
         'plane_inv': r'k_plane_(inv_n|inv_s|tiles)\(', 'energies': r'k_energy_chunks\('}


def test_kernel_sources_name_every_file_with_a_form_of_the_pass():
    for kernel, pattern in FORMS.items():
        listed = bench.KERNEL_SOURCES[kernel]
        assert all(os.path.exists(os.path.join(CSRC, f)) for f in listed), kernel
        holding = [f for f in sorted(os.listdir(CSRC))
                   if any(re.search(pattern, d) for d in re.findall(r'__global__[^;{]*\{', open(os.path.join(CSRC, f)).read()))]
        assert holding and set(holding) <= set(listed), (kernel, holding, listed)
        assert re.fullmatch(r'[0-9a-f]{16}', bench.kernel_sources_hash(kernel))
