"""A new grid's initial state over root sizes whose arrays are not whole 16-byte
words, in device memory that a grid with other contents has just given back:
no leaf, no active voxel, zero sums, and zeros beyond the allocated leaves."""
import numpy as np
import pytest

from test_gpu_check import CLEAN, _violations

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("R", [1, 2, 3, 5, 9])
def test_new_grid_in_used_memory(R, L):
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    N = R * L
    g = sg.Grid(N, {4: 2, 8: 3}[L], 3, max_leaves=R ** 3, max_sums=2)
    g.activate_shell(0, 16 * N * N, False)            # every voxel
    g.fill_hash(0, 3)
    g.fill_hash(1, 4)
    g.reduce_sum(0, 1)
    assert g.read_sums()[1] > 0
    g.close()
    g = sg.Grid(N, {4: 2, 8: 3}[L], 3, max_leaves=R ** 3, max_sums=2)
    assert not g.read_sums().any()
    g.list_gen()
    g.reduce_sum(0, 0)
    assert g.read_sums()[0] == 0.0
    g.activate_shell(0, 16 * N * N, False)
    g.clear(0)
    g.fill_hash(1, 4)
    g.box27(1, 2)                                      # reads the zero leaf beyond the domain
    g.reduce_sum(2, 0)
    first = g.read_sums()[0]
    assert _violations(g.check()) == CLEAN
    g.box27(1, 2)
    g.reduce_sum(2, 0)
    assert np.isfinite(first) and first > 0 and g.read_sums()[0] == first
    g.close()
