"""A read that returns a device error has written nothing: packed fields
(offsets to compute and kept, in place and staged) and reduction results, few
and more than come with the control block."""
import ctypes

import numpy as np
import pytest

from workload import band_bounds

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


def _grid(sg, leaves=512, sums=8):
    g = sg.Grid(64, 3, 2, max_leaves=leaves, max_sums=sums)
    g.activate_shell(*band_bounds(10.0, 20.0), False)
    g.fill_hash(0, 1)
    return g


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("kept", [False, True])
def test_failed_packed_read_writes_nothing(pinned, kept):
    import torch
    import paper_2012_08141_gb300 as sg
    g = _grid(sg)
    n = g.num_active()          # the list is current and its length known
    want = g.read_field_active(0).copy() if kept else None
    out = torch.full((n,), -1.0)
    out = (out.pin_memory() if pinned else out).numpy()
    g.debug_wait_test()         # a bounded wait that gives up
    with pytest.raises(sg.SgError) as e:
        g.read_field_active(0, out=out)
    assert e.value.code == sg.SG_ERR_TIMEOUT
    assert (out == -1.0).all()
    got = g.read_field_active(0, out=out)   # the error was reported once
    assert got.size == n and (got != -1.0).all() and (want is None or np.array_equal(got, want))
    g.close()


@pytest.mark.parametrize("slots", [1, 8, 5000])
@pytest.mark.parametrize("failure", ["wait", "pool"])
def test_failed_sum_read_writes_nothing(slots, failure):
    import paper_2012_08141_gb300 as sg
    g = _grid(sg, sums=slots)
    g.reduce_sum(0, slots - 1)
    want = g.read_sums()
    assert want[slots - 1] > 0
    out = np.full(slots, -1.0)
    if failure == "wait":
        g.debug_wait_test()
    else:
        small = sg.Grid(64, 3, 2, max_leaves=4, max_sums=slots)
        small.activate_shell(*band_bounds(10.0, 20.0), False)
        g.close()
        g = small
    rc = g.lib.sg_read_sums(g.h, ctypes.c_void_p(out.ctypes.data), slots)
    assert rc == (sg.SG_ERR_TIMEOUT if failure == "wait" else sg.SG_ERR_POOL_EXHAUSTED)
    assert (out == -1.0).all()
    if failure == "wait":
        assert np.array_equal(g.read_sums(), want)
    g.close()
