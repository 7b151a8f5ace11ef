"""Advection with a leaf's cells staged in shared memory (fused runs over 8^3
leaves) against the unfused order, which looks every corner up: steps of less
than a cell, about one cell (some traces leave the staged block) and several, one
to three channels, at and away from the faces of the domain.  Bytes equal."""
import numpy as np
import pytest

from workload import tube, tube_fields

pytestmark = pytest.mark.gpu


def _run(channels, scale, opts, r_out):
    import oracle
    import paper_2012_08141_gb300 as sg
    spec = tube(N=64, L=8, r_out=r_out)
    g = sg.Grid(64, 3, 3 + 4 * channels, max_leaves=512, scratch_mask=sum(1 << (5 + 4 * c) for c in range(channels)))
    g.set_opts(opts)
    g.activate_tube(spec.lo2, spec.hi2)
    b, _ = g.read_structure()
    vel, ch = tube_fields(spec, oracle.leaf_coords(b, 64, 8).astype(np.float64))
    for a in range(3):
        g.write_field(a, vel[a])
    for c in range(channels):
        g.write_field(3 + 4 * c, ch[c])
    for _ in range(2):
        for c in range(channels):
            q, qh, qt, qn = 3 + 4 * c, 4 + 4 * c, 5 + 4 * c, 6 + 4 * c
            g.advect(qh, q, 0, scale / 64)
            g.advect(qt, qh, 0, -scale / 64)
            g.maccormack(qn, q, qh, qt, 0, scale / 64)
            g.swap(q, qn)
        g.flush()
    out = [g.read_field(f) for c in range(channels) for f in (3 + 4 * c, 4 + 4 * c)]
    packs = g.stats()["velocity_packs"]
    g.close()
    return out, packs


@pytest.mark.parametrize("channels", [1, 2, 3])
@pytest.mark.parametrize("scale", [0.4, 1.2, 5.0])
@pytest.mark.parametrize("r_out", [0.45, 0.75])
def test_block_equals_lookup(channels, scale, r_out):
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, packs = _run(channels, scale, sg.SG_OPT_ALL, r_out)
    b, none = _run(channels, scale, sg.SG_OPT_ALL & ~sg.SG_OPT_FUSE, r_out)
    assert packs > 0 and none == 0
    for x, y in zip(a, b):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
