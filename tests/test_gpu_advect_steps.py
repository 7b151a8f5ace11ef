"""The two kernels of a fused advection over a list long enough for the choice
between them, which the device makes by the largest packed velocity component:
steps just below, at and above a cell, one fast voxel in a slow field, runs of
different lengths in turn on one grid (a packing's largest component must not be
taken for the next one's), and one to three channels at and away from the faces
of the domain.  Bytes equal to the unfused order, which packs nothing."""
import numpy as np
import pytest

from workload import tube, tube_fields

pytestmark = pytest.mark.gpu

N = 128  # 1,632 leaves and more


def _run(opts, speeds, one_fast):
    import paper_2012_08141_gb300 as sg
    spec = tube(N=N, L=8, r_out=0.45)
    g = sg.Grid(N, 3, 7, max_leaves=4096, scratch_mask=1 << 5)
    g.set_opts(opts)
    g.activate_tube(spec.lo2, spec.hi2)
    b, masks = g.read_structure()
    on = np.unpackbits(masks.view(np.uint8), axis=1, bitorder="little").astype(bool)
    rng = np.random.default_rng(4)
    q = rng.normal(0.0, 1.0, size=on.shape).astype(np.float32)
    out = []
    for speed in speeds:
        for a, s in enumerate((1.0, -0.4, 0.7)):
            vel = np.where(on, np.float32(s * (0.3 if one_fast else speed)), np.float32(0.0)).astype(np.float32)
            if one_fast:
                vel[len(b) // 2, np.flatnonzero(on[len(b) // 2])[0]] = s * speed
            g.write_field(a, vel)
        g.write_field(3, q)
        g.advect(4, 3, 0, 1.0 / N)
        g.advect(5, 4, 0, -1.0 / N)
        g.maccormack(6, 3, 4, 5, 0, 1.0 / N)
        g.flush()
        out += [g.read_field(4), g.read_field(6)]
    packs = g.stats()["velocity_packs"]
    g.close()
    return out, packs


@pytest.mark.parametrize("one_fast", [False, True])
@pytest.mark.parametrize("speeds", [[0.999999], [1.0], [1.000001], [3.0, 0.5, 0.5, 3.0, 0.5], [0.5, 2.0, 0.5, 0.5, 2.0, 2.0]])
def test_either_kernel_equals_lookup(speeds, one_fast):
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    a, packs = _run(sg.SG_OPT_ALL, speeds, one_fast)
    b, none = _run(sg.SG_OPT_ALL & ~sg.SG_OPT_FUSE, speeds, one_fast)
    assert packs == len(speeds) and none == 0
    for x, y in zip(a, b):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))


@pytest.mark.parametrize("channels", [1, 2, 3])
@pytest.mark.parametrize("scale", [0.9, 1.2, 5.0])
@pytest.mark.parametrize("r_out", [0.45, 0.75])
def test_staged_block_equals_lookup(channels, scale, r_out):
    import oracle
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spec = tube(N=N, L=8, r_out=r_out)
    outs = []
    for opts in (sg.SG_OPT_ALL, sg.SG_OPT_ALL & ~sg.SG_OPT_FUSE):
        g = sg.Grid(N, 3, 3 + 4 * channels, max_leaves=4096, scratch_mask=sum(1 << (5 + 4 * c) for c in range(channels)))
        g.set_opts(opts)
        g.activate_tube(spec.lo2, spec.hi2)
        b, _ = g.read_structure()
        assert len(b) >= 1024
        vel, ch = tube_fields(spec, oracle.leaf_coords(b, N, 8).astype(np.float64))
        for a in range(3):
            g.write_field(a, vel[a])
        for c in range(channels):
            g.write_field(3 + 4 * c, ch[c])
        for c in range(channels):
            q, qh, qt, qn = 3 + 4 * c, 4 + 4 * c, 5 + 4 * c, 6 + 4 * c
            g.advect(qh, q, 0, scale / N)
            g.advect(qt, qh, 0, -scale / N)
            g.maccormack(qn, q, qh, qt, 0, scale / N)
        outs.append([g.read_field(f + 4 * c) for c in range(channels) for f in (4, 6)])
        g.close()
    for x, y in zip(*outs):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
