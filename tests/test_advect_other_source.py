"""A backward advection is fused with the MacCormack correction that reads its
output only if it advects the correction's q^ back: a correction whose q~ comes
from another field takes that field's value."""
import numpy as np
import pytest

import paper_2012_08141_gb300 as sg
from workload import tube


def _queue(g, other):
    g.advect(4, 3, 0, 1e-2)
    g.advect(5, 7 if other else 4, 0, -1e-2)
    g.maccormack(6, 3, 4, 5, 0, 1e-2)
    g.flush()


@pytest.mark.parametrize("other", [False, True])
def test_launches(other):
    """One velocity packing, the forward launch and the fused backward one; with
    another source both advections are traced by launches without correction."""
    g = sg.Grid(64, 3, 8, max_leaves=1024, scratch_mask=1 << 5, dry_run=True)
    g.activate_tube(1000, 3000)
    g.list_gen()
    g.flush()
    before = g.stats()["launches"]
    _queue(g, other)
    assert g.stats()["launches"] - before == (4 if other else 3)


@pytest.mark.gpu
@pytest.mark.parametrize("L", [4, 8])
def test_bytes_equal_the_unfused_order(L):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    spec = tube(N=64, L=L, r_out=0.45)
    outs = []
    for opts in (sg.SG_OPT_ALL, sg.SG_OPT_ALL & ~sg.SG_OPT_FUSE):
        g = sg.Grid(64, {4: 2, 8: 3}[L], 8, max_leaves=4096, scratch_mask=1 << 5)
        g.set_opts(opts)
        g.activate_tube(spec.lo2, spec.hi2)
        b, masks = g.read_structure()
        on = np.unpackbits(masks.view(np.uint8), axis=1, bitorder="little").astype(bool)[:, :L ** 3]
        rng = np.random.default_rng(5)
        for f in (0, 1, 2, 3, 7):
            g.write_field(f, np.where(on, rng.normal(0.0, 0.6, size=on.shape), 0.0).astype(np.float32))
        _queue(g, True)
        outs.append([g.read_field(f) for f in (4, 6)])
        g.close()
    for x, y in zip(*outs):
        assert np.array_equal(x.view(np.uint32), y.view(np.uint32))
