"""Task rounds of the j-run sweeps: lists with fewer tasks than resident warps,
about as many, and just past one and two rounds, so that the last round, which
is dealt to every CTA, is empty, partial and nearly full.  Fields are
bit-identical to the leaf-triple sweep's, alone and in a batch."""
import numpy as np
import pytest

from workload import band512

pytestmark = pytest.mark.gpu

# (domain edge, radius, half-width): 8^3 leaves from 56 to about 14,000
BANDS = [(64, 20.0, 4.0), (256, 100.0, 8.0), (256, 106.0, 8.0), (320, 140.0, 8.0), (320, 150.0, 4.0), (384, 150.0, 8.0)]


def _grid(spec, variant):
    import paper_2012_08141_gb300 as sg
    g = sg.Grid(spec.N, 3, 3, max_leaves=(spec.N // 8) ** 3, max_sums=1, scratch_mask=0b010)
    g.set_stencil_variant(variant)
    g.activate_shell(spec.lo2, spec.hi2, spec.lo_strict)
    g.list_gen()
    g.fill_hash(0, 17)
    return g


def _step(g):
    g.clear(1)
    g.diffuse7(0, 1, 0.1)
    g.box27(1, 2)
    g.swap(0, 2)
    g.reduce_sum(0, 0)
    g.flush()


@pytest.mark.parametrize("n,r,h", BANDS)
def test_last_round_alone(n, r, h):
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = []
    for variant in (sg.SG_VARIANT_SWEEP, sg.SG_VARIANT_SWEEP_JRUNS):
        g = _grid(band512(N=n, r=r, h=h), variant)
        for _ in range(3):
            _step(g)
        out.append((g.read_field(0), g.read_sums(1)[0]))
        g.close()
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
    assert abs(out[0][1] - out[1][1]) <= 1e-6 * abs(out[0][1])  # FP32 partials, another order


def test_last_round_in_a_batch():
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for some in (BANDS[:1], BANDS[:3], BANDS):
        grids = [_grid(band512(N=n, r=r, h=h), sg.SG_VARIANT_SWEEP_JRUNS) for n, r, h in some]
        alone = [_grid(band512(N=n, r=r, h=h), sg.SG_VARIANT_SWEEP) for n, r, h in some]
        b = sg.Batch(grids, 0, 1, 2, 0.1)
        for _ in range(2):
            b.step()
            for g in alone:
                _step(g)
        sums = b.read_sums()
        for q, (g, a) in enumerate(zip(grids, alone)):
            assert np.array_equal(g.read_field(0).view(np.uint32), a.read_field(0).view(np.uint32))
            assert abs(sums[q] - a.read_sums(1)[0]) <= 1e-6 * abs(sums[q])
        b.close()
        for g in grids + alone:
            g.close()
