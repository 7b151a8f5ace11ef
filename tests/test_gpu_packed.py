"""Packed (active-voxel) reads at the edges of the gather kernel's tiles: lists
that end inside, at and past a tile, leaves with no active voxel in the list,
values that start at every offset of a 16-byte group, both leaf sizes, pinned
and pageable destinations.  Bytes equal the whole-leaf read under the mask."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _grid(leaf_log2, n_leaves, seed):
    """n_leaves leaves of a 64^3 grid with random voxels, from one to all of a leaf's."""
    import torch
    import paper_2012_08141_gb300 as sg
    L, N = 1 << leaf_log2, 64
    R = N // L
    rng = np.random.default_rng(seed)
    b = np.sort(rng.choice(R ** 3, size=n_leaves, replace=False))
    xyz = []
    for q, leaf in enumerate(b):
        count = [1, L ** 3, int(rng.integers(1, L ** 3))][q % 3]
        l = rng.choice(L ** 3, size=count, replace=False)
        xyz.append(np.stack([leaf // (R * R) * L + l // (L * L), leaf // R % R * L + l // L % L, leaf % R * L + l % L], -1))
    g = sg.Grid(N, leaf_log2, 2, max_leaves=R ** 3)
    g.activate_coords(torch.from_numpy(np.concatenate(xyz).astype(np.int32)).cuda())
    g.list_gen()
    g.fill_hash(0, seed)
    return g


@pytest.mark.parametrize("leaf_log2,n_leaves", [(3, 1), (3, 7), (3, 8), (3, 9), (3, 512), (2, 1), (2, 63), (2, 64),
                                                (2, 65), (2, 3000)])
def test_packed_read_equals_masked_leaves(leaf_log2, n_leaves):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = _grid(leaf_log2, n_leaves, 11 * n_leaves + leaf_log2)
    _, masks = g.read_structure()
    on = np.unpackbits(masks.view(np.uint8), axis=1, bitorder="little").astype(bool)
    want = g.read_field(0)[on]
    assert (want != 0).any()
    got = g.read_field_active(0)
    assert np.array_equal(got, want)
    pinned = torch.full((want.size + 8,), -1.0).pin_memory().numpy()
    got = g.read_field_active(0, out=pinned)
    assert np.array_equal(got, want) and (pinned[want.size:] == -1.0).all()
    g.close()


def test_packed_read_capacity_and_versions():
    """The count is compared with the buffer's capacity before anything is
    written -- with offsets to compute and with kept ones, in place and staged
    -- and a structure change between two reads is followed."""
    import torch
    import paper_2012_08141_gb300 as sg
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    g = _grid(3, 9, 5)
    n = g.num_active()
    for out in (torch.full((n,), -1.0).pin_memory().numpy(), np.full(n, -1.0, np.float32)):
        for _ in range(2):  # offsets computed, then kept
            with pytest.raises(sg.SgError):
                g.read_field_active(0, out=out[:n - 1])
            assert (out == -1.0).all()
        assert np.array_equal(g.read_field_active(0, out=out), g.read_field(0)[_bits(g)])
        out[:] = -1.0
    g.activate_coords(torch.tensor([[1, 1, 1], [62, 62, 62], [33, 2, 9]], dtype=torch.int32, device="cuda"))
    g.fill_hash(0, 6)
    big = torch.full((n + 3,), -1.0).pin_memory().numpy()
    got = g.read_field_active(0, out=big)
    assert np.array_equal(got, g.read_field(0)[_bits(g)]) and got.size >= n
    g.deactivate_all()
    assert g.read_field_active(0, out=big).size == 0
    g.close()


def _bits(g):
    _, masks = g.read_structure()
    return np.unpackbits(masks.view(np.uint8), axis=1, bitorder="little").astype(bool)
