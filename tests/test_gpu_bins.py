"""The column sums of 4^3 bins (a 4^3 leaf, an octant of an 8^3 one) at their
edges: bins of one particle, one warp, just up to and past one and two chunks
(736 particles, 384 with C), with every cell of the bin or a single one
occupied, and (fused G2P2G) particles that have left their bin by less than a
cell, by one cell and by several in each direction since they were binned.
Against the oracle, with the particle tests' tolerances.  And the binning itself
over root sizes at the edges of its tiles of 1,024 bins and on both sides of the
line from which the tile sums are scanned by a kernel of their own."""
import numpy as np
import pytest

from test_gpu_g2p2g import fused_step_check
from test_gpu_particles import apic_step_compare, one_step_compare
from workload import ParticleSpec

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


def _leaf(n, cells, seed, L, N=32):
    """n particles whose base nodes lie in the first `cells` cells of one 4^3 bin."""
    rng = np.random.default_rng(seed)
    c = rng.integers(0, cells, size=n)
    base = np.stack([8 + c // 16, 12 + c // 4 % 4, 16 + c % 4], -1)
    x = ((base + rng.uniform(0.5, 1.5, size=(n, 3))) / N).astype(np.float32)
    v = rng.normal(0.0, 0.1, size=(n, 3)).astype(np.float32)
    return ParticleSpec(N, L, n, np.zeros((3, 3)), np.zeros(3), x, v, note="one leaf")


SIZES = [(1, 64), (33, 64), (384, 64), (385, 1), (735, 64), (736, 1), (737, 64), (1473, 64)]


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,cells", SIZES)
def test_one_bin_pic(n, cells, L):
    one_step_compare(_leaf(n, cells, n, L), 512)


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,cells", SIZES)
def test_one_bin_apic(n, cells, L):
    C0 = np.random.default_rng(n + 1).normal(0.0, 1.0, size=(n, 9)).astype(np.float32)
    apic_step_compare(_leaf(n, cells, n, L), 512, C0)


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,cells", SIZES)
@pytest.mark.parametrize("moved", [0.0, 0.9, 1.9, 7.0])
def test_one_bin_g2p2g(n, cells, L, moved):
    """Positions up to `moved` cells from where they were binned."""
    spec = _leaf(n, cells, n, L)
    rng = np.random.default_rng(n + 1)
    C0 = rng.normal(0.0, 1.0, size=(n, 9)).astype(np.float32)
    fused_step_check(spec, C0, 512, shift=rng.uniform(-moved, moved, size=(n, 3)) / spec.N)


@pytest.mark.parametrize("N,L", [(8, 4), (40, 4), (44, 4), (1020, 4), (1024, 4), (8, 8), (40, 8), (48, 8), (1016, 8), (1024, 8)])
def test_binning_order_and_reach(N, L):
    """Particles all over the domain and outside of it, binned afresh and from
    the last order: sorted, they are the same particles in ascending leaves, the
    outside ones last; and every node that a stencil reaches was allocated (the
    grid holds the mass of the inside ones: at most 64 + 27 FP32 roundings on
    each node's sum, 91 * 2^-24 < 1e-5 of it)."""
    import torch
    import paper_2012_08141_gb300 as sg
    n, R = 3000, N // L
    rng = np.random.default_rng(N)
    cells = rng.uniform(1.0, N - 2.0, size=(n, 3))       # stencils inside the domain
    cells[:8] = [[1.0 + (N - 3.0) * (q >> a & 1) for a in range(3)] for q in range(8)]
    out = np.arange(n) % 100 == 99
    cells[out, n % 3] = -5.0
    x = torch.from_numpy((cells / N).astype(np.float32)).cuda()
    v = torch.zeros(n, 3, device="cuda")
    ids = torch.arange(n, dtype=torch.int64, device="cuda")
    g = sg.Grid(N, {4: 2, 8: 3}[L], 4, max_leaves=min(R ** 3, 8 * n), max_sums=1)
    for _ in range(3):
        g.deactivate_all()
        g.p2g(x, v, 1.0, 0, 1)
        g.reduce_sum(0, 0)
        assert abs(g.read_sums()[0] - (n - out.sum())) <= 1e-5 * n
        g.sort_particles(x, v, ids=ids)
        g.sync()
        at = ids.cpu().numpy()
        assert np.array_equal(np.sort(at), np.arange(n))
        X = x.cpu().numpy() * np.float32(N)
        assert np.array_equal(X, (cells / N).astype(np.float32)[at] * np.float32(N))
        assert out[at][n - out.sum():].all()
        b = np.floor(X[:n - out.sum()] - np.float32(0.5)).astype(np.int64) // L
        assert np.all(np.diff((b[:, 0] * R + b[:, 1]) * R + b[:, 2]) >= 0)
    g.close()
