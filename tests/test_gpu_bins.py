"""The column sums of 4^3 bins at their edges: bins of one particle, one warp,
just up to and past one and two chunks (736 particles, 384 with C), with every
cell of the leaf or a single one occupied, and (fused G2P2G) particles that have
left their leaf by less than a cell, by one cell and by several in each
direction since they were binned.  Against the oracle, with the particle tests'
tolerances."""
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


def _leaf(n, cells, seed, N=32):
    """n particles whose base nodes lie in the first `cells` cells of one 4^3 leaf."""
    rng = np.random.default_rng(seed)
    c = rng.integers(0, cells, size=n)
    base = np.stack([8 + c // 16, 12 + c // 4 % 4, 16 + c % 4], -1)
    x = ((base + rng.uniform(0.5, 1.5, size=(n, 3))) / N).astype(np.float32)
    v = rng.normal(0.0, 0.1, size=(n, 3)).astype(np.float32)
    return ParticleSpec(N, 4, n, np.zeros((3, 3)), np.zeros(3), x, v, note="one leaf")


SIZES = [(1, 64), (33, 64), (384, 64), (385, 1), (735, 64), (736, 1), (737, 64), (1473, 64)]


@pytest.mark.parametrize("n,cells", SIZES)
def test_one_bin_pic(n, cells):
    one_step_compare(_leaf(n, cells, n), 512)


@pytest.mark.parametrize("n,cells", SIZES)
def test_one_bin_apic(n, cells):
    C0 = np.random.default_rng(n + 1).normal(0.0, 1.0, size=(n, 9)).astype(np.float32)
    apic_step_compare(_leaf(n, cells, n), 512, C0)


@pytest.mark.parametrize("n,cells", SIZES)
@pytest.mark.parametrize("moved", [0.0, 0.9, 1.9, 7.0])
def test_one_bin_g2p2g(n, cells, moved):
    """Positions up to `moved` cells from where they were binned."""
    spec = _leaf(n, cells, n)
    rng = np.random.default_rng(n + 1)
    C0 = rng.normal(0.0, 1.0, size=(n, 9)).astype(np.float32)
    fused_step_check(spec, C0, 512, shift=rng.uniform(-moved, moved, size=(n, 3)) / spec.N)
