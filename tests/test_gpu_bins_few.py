"""Particle bins far emptier and far fuller than a chunk, and fused G2P2G of
particles that have moved since they were binned, against the oracle with the
particle tests' tolerances: more bins of up to 32 particles than a launch gives
to whole CTAs (one a bin, a dozen, and a mix with fuller ones), a few crowded
bins that several CTAs share, and the number of moved particles from which a
chunk is summed over the cells around the bin's own."""
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


def _box(n, lo, hi, L, seed, N=128):
    rng = np.random.default_rng(seed)
    x = (rng.uniform(lo, hi, size=(n, 3)) / N).astype(np.float32)
    v = rng.normal(0.0, 0.1, size=(n, 3)).astype(np.float32)
    return ParticleSpec(N, L, n, np.zeros((3, 3)), np.zeros(3), x, v, note="box")


def _affine(n, seed):
    return np.random.default_rng(seed).normal(0.0, 1.0, size=(n, 9)).astype(np.float32)


# whole domain and beyond: a particle a bin; about 15 and 24 a bin; 3 crowded bins
BOXES = [(4000, -1.0, 128.5), (60000, 30.0, 94.0), (100000, 30.0, 94.0), (20000, 40.5, 45.5)]


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,lo,hi", BOXES)
def test_pic(n, lo, hi, L):
    one_step_compare(_box(n, lo, hi, L, n), (128 // L) ** 3, interior=False)


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,lo,hi", BOXES)
def test_apic(n, lo, hi, L):
    apic_step_compare(_box(n, lo, hi, L, n), (128 // L) ** 3, _affine(n, 1))


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,lo,hi", BOXES)
@pytest.mark.parametrize("moved", [0.0, 0.9, 7.0])
def test_g2p2g(n, lo, hi, L, moved):
    rng = np.random.default_rng(n + 1)
    spec = _box(n, lo, hi, L, n)
    fused_step_check(spec, _affine(n, 2), (128 // L) ** 3, shift=rng.uniform(-moved, moved, size=(n, 3)) / spec.N)


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,moved", [(200, 0), (200, 1), (200, 24), (200, 25), (200, 200), (1473, 30), (1473, 1473)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_moved_into_the_cells_around(n, moved, axis, L, N=32):
    """The first `moved` particles of one bin go one cell up (into the cells
    around the bin's own) or, every fifth, two (further out)."""
    rng = np.random.default_rng(n + moved)
    base = np.array([8, 12, 16]) + rng.integers(0, 4, size=(n, 3))
    base[:, axis] = (8, 12, 16)[axis] + 3
    x = ((base + rng.uniform(0.5, 1.5, size=(n, 3))) / N).astype(np.float32)
    v = rng.normal(0.0, 0.01, size=(n, 3)).astype(np.float32)
    shift = np.zeros((n, 3))
    shift[:moved, axis] = np.where(np.arange(moved) % 5 == 4, 2.0, 1.0) / N
    fused_step_check(ParticleSpec(N, L, n, np.zeros((3, 3)), np.zeros(3), x, v, note="one bin"), _affine(n, 3), 512, shift=shift)
