"""Several fused G2P2G launches over one binning, from positions set before each:
the second form of the kernel (sums over the cells around a bin's own) runs once
a launch has found many particles outside their bins' cells, and the first again
when they are few.  Each launch against the oracle, with the particle tests'
tolerances: particles moved by less than a cell, a cell and several, in one bin
of one and of three chunks, in sparse and in full bins, across the domain's
faces."""
import numpy as np
import pytest

import oracle
from sgtest import rel_linf
from test_gpu_g2p2g import TOL, _setup
from workload import ParticleSpec, cube_particles

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    yield


def _steps(spec, max_leaves, shifts):
    import torch
    C0 = np.random.default_rng(spec.n).normal(0.0, 1.0, size=(spec.n, 9)).astype(np.float32)
    A, B, oA, x, v, ox, ov = _setup(spec, C0, max_leaves)
    A.sync()
    x0 = ox.copy()
    for shift in shifts:
        ox = (x0 + shift).astype(np.float32)
        x.copy_(torch.from_numpy(ox))
        torch.cuda.synchronize()
        B.deactivate_all()
        A.g2p2g(B, x, v, spec.dt, 1, spec.pmass, 0, 1)
        B.sync()
        oC = np.zeros((spec.n, 9), np.float32)
        oA.g2p_apic(ox, ov, oC, spec.dt, 1)
        gx, gv = x.cpu().numpy(), v.cpu().numpy()
        assert rel_linf(gv, ov) <= TOL
        assert np.max(np.abs(gx.astype(np.float64) - ox)) <= 4e-7
        oB = oracle.Grid(spec.N, spec.L, 4)
        oB.p2g_apic(gx, ov, oC, spec.pmass, 0, 1)
        gb, gm = B.read_structure()
        ob, om = oB.structure()
        np.testing.assert_array_equal(gb, ob)
        np.testing.assert_array_equal(gm, om)
        for f in range(4):
            assert rel_linf(B.read_field(f), oB.read_field(f)) <= TOL, f
    A.close()
    B.close()


def _many_few(shift):
    """Many moved twice, few twice: first form, second, second, first."""
    few = shift.copy()
    few[len(shift) // 20:] = 0.0
    return [shift, shift, few, few]


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n", [40, 200, 1473])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("cells", [1.0, -1.0])
def test_one_bin(n, axis, cells, L, N=32):
    rng = np.random.default_rng(n + axis)
    base = np.array([8, 12, 16]) + rng.integers(0, 4, size=(n, 3))
    x = ((base + rng.uniform(0.5, 1.5, size=(n, 3))) / N).astype(np.float32)
    v = rng.normal(0.0, 0.01, size=(n, 3)).astype(np.float32)
    shift = np.zeros((n, 3))
    shift[:, axis] = np.where(np.arange(n) % 5 == 4, 2.0 * cells, cells) / N
    _steps(ParticleSpec(N, L, n, np.zeros((3, 3)), np.zeros(3), x, v, note="one bin"), 512, _many_few(shift))


@pytest.mark.parametrize("L", [4, 8])
@pytest.mark.parametrize("n,lo,hi", [(3000, 20.0, 50.0), (60000, 20.0, 50.0)])
@pytest.mark.parametrize("moved", [0.6, 0.99, 3.0])
def test_box(n, lo, hi, moved, L, N=64):
    rng = np.random.default_rng(n)
    x = (rng.uniform(lo, hi, size=(n, 3)) / N).astype(np.float32)
    v = rng.normal(0.0, 0.1, size=(n, 3)).astype(np.float32)
    shift = rng.uniform(-moved, moved, size=(n, 3)) / N
    _steps(ParticleSpec(N, L, n, np.zeros((3, 3)), np.zeros(3), x, v, note="box"), (N // L) ** 3, _many_few(shift))


@pytest.mark.parametrize("L", [4, 8])
def test_domain_faces(L):
    spec = cube_particles(seed=33 + L, n=20000, N=64, L=L, pad_cells=3.0)
    shift = np.random.default_rng(7).uniform(-1.5, 1.5, size=(spec.n, 3)) / spec.N
    _steps(spec, (64 // L) ** 3, _many_few(shift))
