"""The particle kernels' check that a chunk's sort has no more particles than
the chunk can hold: a scan of larger counts latches the error with its site (the
loops over the records take no more than there are), one of counts that fit does
not.  The scans are called by a kernel of the test's own, on counts it sets."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "%s/sg_g2p2g.cu"
using namespace sg;
template <typename S, int CELLS, bool MOVED>
__global__ void k_scan(DevGrid g, int per_cell, int cap, int *total)
{
    __shared__ S s;
    for (int q = threadIdx.x; q <= CELLS; q += 32) s.cnt[q] = per_cell;
    if (threadIdx.x == 0) for (auto &m : s.all) m = 0;
    __syncwarp();
    if constexpr (MOVED) moved_scan(g, s, cap);
    else bin_scan(g, s, cap);
    __syncwarp();
    if (threadIdx.x == 0) *total = s.start[CELLS + 1];
}
extern "C" int run(int moved, int per_cell, int cap, int *out)
{
    DevGrid g{};
    int *total = nullptr;
    Ctrl c{};
    if (cudaMalloc((void **)&g.ctrl, sizeof(Ctrl)) || cudaMalloc((void **)&total, sizeof(int)) ||
        cudaMemset(g.ctrl, 0, sizeof(Ctrl)))
        return 1;
    if (moved) k_scan<MovedSort, kFarCell, true><<<1, 32>>>(g, per_cell, cap, total);
    else k_scan<BinSort, 64, false><<<1, 32>>>(g, per_cell, cap, total);
    if (cudaMemcpy(&c, g.ctrl, sizeof c, cudaMemcpyDeviceToHost) || cudaMemcpy(out, total, sizeof(int), cudaMemcpyDeviceToHost))
        return 2;
    out[1] = c.err;
    out[2] = c.timeout_site;
    cudaFree(g.ctrl);
    cudaFree(total);
    return 0;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2012_08141_gb300 import build as sgbuild
    d = tmp_path_factory.mktemp("scan")
    src, lib = d / "scan.cu", d / "libscan.so"
    src.write_text(SOURCE % sgbuild.CSRC)
    subprocess.run([sgbuild.nvcc(), "-shared", "-std=c++17", "-O1", "-Xcompiler", "-fPIC", "-cudart", "static",
                    f"-I{os.path.join(sgbuild.ROOT, 'include')}", *sgbuild.GENCODE, str(src), "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib)).run


@pytest.mark.parametrize("moved,cells,site", [(0, 65, 107), (1, 217, 106)])
@pytest.mark.parametrize("per_cell", [0, 1, 3, 12])
def test_a_sort_that_does_not_fit_is_an_error(run, moved, cells, site, per_cell):
    out = (ctypes.c_int * 3)()
    assert run(moved, per_cell, 736, out) == 0
    assert out[0] == cells * per_cell
    over = cells * per_cell > 736
    assert (out[1] != 0, out[2]) == (over, site if over else 0)
