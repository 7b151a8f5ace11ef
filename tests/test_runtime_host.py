"""CPU tests of the library's host side over a fake CUDA runtime
(fake_cudart.cpp linked with the library's objects): what it asks of the
runtime on several devices, while a stream is recorded and after refused calls.
Kernels do not run; their launches are logged."""
import ctypes
import glob
import os
import subprocess

import pytest

import paper_2012_08141_gb300 as sg
from paper_2012_08141_gb300 import build as sgbuild

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    sgbuild.build(force=sgbuild.is_stale() or not all(
        os.path.exists(os.path.join(sgbuild.BUILD, s.replace(".cu", ".o"))) for s in sgbuild.SOURCES))
    objs = [os.path.join(sgbuild.BUILD, s.replace(".cu", ".o")) for s in sgbuild.SOURCES]
    out = str(tmp_path_factory.mktemp("fake") / "libsgrid_fake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(sgbuild.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", f"-I{include}",
                    os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-o", out], check=True)
    real = sg.load_library()
    lib = ctypes.CDLL(out)
    for name in sg.header_functions():
        fn, ref = getattr(lib, name), getattr(real, name)
        fn.argtypes, fn.restype = ref.argtypes, ref.restype
    lib.fake_log.restype = lib.sg_last_error.restype = ctypes.c_char_p
    return lib


class Grid:
    """A grid over the fake runtime: the C calls, errors as codes."""

    def __init__(self, lib, device=0, stream=None, lg2=2, fields=4):
        self.lib, self.h = lib, ctypes.c_void_p()
        lib.fake_device(device)
        d = sg.SgDesc(64, lg2, fields, 4, 512, 0, 0)
        self.rc = lib.sg_create(ctypes.byref(d), stream, ctypes.byref(self.h))

    def __call__(self, name, *args):
        return getattr(self.lib, name)(self.h, *args)

    def log(self, *names):
        """How often each of the kernels was launched since the last look."""
        text = self.lib.fake_log().decode().split(";")
        self.lib.fake_clear_log()
        return [sum(n in t for t in text) for n in names]


def _particles(n):
    return [ctypes.cast((ctypes.c_float * (k * n))(), ctypes.c_void_p) for k in (3, 3, 9)]


@pytest.mark.parametrize("lg2", [2, 3])
@pytest.mark.parametrize("affine", [False, True])
def test_particle_transfers_on_every_device(lib, lg2, affine):
    """Each device's first P2G and G2P2G allow their shared memory there."""
    x, v, C = _particles(10)
    for device in (0, 1, 3, 0):
        a, b = Grid(lib, device, lg2=lg2), Grid(lib, device, lg2=lg2)
        a.log()
        assert a("sg_p2g_apic", x, v, C if affine else None, 10, 1.0, 0, 1) == 0
        assert a("sg_flush") == 0, lib.sg_last_error()
        assert lib.sg_g2p2g(a.h, b.h, x, v, 10, 0.1, 1, 1.0, 0, 1) == 0, lib.sg_last_error()
        assert a.log("k_p2g_gather", "k_g2p2g") == [1, 2]  # two forms of G2P2G, the device picks one
        assert a("sg_destroy") == b("sg_destroy") == 0
    lib.fake_device(0)


def test_refused_shared_memory_is_an_error(lib):
    """A device that refuses the shared memory: an error, nothing launched, and
    the same call passes once it is allowed."""
    x, v, _ = _particles(10)
    g = Grid(lib, 7)
    g.log()
    lib.fake_refuse_attributes(1)
    assert g("sg_p2g", x, v, 10, 1.0, 0, 1) == 0
    assert g("sg_flush") == sg.SG_ERR_CUDA
    lib.fake_refuse_attributes(0)
    assert g.log("k_") == [0]
    assert g("sg_p2g", x, v, 10, 1.0, 0, 1) == 0
    assert g("sg_flush") == 0, lib.sg_last_error()
    assert g.log("k_p2g_bin", "k_p2g_gather") == [1, 1]
    assert g("sg_destroy") == 0
    lib.fake_device(0)


@pytest.mark.parametrize("refused", ["recording", "device"])
def test_refused_binning_leaves_no_order(lib, refused):
    """A P2G that was refused (in a recording, or by the device) has put no
    particle order in memory: nothing of it is launched or recorded, the next
    P2G bins from the positions, G2P takes the input order, and G2P2G and the
    reordering are refused."""
    x, v, _ = _particles(10)
    stream = ctypes.c_void_p(4096)
    a, b = Grid(lib, 0, stream), Grid(lib, 0, stream)
    a.log()
    assert a("sg_p2g", x, v, 10, 1.0, 0, 1) == 0
    if refused == "recording":
        assert lib.sg_graph_begin(stream) == 0
        assert a("sg_flush") == sg.SG_ERR_INVALID
        graph = ctypes.c_void_p()
        assert lib.sg_graph_end(stream, ctypes.byref(graph)) == lib.sg_graph_destroy(graph) == 0
    else:
        lib.fake_device(8)
        lib.fake_refuse_attributes(1)
        assert a("sg_flush") == sg.SG_ERR_CUDA
        lib.fake_refuse_attributes(0)
        lib.fake_device(0)
    assert a.log("k_") == [0]
    assert lib.sg_g2p2g(a.h, b.h, x, v, 10, 0.1, 1, 1.0, 0, 1) == sg.SG_ERR_INVALID
    assert a("sg_sort_particles", x, v, None, None, 10) == 0 and a("sg_flush") == sg.SG_ERR_INVALID
    assert a("sg_g2p", x, v, 10, 0.1, 1) == a("sg_flush") == 0
    assert a.log("k_g2p_binned", "k_g2p") == [0, 1]
    for rebin in (0, 1):
        assert a("sg_p2g", x, v, 10, 1.0, 0, 1) == a("sg_flush") == 0, lib.sg_last_error()
        assert a.log("k_p2g_rebin", "k_p2g_bin") == [rebin, 1 - rebin]
    assert a("sg_destroy") == b("sg_destroy") == 0


def test_recorded_g2p2g_records_nothing(lib):
    x, v, _ = _particles(10)
    stream = ctypes.c_void_p(4096)
    a, b = Grid(lib, 0, stream), Grid(lib, 0, stream)
    assert a("sg_p2g", x, v, 10, 1.0, 0, 1) == a("sg_flush") == 0
    a.log()
    assert lib.sg_graph_begin(stream) == 0
    assert lib.sg_g2p2g(a.h, b.h, x, v, 10, 0.1, 1, 1.0, 0, 1) == sg.SG_ERR_INVALID
    assert a.log("k_g2p2g") == [0]
    graph = ctypes.c_void_p()
    assert lib.sg_graph_end(stream, ctypes.byref(graph)) == lib.sg_graph_destroy(graph) == 0
    assert lib.sg_g2p2g(a.h, b.h, x, v, 10, 0.1, 1, 1.0, 0, 1) == 0, lib.sg_last_error()
    assert a("sg_destroy") == b("sg_destroy") == 0


def test_create_beside_an_earlier_error(lib):
    """An error that an earlier call left with the thread (here a read from a
    stream being recorded) is not the new grid's."""
    a = Grid(lib, 0, ctypes.c_void_p(4096))
    assert lib.sg_graph_begin(ctypes.c_void_p(4096)) == 0
    assert a("sg_read_sums", (ctypes.c_double * 4)(), 4) == sg.SG_ERR_CUDA
    b = Grid(lib, 0, ctypes.c_void_p(8192))
    assert b.rc == 0, lib.sg_last_error()
    graph = ctypes.c_void_p()
    assert lib.sg_graph_end(ctypes.c_void_p(4096), ctypes.byref(graph)) == lib.sg_graph_destroy(graph) == 0
    assert a("sg_destroy") == b("sg_destroy") == 0
