"""What the library launches, without a GPU: its object files linked with a runtime that records the
launches (tests/host/fake_cudart.cpp).  Here the shapes of the launches count, which no result on a
GPU shows: the outputs of a launch that relies on undefined behaviour can be right by chance."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
PTR = 1 << 32   # any 256-byte aligned address: nothing is read through it


@pytest.fixture(scope="module")
def native(tmp_path_factory):
    """(the package's ctypes declarations, the library on the recording runtime)"""
    from paper_2104_08863_gb300 import _native
    from paper_2104_08863_gb300 import build as b
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    b.build()
    objs = [os.path.join(b.OBJDIR, os.path.basename(s)[:-3] + ".o") for s in b.sources()]
    if not all(map(os.path.exists, objs)):
        b.build(force=True)
    out = str(tmp_path_factory.mktemp("recorded") / "libpoisson_recorded.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b._nvcc()))), "include")
    subprocess.run([cxx, "-shared", "-fPIC", "-std=c++17", "-I" + inc, "-o", out, "-Wl,-Bsymbolic,-z,defs",
                    os.path.join(HERE, "host", "fake_cudart.cpp"), *objs], check=True)
    L = ctypes.CDLL(out)
    L.fake_name.restype = ctypes.c_char_p
    L.poisson_solve.argtypes = [ctypes.c_void_p] * 4
    L.poisson_set_workspace.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]
    return _native, L


def _plan(native, nx, ny, nz, precision, **kw):
    N, L = native
    faces = np.ascontiguousarray(W.tanh_faces(ny, 1.5))
    d = N.PoissonDesc(nx, ny, nz, 2 * np.pi, np.pi, faces.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), precision,
                      kw.get("tridiag", 0), kw.get("pdd_parts", 0), 4, kw.get("refine_steps", 1), kw.get("flags", 0))
    h, size = ctypes.c_void_p(), ctypes.c_size_t()
    assert L.poisson_plan_create(ctypes.byref(d), ctypes.byref(h)) == 0
    assert L.poisson_workspace_size(h, ctypes.byref(size)) == 0
    return h, size.value


def _solve(native, h, size):
    """[(kernel, block threads, shared bytes)] of one solve; the call has to succeed."""
    L = native[1]
    assert L.poisson_set_workspace(h, PTR, size, None) == 0
    L.fake_clear()
    assert L.poisson_solve(h, PTR, PTR << 1, None) == 0
    out = []
    for i in range(L.fake_count()):
        v = (ctypes.c_ulonglong * 7)()
        L.fake_dims(i, v)
        out.append((L.fake_name(i).decode(), v[3] * v[4] * v[5], v[6]))
    return out


HALF = [2 ** a * 3 ** b for a in range(11) for b in range(7)
        if 8 <= 2 ** a * 3 ** b <= 1024 and 2 ** a * 3 ** b not in (864, 972)]


@pytest.mark.parametrize("generic", [0, 4])
@pytest.mark.parametrize("half", HALF)
def test_gauge_sum_runs_in_whole_warps(native, half, generic):
    """The inverse x-transform that adds up the refined pressure's weighted sum does so with shuffles of all
    32 lanes, so its CTAs are whole warps."""
    h, size = _plan(native, 2 * half, 8, 16, 2, refine_steps=2, flags=generic)
    inv = [k for k in _solve(native, h, size) if "inv_x" in k[0]]
    assert len(inv) == 3
    assert all(t % 32 == 0 for _, t, _ in inv[:2]), inv   # the last pass adds nothing up
    native[1].poisson_plan_destroy(h)


def test_limits_and_grids_are_set_up_on_each_device(native):
    """A kernel's shared-memory limit and the number of its CTAs that are resident belong to a device: the
    second device's first call raises its own limits (a launch above 48 KB fails without) and asks for
    its own grid size."""
    L = native[1]
    h, size = _plan(native, 1536, 96, 64, 2, tridiag=2, pdd_parts=4)   # piped x-transform, PDD blocks of 24 rows
    queries = []
    try:
        for dev in (1, 2):   # no other test runs on these
            L.fake_set_device(dev)
            kernels = _solve(native, h, size)
            queries.append(L.fake_occupancy_queries())
            assert any(smem > 48 << 10 for _, _, smem in kernels)
    finally:
        L.fake_set_device(0)
        L.poisson_plan_destroy(h)
    assert queries[0] == queries[1] == 1


@pytest.mark.parametrize("flags", [0, 4])
@pytest.mark.parametrize("nx,ny,nz", [(24, 100, 96), (108, 5, 432), (128, 55, 36), (128, 18, 108), (972, 33, 8)])
def test_fp64_grids_that_just_fit_the_static_workspace(native, nx, ny, nz, flags):
    """FP64 plans hold one form of the unit roots per direction: with the unit roots alone these grids leave
    256 to 8,192 bytes of the library's 8 MB workspace, and the (cos, tan) form takes no more."""
    L = native[1]
    h, size = _plan(native, nx, ny, nz, 0, flags=flags)
    assert size <= 8 << 20
    L.poisson_solve_static_ws.argtypes = [ctypes.c_void_p] * 4
    assert L.poisson_solve_static_ws(h, PTR, PTR << 1, None) == 0
    L.poisson_plan_destroy(h)


@pytest.mark.parametrize("tridiag", [2, 3])
@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("ny", [24, 37, 96, 130, 221, 247, 253, 289, 377])
def test_naming_the_automatic_partition_gives_the_automatic_plan(native, ny, precision, tridiag):
    """poisson_autotune names its candidates, and so does a caller who keeps a partition: the partition that
    0 stands for gives the same kernels and the same workspace when it is named."""
    def kernels(parts):
        h, size = _plan(native, 36, ny, 16, precision, tridiag=tridiag, pdd_parts=parts)
        out = _solve(native, h, size)
        native[1].poisson_plan_destroy(h)
        return size, out
    auto = kernels(0)
    if precision and ny in (221, 247, 253):   # blocks of 17, 19, 23 rows
        assert any("k_tridiag_reg" in k[0] for k in auto[1])
    same = [p for p in range(1, 257) if ny % p == 0 and (p <= 32 or (precision and ny // p in (1, 2, 3, 4, 6, 8)))
            and kernels(p) == auto]
    assert len(same) >= 1


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("nx,ny,nz", [(16, 8, 16), (162, 90, 108), (16, 3072, 16), (16, 3456, 16), (16, 8192, 16)])
def test_launch_count_is_what_was_launched(native, nx, ny, nz, precision):
    """Above 3072 rows the modes solved apart are a launch of their own."""
    h, size = _plan(native, nx, ny, nz, precision, refine_steps=2)
    kernels = _solve(native, h, size)
    assert native[1].poisson_last_launch_count(h) == len(kernels)
    native[1].poisson_plan_destroy(h)
