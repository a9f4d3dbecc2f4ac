"""A CUDA call that fails inside gs_bin_sort is returned, and nothing that reads what it would have written is launched:
the library's own host code against a stand-in for the CUDA runtime (no GPU)."""
import ctypes
import glob
import os
import subprocess

import pytest

from paper_2509_06433_gb300 import _lib, build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def faked(tmp_path_factory):
    lib = build()
    objs = sorted(glob.glob(os.path.join(os.path.dirname(lib), "*.o")))
    out = str(tmp_path_factory.mktemp("fake") / "libgs_fake.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{cuda}/include", os.path.join(HERE, "fake_cudart.cpp"),
                    *objs, "-o", out, "-Wl,-Bsymbolic", "-ldl", "-lpthread"], check=True)
    L = ctypes.CDLL(out, mode=os.RTLD_LOCAL)
    L.fake_launched.restype = ctypes.c_char_p
    return L


def _bin_sort(L, width, height, n, fail_attr=b"", fail_launch=b""):
    cfg = _lib.GsConfig()
    ctypes.memset(ctypes.byref(cfg), 0, ctypes.sizeof(cfg))
    cfg.width, cfg.height, cfg.tile, cfg.num_views, cfg.num_gaussians = width, height, 16, 1, n
    cfg.pair_capacity, cfg.near_plane, cfg.lambda_depth = 1 << 16, 0.2, 0.1
    size = ctypes.c_size_t()
    assert L.gs_workspace_size(ctypes.byref(cfg), ctypes.byref(size)) == 0
    L.fake_reset(fail_attr, fail_launch)
    code = L.gs_bin_sort(ctypes.byref(cfg), ctypes.c_void_p(1 << 20), size, None)  # (never read: nothing runs)
    launched = L.fake_launched().decode()
    assert L.cudaGetLastError() == 0  # no error left for the next call of the process to find
    return code, launched


@pytest.mark.parametrize("width,height,n", [(640, 480, 1000), (5000, 48, 1000), (64, 48, 1000)])
def test_the_chain_without_a_failure(faked, width, height, n):
    code, launched = _bin_sort(faked, width, height, n)
    assert code == 0 and "k_tile_scan" in launched
    assert ("k_tile_emit" in launched) == (width * height > 152 * 256)


@pytest.mark.parametrize("width,height,n", [(640, 480, 1000), (5000, 48, 1000), (64, 48, 1000)])
def test_tile_scan_that_cannot_be_launched(faked, width, height, n):
    code, launched = _bin_sort(faked, width, height, n, fail_launch=b"k_tile_scan")
    assert code == 5 and "emit" not in launched and "k_tile_sort" not in launched


def test_tile_scan_without_its_shared_memory(faked):
    code, launched = _bin_sort(faked, 5000, 48, 1000, fail_attr=b"k_tile_scan")
    assert code == 5 and "scan" not in launched and "emit" not in launched and "k_tile_sort" not in launched
