"""Bounds-check builds with warps that have tiles of their own: an index that is out of range in any warp
of a CTA is flagged, and the kernels of one or two warps per tile pass their tests in such a build."""
import ctypes
import os
import subprocess
import sys

import pytest
import torch

from paper_1607_03062_gb300 import build as Bd

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Four warps check their own index and range; nothing is accessed with either.
SHIM = r"""
#include "dsp_device.cuh"
__global__ void check(int bad_tile, int bad_range, int *err)
{
    dsp::ReqDesc R;
    R.n_tiles = 4;
    R.table_steps = 10;
    R.step_begin = 0;
    const int w = threadIdx.x >> 5;
    R.step_end = w == bad_range ? 11 : 10;
    (void)dsp::tile_ok(R, w == bad_tile ? 4 : w, err);
    (void)dsp::table_range_ok(R, R.step_begin, err);
}
extern "C" int run(int bad_tile, int bad_range, int *err)
{
    check<<<1, 128>>>(bad_tile, bad_range, err);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    d = tmp_path_factory.mktemp("bounds")
    (d / "shim.cu").write_text(SHIM)
    lib = d / "libshim.so"
    subprocess.run([Bd._nvcc(), "-shared", str(d / "shim.cu"), "-o", str(lib), "-DDSP_BOUNDS_CHECK"]
                   + Bd.COMMON + Bd.ARCH, check=True)
    fn = ctypes.CDLL(os.fspath(lib)).run
    fn.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p]

    def run(bad_tile, bad_range):
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert fn(bad_tile, bad_range, err.data_ptr()) == 0
        return int(err.item())
    return run


def test_any_warp_flags_its_index(check):
    assert check(-1, -1) == 0
    for w in range(4):
        assert check(w, -1) == 2 and check(-1, w) == 2, w


def test_warp_tiles_under_bounds_check_build():
    lib = Bd.build(bounds_check=True)
    env = dict(os.environ, DSP_LIBRARY=lib)
    files = ("test_expanded_groups.py", "test_f64_shapes.py", "test_expansion_wide.py")
    out = subprocess.run([sys.executable, "-m", "pytest", "-q", "-p", "no:cacheprovider", "-m", "gpu"]
                         + [os.path.join(ROOT, "tests", f) for f in files],
                         cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stdout[-3000:] + out.stderr[-2000:]
    assert " passed" in out.stdout
