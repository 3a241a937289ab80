"""Index range of the combine's grid-stride loop, through a small harness
compiled against libnm.so: totals around 2^32, where a 32-bit counter would
wrap and the loop never end."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1906_11082_gb300")

HARNESS = r"""
#include "kernels.h"
extern "C" int fits(int64_t total, int64_t stride) { return nm::fits_u32(total, stride); }
// rows that share one row of memory: any number of rows in a few hundred bytes
extern "C" int combine(int64_t rows, int b, const float* x, const float* e, double* out) {
    nm::CombineArgs a;
    a.rows = rows;
    a.b = b;
    a.x32 = x;
    a.e32 = e;
    a.out = out;
    return nm::launch_combine(a, 0);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1906_11082_gb300 import _build
    _build.build()
    d = tmp_path_factory.mktemp("combine")
    src, out = d / "harness.cu", d / "libharness.so"
    src.write_text(HARNESS)
    subprocess.run([_build._nvcc(), _build.ARCH, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I",
                    os.path.join(PKG, "csrc"), "-o", str(out), str(src), "-L", PKG, "-lnm", "-Xlinker",
                    "-rpath=" + PKG], check=True)
    return C.CDLL(str(out))


@pytest.mark.parametrize("total", [1, 2 ** 31, 2 ** 32 - 1_245_185, 2 ** 32 - 1_245_184, 2 ** 32 - 1, 2 ** 32, 2 ** 33])
def test_no_wrap(lib, total):
    """The largest counter before the last step plus the stride stays in range."""
    stride = 152 * 32 * 256
    last = total - 1
    wraps = (last + stride) % 2 ** 32 < total and last + stride >= 2 ** 32 or total >= 2 ** 32
    assert not (lib.fits(C.c_int64(total), C.c_int64(stride)) and wraps)
    assert lib.fits(C.c_int64(2 ** 30), C.c_int64(stride))   # every block that fits a device


@pytest.mark.gpu
@pytest.mark.parametrize("rows,b", [(2 ** 32 - 1000, 1), (138_547_333, 31), (2 ** 27, 32), (3 * 2 ** 28 + 1, 24)])
def test_combine_of_many_rows(lib, rows, b):
    torch = pytest.importorskip("torch")
    x, e = torch.randn(2, b, device="cuda")
    x, e = x.clone(), e.clone()
    out = torch.zeros(b, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    rc = lib.combine(C.c_int64(rows), b, C.c_void_p(x.data_ptr()), C.c_void_p(e.data_ptr()), C.c_void_p(out.data_ptr()))
    assert rc == 0
    torch.cuda.synchronize()
    assert bool((out == x.double() + e.double()).all())
