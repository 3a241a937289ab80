"""Failed allocations while the row clusters are built (no GPU): the call
reports it, nothing is thrown or aborted, and the matrix stays eligible for the
next call. A small program linked against libnm.so replaces operator new, so
that the n-th allocation after arming fails; without a device every device
allocation fails by itself."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1906_11082_gb300")

PROGRAM = r"""
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <new>
#include "kernels.h"
#include "nm_internal.h"
static std::atomic<long> left{-1};
void* operator new(std::size_t n) {
    if (left.load() >= 0 && left.fetch_sub(1) == 0) throw std::bad_alloc();
    void* p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
int main(int argc, char** argv) {
    nm::DevCSR A;
    const int n = 1000, half = 4;
    A.h_rowptr.push_back(0);
    for (int i = 0; i < n; ++i) {
        for (int j = i - half; j <= i + half; ++j)
            if (j >= 0 && j < n) A.h_col.push_back(j);
        A.h_rowptr.push_back((int)A.h_col.size());
    }
    A.nrows = A.ncols = n;
    A.nnz = A.h_rowptr.back();
    left = std::atol(argv[1]);
    const int rc = nm::build_clusters(A, nullptr);
    const bool hit = left.load() < 0 && std::atol(argv[1]) >= 0;
    left = -1;
    std::printf("%d %d %d\n", rc, A.cl_state, (int)hit);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("device allocations succeed here")
    from paper_1906_11082_gb300 import _build
    _build.build()
    d = tmp_path_factory.mktemp("clusters")
    src, out = d / "program.cpp", d / "program"
    src.write_text(PROGRAM)
    subprocess.run([_build._nvcc(), _build.ARCH, "-std=c++17", "-I", os.path.join(PKG, "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-o", str(out), str(src), "-L", PKG, "-lnm", "-Xlinker",
                    "-rpath=" + PKG], check=True)
    return str(out)


# -1: the host part succeeds and the first device allocation fails
@pytest.mark.parametrize("nth", [-1, 0, 2, 5, 20, 40])
def test_failed_allocation(program, nth):
    r = subprocess.run([program, str(nth)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    rc, state, hit = map(int, r.stdout.split())
    assert hit == (nth >= 0)
    assert rc != 0 and state == 0
    if nth >= 0:
        assert rc == 2   # NM_ENOMEM
