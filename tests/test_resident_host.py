"""Host side of the resident solves (CPU only): a small program that includes the
headers is compiled and run here, without a GPU.  It checks what the launch code
decides before anything runs."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cstdio>
#include "resident.cuh"
using namespace sa;
static int bad = 0;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); bad = 1; } } while (0)

// Layout of the FP64 grid team on 152 SMs, as launch_resident_cg makes it.
static ResLayout grid_layout(int n, int W, int reach) {
    const int ns = (n + 31) / 32;
    int nblk = (ns + 3) / 4;
    if (nblk > 152) nblk = 152;
    ResLayout L;
    CHECK(res_layout(n, W, reach, nblk, 8, 232448 - 2048, &L));
    return L;
}

int main() {
    // The sizes of the offset-view solves: x does not fit in shared memory.
    CHECK(grid_layout(1001 * 1001, 5, 1001).x_in == 0);
    CHECK(grid_layout(30000, 5, 14000).x_in == 0);
    CHECK(grid_layout(30000, 5, 100).x_in == 1);
    return bad;
}
'''


def test_host_decisions(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "host.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "host"
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                        "arch=compute_103a,code=sm_103a", "-I",
                        os.path.join(ROOT, "paper_2309_02156_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
