"""A wait between the blocks of a resident solve that runs out: every block leaves,
the status says so and the context stays usable.  The headers are compiled with a
limit of no polls, so that each block gives up at its first wait."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2309_02156_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include <cstring>
#include <vector>
#include <cuda_runtime.h>
#include "resident_cg.cuh"
#include "resident_gmres.cuh"
using namespace sa;
template <class T> static T* room(size_t n) {
    T* p = nullptr;
    if (cudaMalloc(&p, n * sizeof(T)) != cudaSuccess || cudaMemset(p, 0, n * sizeof(T)) != cudaSuccess) return nullptr;
    return p;
}
int main() {
    const int n = 30000, ns = (n + 31) / 32, R = 5;          // above the cluster's sizes; A = 2 I, one slot
    std::vector<int2> slot(ns, make_int2(0, -1));
    slot[ns - 1].y = (1 << (n - 32 * (ns - 1))) - 1;
    std::vector<double> two(32 * ns, 2.0), half(n, 0.5), one(n, 1.0);
    int2* d_slot = room<int2>(ns);
    double *val = room<double>(32 * ns), *b = room<double>(n), *x = room<double>(n);
    double* v[8];
    for (double*& p : v) p = room<double>((R + 1) * (size_t)32 * ns);
    TeamSlot* team = (TeamSlot*)room<unsigned char>(kTeamSlotBytes);
    KState *ks = room<KState>(1), h;
    DevArgs* d_args = room<DevArgs>(1);
    cudaMemcpy(d_slot, slot.data(), sizeof(int2) * ns, cudaMemcpyHostToDevice);
    cudaMemcpy(val, two.data(), 8 * two.size(), cudaMemcpyHostToDevice);
    cudaMemcpy(b, one.data(), 8 * n, cudaMemcpyHostToDevice);
    DevArgs a;
    memset(&a, 0, sizeof a);
    a.b = b;
    a.x = x;
    a.sell_val = val;
    a.slot = d_slot;
    a.n = a.nnz = n;
    a.max_iters = 100;
    a.slot_w = a.slot_off.count = 1;
    a.tol = 1e-10;
    cudaMemcpy(d_args, &a, sizeof a, cudaMemcpyHostToDevice);
    cudaMemcpy(v[2], half.data(), 8 * n, cudaMemcpyHostToDevice);
    SlotPlan plan = {};
    plan.W = plan.list.count = 1;
    int bad = 0;
    for (int form = 0; form < 3; ++form) {                   // CG, GMRES, GMRES with sweeps
        GmresArgs<double> A = {};
        A.V = v[0];
        A.ldv = 32 * (size_t)ns;
        A.R = R;
        A.kpart = v[1];
        A.team = team;
        A.sweeps = form == 2 ? 3 : 0;
        A.omega = 0.8;
        A.dinv = v[2];
        A.za = v[3];
        A.zb = v[4];
        A.t = v[5];
        const bool taken = form == 0
            ? launch_resident_cg<SysF64>(d_args, ks, v[0], v[1], v[6], team, n, 1, 0, (cudaStream_t)0)
            : launch_resident_gmres<SysF64>(d_args, ks, A, n, plan, (cudaStream_t)0);
        const cudaError_t e = cudaDeviceSynchronize();
        cudaMemcpy(&h, ks, sizeof h, cudaMemcpyDeviceToHost);
        printf("form %d taken %d status %d finished %d: %s\n", form, taken, h.status, h.finished,
               cudaGetErrorString(e));
        bad |= !taken || e != cudaSuccess || h.status != ST_OUTCOME || h.finished != 1;
        cudaMemset(ks, 0, sizeof h);
        cudaMemset(x, 0, 8 * n);
    }
    // the context goes on
    bad |= cudaMemcpy(one.data(), b, 8 * n, cudaMemcpyDeviceToHost) != cudaSuccess || one[n - 1] != 1.0;
    return bad;
}
'''


@pytest.mark.parametrize("polls,status", [("1 << 21", "ST_OK"), ("0", "ST_TIMEOUT")])
def test_waits_that_run_out(tmp_path, polls, status):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    for name in os.listdir(CSRC):
        if name.endswith((".cuh", ".h")):
            text = open(os.path.join(CSRC, name)).read()
            if name == "resident.cuh":
                assert text.count("kTeamPolls = 1 << 21;") == 1
                text = text.replace("kTeamPolls = 1 << 21;", f"kTeamPolls = {polls};")
            (tmp_path / name).write_text(text)
    src, exe = tmp_path / "waits.cu", tmp_path / "waits"
    src.write_text(PROGRAM.replace("ST_OUTCOME", status))
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode",
                        "arch=compute_103a,code=sm_103a", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
