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
#include <set>
#include <cuda_runtime.h>

// What the launch code asks the driver, answered for a GPU of 152 SMs.
static std::set<int> limits;                 // shared-memory limits that were set
static cudaError_t fake_device(int* d) { *d = 0; return cudaSuccess; }
static cudaError_t fake_attribute(int* v, cudaDeviceAttr a, int) {
    *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 1;
    return cudaSuccess;
}
template <class F> static cudaError_t fake_limit(F, cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limits.insert(v);
    return cudaSuccess;
}
template <class F> static cudaError_t fake_blocks(int* b, F, int, size_t) { *b = 1; return cudaSuccess; }
static cudaError_t fake_clusters(int* c, const void*, const cudaLaunchConfig_t*) { *c = 1; return cudaSuccess; }
static cudaError_t fake_memset(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
static cudaError_t refusal = cudaSuccess, pending = cudaSuccess;    // of launches
static int launches = 0;
static cudaError_t fake_last() { const cudaError_t e = pending; pending = cudaSuccess; return e; }
template <class... A> static cudaError_t fake_launch(A&&...) { ++launches; return pending = refusal; }
#define cudaGetDevice fake_device
#define cudaDeviceGetAttribute fake_attribute
#define cudaFuncSetAttribute fake_limit
#define cudaOccupancyMaxActiveBlocksPerMultiprocessor fake_blocks
#define cudaOccupancyMaxActiveClusters fake_clusters
#define cudaMemsetAsync fake_memset
#define cudaGetLastError fake_last
#define cudaLaunchKernelEx fake_launch
#define cudaLaunchCooperativeKernel fake_launch
#include "resident_cg.cuh"
#include "resident_gmres.cuh"
using namespace sa;
static int bad = 0;
#define CHECK(c) do { if (!(c)) { printf("line %d: %s\n", __LINE__, #c); bad = 1; } } while (0)

// Layout of the FP64 grid team.
static ResLayout layout(int n, int W, int reach) {
    ResLayout L;
    CHECK(grid_layout(n, W, reach, 8, team_room(), &L));
    return L;
}

static SlotPlan five(int reach) {
    SlotPlan p = {};
    p.W = p.list.count = 5;
    p.reach = reach;
    const int off[5] = {-reach, -1, 0, 1, reach};
    for (int k = 0; k < 5; ++k) p.list.off[k] = off[k];
    return p;
}
template <class Sys> static bool cg(int n, int reach) {
    return launch_resident_cg<Sys>(nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, n, 5, reach,
                                   nullptr);
}
template <class Sys> static bool gmres(int n, int reach, int sweeps) {
    GmresArgs<typename Sys::T> A = {};
    A.R = 30;
    A.sweeps = sweeps;
    return launch_resident_gmres<Sys>(nullptr, nullptr, A, n, five(reach), nullptr);
}

// The limit of a kernel's dynamic shared memory belongs to the process: whatever
// the size of a launch, it is set to the same value.
static void one_limit() {
    for (int f = 0; f < 2; ++f) {
        limits.clear();
        for (int n : {33, 4096, 20000, 30000, 70000, 262144})
            CHECK(f ? cg<SysF32>(n, 100) : cg<SysF64>(n, 100));
        CHECK(limits.size() == 1);
        limits.clear();
        for (int n : {33, 4096, 20000, 30000})
            for (int sweeps : {0, 3}) CHECK(f ? gmres<SysF32>(n, 100, sweeps) : gmres<SysF64>(n, 100, sweeps));
        CHECK(limits.size() == 1);
    }
}

// The grid's wait counter past 2^32: 152 blocks add one each per wait.
static void counter_wraps() {
    for (unsigned long long waits : {1ull, 28256362ull, 28256363ull, 28256364ull, 56512727ull, 4294967297ull}) {
        const unsigned want = (unsigned)waits * 152u;
        for (unsigned k = 0; k <= 304; ++k) {      // this wait's and the next one's arrivals
            const unsigned seen = want - 152u + k;
            CHECK(team_arrived(seen, want) == (k >= 152));
        }
    }
}

// Rule and launch agree: a solve is launched where a team is said to take it.
static void takes() {
    for (int n : {33, 1000, 20000, 30000, 65000, 65536, 262144, 1000000})
        for (int reach : {0, 100, 4000, 5000, 6000, 9999, 14000, 16000, 28000, 40000}) {
            if (reach >= n) continue;
            CHECK(cg<SysF64>(n, reach) == resident_cg_takes(n, 5, reach, 8, team_room()));
            CHECK(cg<SysF32>(n, reach) == resident_cg_takes(n, 5, reach, 4, team_room()));
        }
    CHECK(!cg<SysF64>(65000, 28000) && cg<SysF64>(65000, 9999));
    // the line of the long reaches: 64^3, 80^3, 100^3, flat grids; FP32 has none
    CHECK(cg<SysF64>(262144, 4096) && !cg<SysF64>(512000, 6400) && !cg<SysF64>(1000000, 10000));
    CHECK(cg<SysF64>(1000000, 8000) && !cg<SysF64>(200000, 10000) && cg<SysF64>(65535, 10000));
    CHECK(cg<SysF64>(70000, 4523) && !cg<SysF64>(70000, 4524));
    CHECK(cg<SysF32>(512000, 6400) && cg<SysF32>(1000000, 10000) && cg<SysF32>(200000, 10000));
}

// A launch that the driver refuses is no solve: the caller takes the streaming
// kernels, and no error is left behind for its next check.
static void refused() {
    refusal = cudaErrorCooperativeLaunchTooLarge;
    for (int n : {4096, 30000, 262144}) {
        launches = 0;
        CHECK(!cg<SysF64>(n, 100) && !cg<SysF32>(n, 100) && launches >= 2 && pending == cudaSuccess);
    }
    launches = 0;
    CHECK(!gmres<SysF64>(10000, 100, 0) && !gmres<SysF32>(10000, 100, 3) && launches == 2 &&
          pending == cudaSuccess);
    refusal = cudaSuccess;
}

int main() {
    one_limit();
    takes();
    refused();
    counter_wraps();
    // The sizes of the offset-view solves: x does not fit in shared memory.
    CHECK(layout(1001 * 1001, 5, 1001).x_in == 0);
    CHECK(layout(30000, 5, 14000).x_in == 0);
    CHECK(layout(30000, 5, 100).x_in == 1);
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


BATCH = r'''
#include <cstdio>
#include "batch_layout.cuh"
using namespace sa;
int main() {
    int bad = 0;
    for (int M = 1; M <= kBatchMaxM; ++M)
        for (int s = 1; s <= kBatchMaxS; ++s) {
            // two blocks on an SM (228 KB, 1 KB of each reserved, 4 KB for static arrays)
            if (2 * (batch_smem_bytes(s, M) + 5 * 1024) > 228 * 1024) bad = printf("room: %d %d\n", M, s);
            // what follows the sketch lies below its sum
            if (after_sketch_doubles(s, M) > sketch_regions_doubles(s, M + 1)) bad = printf("over: %d %d\n", M, s);
        }
    // a cluster's CTAs keep a sequence on the chip up to a reach of half their rows
    ResLayout L;
    const size_t room = 220 * 1024;
    if (!batch_resident(20480, 5, 1280, 8, room, &L) || batch_resident(20480, 5, 1281, 8, room, &L) ||
        !batch_resident(3000, 5, 1499, 1, room, &L)) bad = printf("reach");
    return bad != 0;
}
'''


def test_two_batch_blocks_fit_on_an_sm(tmp_path):
    """Every size of a batch leaves room for the two blocks per SM that a schedule
    may name."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "batch.cu", tmp_path / "batch"
    src.write_text(BATCH)
    r = subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                        os.path.join(ROOT, "paper_2309_02156_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


# Lines of the resident GMRES: the sizes, and the reach at which fetching the
# neighbours' rows costs more than the streaming kernels' launches.
GMRES_LINES = r'''
int main() {
    CHECK(gmres<SysF64>(10000, 4500, 0) && gmres<SysF64>(92160, 303, 0) && !gmres<SysF64>(92161, 303, 0));
    CHECK(gmres<SysF64>(38912, 3001, 0) && gmres<SysF64>(38913, 3000, 0) && !gmres<SysF64>(38913, 3001, 0));
    CHECK(gmres<SysF64>(77825, 1000, 0) && !gmres<SysF64>(77825, 1001, 0));
    CHECK(gmres<SysF64>(30000, 1000, 8) && !gmres<SysF64>(30000, 1001, 8));
    CHECK(gmres<SysF64>(40000, 333, 8) && !gmres<SysF64>(40000, 334, 8));
    CHECK(gmres<SysF64>(77824, 279, 8) && !gmres<SysF64>(77825, 279, 8) && gmres<SysF64>(77825, 279, 1));
    CHECK(!long_fetch(9, 177, 8, 16, 8) && long_fetch(9, 178, 8, 16, 8) && !long_fetch(5, 178, 8, 16, 8));
    CHECK(gmres<SysF32>(20000, 1800, 0) && !gmres<SysF32>(20000, 1801, 0));
    CHECK(gmres<SysF32>(196608, 443, 0) && !gmres<SysF32>(196609, 443, 0));
    CHECK(gmres<SysF32>(20000, 277, 8) && !gmres<SysF32>(20000, 278, 8));
    CHECK(gmres<SysF32>(73728, 271, 8) && !gmres<SysF32>(73729, 271, 8));
    return bad;
}
'''


def test_gmres_lines(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "lines.cu", tmp_path / "lines"
    src.write_text(PROGRAM.split("int main()")[0] + GMRES_LINES)
    r = subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                        "arch=compute_103a,code=sm_103a", "-I",
                        os.path.join(ROOT, "paper_2309_02156_gb300", "csrc"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
