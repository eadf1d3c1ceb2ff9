"""The host side of the small-lattice solves (csrc/cg_cluster.cu) against a fake
CUDA runtime: two devices that allow different things, grants and allocations
that are refused.  No GPU.

The host program links the compiled cg_cluster.cu with stand-ins for the
kernels' launchers and for the runtime calls it makes; it prints one line per
check that fails.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1111_0125_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <string>
#include "cg_cluster.cuh"
using namespace stg;

static int device = 0, queries = 0, fail_host = 0, launches = 0;
// device 0: seven clusters of 16 CTAs; device 1: none; device 2: seven, kernels not granted
extern "C" cudaError_t __wrap_cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t __wrap_cudaMalloc(void **p, size_t n) { *p = calloc(1, n); return cudaSuccess; }
extern "C" cudaError_t __wrap_cudaMallocHost(void **p, size_t n)
{
    if (fail_host) return cudaErrorMemoryAllocation;
    *p = calloc(1, n);
    return cudaSuccess;
}
extern "C" cudaError_t __wrap_cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t)
{
    memcpy(d, s, n);
    return cudaSuccess;
}
extern "C" cudaError_t __wrap_cudaMemsetAsync(void *, int, size_t, cudaStream_t) { return cudaSuccess; }
extern "C" cudaError_t __wrap_cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
namespace stg {
int cl_active_clusters(int ctas) { ++queries; return device == 1 ? 0 : 112 / ctas; }
bool cl_granted_wide(int, int, int) { return device != 2; }
bool cl_granted_16(int, int, int) { return device != 2; }
cudaError_t cl_dispatch_wide(int, int, const ClArgs &a, int n, int, cudaStream_t)
{
    ++launches;
    for (int k = 0; k < n; ++k) a.sys[k].status = CL_OK;
    return cudaSuccess;
}
cudaError_t cl_dispatch_16(int, int, const ClArgs &, int, int, cudaStream_t) { return cudaErrorInvalidValue; }
void set_error(const std::string &) {}
stg_status cuda_fail(cudaError_t, const char *) { return STG_ERR_CUDA; }
const LinkField *links_for(const stg_gauge *g, int prec) { return prec == P64 ? &g->hi : &g->lo; }
stg_status unpack_field(const Geom &, int, const void *, double *, cudaStream_t) { return STG_OK; }
}

static int bad = 0;
static void check(bool ok, const char *what)
{
    if (!ok) { printf("failed: %s\n", what); ++bad; }
}

int main(void)
{
    stg_gauge g = {};
    g.geom.Vh = 2048;
    g.hi.fix = true;
    g.hi.prec = P64;
    g.lo.prec = P32;
    g.lo.recon = 12;
    device = 0;
    check(cluster_ctas(&g, P32, 1, false) == 16, "device 0, first call");
    const int q = queries;
    check(cluster_ctas(&g, P32, 1, false) == 16 && queries == q, "device 0 is asked once");
    device = 1;
    check(cluster_ctas(&g, P32, 1, false) == 0, "device 1 runs no cluster: four kernels");
    check(cluster_ctas(&g, P32, 8, true) == 0, "device 1, batch");
    device = 2;
    check(cluster_ctas(&g, P32, 1, false) == 0, "device 2 does not grant the kernel: four kernels");
    check(cluster_ctas(&g, P64, 1, false) == 0, "device 2, plain FP64");
    check(cluster_ctas(&g, P32, 8, true) == 0, "device 2, batch");
    device = 0;
    check(cluster_ctas(&g, P32, 1, false) == 16, "device 0 again");

    // a refused pinned allocation is an error now and no null pointer later
    Workspace ws;
    ClFields f = {};
    double x = 0, mass = 0.1;
    stg_cg_params p = {};
    fail_host = 1;
    check(cluster_solve(&g, &ws, 16, 1, false, f, &x, &x, &mass, 1e-10, &p, P32, nullptr, 0) != STG_OK, "refused");
    check(cluster_solve(&g, &ws, 16, 1, false, f, &x, &x, &mass, 1e-10, &p, P32, nullptr, 0) != STG_OK,
          "refused again");
    fail_host = 0;
    check(cluster_solve(&g, &ws, 16, 1, false, f, &x, &x, &mass, 1e-10, &p, P32, nullptr, 0) == STG_OK && launches == 1,
          "granted after that");
    printf("done %d\n", bad);
    return bad != 0;
}
"""


FAKES = ["cudaGetDevice", "cudaMalloc", "cudaMallocHost", "cudaMemcpyAsync", "cudaMemsetAsync",
         "cudaStreamSynchronize"]


def _nvcc():
    return shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)


def test_devices_and_refusals(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not available")
    src = tmp_path / "cluster_host_check.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "cluster_host_check"
    r = subprocess.run([nvcc, "-O1", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                        "-gencode", "arch=compute_103a,code=sm_103a",
                        *[a for f in FAKES for a in ("-Xlinker", f"--wrap={f}")], str(src), os.path.join(CSRC, "cg_cluster.cu"), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and "done 0" in r.stdout, r.stdout[-2000:]
