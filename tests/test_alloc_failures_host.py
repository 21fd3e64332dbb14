"""Device memory that runs out while a grid is built (no GPU): csrc/build_gpu.cu
and csrc/layout.cu are compiled with nvcc and linked against a fake of the CUDA
runtime that launches nothing and refuses one allocation after the other. Each
time every buffer is given back, and no error stays behind for the next call's
launch check to find."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1310_1854_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

FAKE = r"""
#include <cuda_runtime.h>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include "internal.h"
#include "kernels.h"

static std::set<void *> live;
static int bad_frees = 0, refuse = -1, asked = 0;
static cudaError_t last = cudaSuccess;

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
    if (asked++ == refuse) return last = cudaErrorMemoryAllocation;
    live.insert(*p = calloc(n, 1));
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (p && !live.erase(p)) bad_frees++;
    else free(p);
    return cudaSuccess;
}
cudaError_t cudaGetLastError() {
    const cudaError_t e = last;
    last = cudaSuccess;
    return e;
}
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *, int, size_t, unsigned) {
    *n = 1;
    return cudaSuccess;
}
// kernel launches do nothing
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void *) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(void *, const void *) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
}

namespace vg {
void count_launches(int64_t) {}
int64_t scan_tmp_elems(int64_t) { return 1; }
cudaError_t launch_exclusive_scan(int64_t *, int64_t, int64_t *, cudaStream_t) { return cudaGetLastError(); }
}  // namespace vg

int main() {
    const int64_t M = 64;
    double S[3 * M], box[] = {-1, -1, -1, 1, 1, 1};
    for (int i = 0; i < 3 * M; i++) S[i] = (i % 31) / 32.0 - 0.5;
    std::string err;
    for (refuse = 0;; refuse++) {
        asked = 0;
        vg::CellsOut out;
        int64_t host = 0;
        const int rc = vg::build_cells_gpu(S, M, box, 1, out, err, &host);
        const bool refused = asked > refuse;
        for (void *p : {(void *)out.d_off, (void *)out.d_idx, (void *)out.d_bbox}) cudaFree(p);
        printf("cells %d %d %d %zu %d\n", refused, rc != 0, bad_frees, live.size(), (int)cudaGetLastError());
        if (!refused) break;
    }
    float4 site[M] = {};
    int32_t perm[M] = {}, idx[1] = {};
    int64_t off[M + 1] = {};
    double bbox[6 * M] = {};
    for (refuse = 0;; refuse++) {
        asked = 0;
        vg::LayoutIn in{M, 4, box, 1.0f, {4, 4, 4}, {4, 4, 4}, site, perm, off, idx, bbox, nullptr, nullptr, nullptr};
        vg::LayoutOut out{};
        const int rc = vg::build_layout(in, out, err);
        const bool refused = asked > refuse;
        if (rc == vg::LAYOUT_OK)
            for (void *p : {(void *)out.site, (void *)out.cells, (void *)out.rel, (void *)out.blk_rec, (void *)out.perm,
                            (void *)out.blk_off, (void *)out.dens}) cudaFree(p);
        printf("layout %d %d %d %zu %d\n", refused, rc == vg::LAYOUT_NOMEM, bad_frees, live.size(),
               (int)cudaGetLastError());
        if (!refused) break;
    }
    return 0;
}
"""


def test_every_allocation_refused_in_turn(tmp_path):
    nvcc = shutil.which("nvcc") or os.path.join(CUDA, "bin", "nvcc")
    if shutil.which("g++") is None or not os.path.exists(nvcc):
        pytest.skip("needs nvcc and g++")
    objs = []
    for src in ("build_gpu.cu", "layout.cu"):
        objs.append(str(tmp_path / (src + ".o")))
        subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17", "-cudart", "none",
                               "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-x", "cu", "-c",
                               os.path.join(CSRC, src), "-o", objs[-1]])
    prog, exe = tmp_path / "prog.cpp", str(tmp_path / "prog")
    prog.write_text(FAKE)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", os.path.join(CUDA, "include"), "-I",
                           os.path.join(ROOT, "include"), "-I", CSRC, str(prog), os.path.join(CSRC, "build.cpp"), *objs,
                           "-lpthread", "-o", exe])
    out = [l.split() for l in subprocess.run([exe], capture_output=True, text=True, check=True, timeout=60).stdout.split("\n")
           if l]
    for part in ("cells", "layout"):
        rows = [[int(v) for v in l[1:]] for l in out if l[0] == part]
        assert len(rows) > 10 and rows[-1] == [0, 0, 0, 0, 0]
        # the polyhedra's buffer is asked for again at half the size
        assert sum(r[1] == 0 for r in rows[:-1]) == (1 if part == "cells" else 0)
        for r in rows[:-1]:
            assert r[0] == 1 and r[2:] == [0, 0, 0], (part, r)
