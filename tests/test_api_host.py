"""Host logic of the C entry points on failing ways out (no GPU).

csrc/api.cu is compiled for the host with g++ against fakes of the CUDA runtime
and of the device-side parts: device memory is host memory that is counted,
and memory given back is overwritten and kept, so that a use after it shows.
"""
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
#include <malloc.h>
#include <new>
#include <set>
#include <string>
#include "internal.h"
#include "kernels.h"
#include "vgrid.h"

// freed host memory is overwritten and never handed out again
void *operator new(size_t n) { return malloc(n ? n : 1); }
void operator delete(void *p) noexcept { if (p) memset(p, 0xdb, malloc_usable_size(p)); }
void operator delete(void *p, size_t) noexcept { operator delete(p); }

static std::set<void *> &live() { static std::set<void *> *s = new std::set<void *>(); return *s; }
static int bad_frees = 0;

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
    *p = malloc(n);
    live().insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    if (p && !live().erase(p)) bad_frees++;
    return cudaSuccess;
}
cudaError_t cudaMemcpy(void *d, const void *s, size_t n, cudaMemcpyKind) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
}

static int layout_rc = vg::LAYOUT_OK;

namespace vg {
template <class T> static T *dev(int64_t n) {
    void *p;
    cudaMalloc(&p, sizeof(T) * n);
    return (T *)p;
}
int build_cells_gpu(const double *, int64_t M, const double *, int, CellsOut &out, std::string &, int64_t *) {
    out.off.assign(M + 1, 0);
    out.vol.assign(M, 0.0);
    out.bbox.assign(6 * M, 0.0);
    out.d_off = dev<int64_t>(M + 1);
    out.d_idx = dev<int32_t>(1);
    out.d_bbox = dev<double>(6 * M);
    return 0;
}
int build_layout(const LayoutIn &in, LayoutOut &out, std::string &err) {
    if (layout_rc != LAYOUT_OK) {
        err = "fake";
        return layout_rc;
    }
    out.site = dev<float4>(in.M);
    out.cells = dev<float4>(1);
    out.rel = dev<float4>(1);
    out.blk_rec = dev<float4>(1);
    out.perm = dev<int32_t>(in.M);
    out.blk_off = dev<int32_t>(1);
    out.dens = dev<float>(1);
    return LAYOUT_OK;
}
cudaError_t launch_put_grid(GridDev *, const GridDev &, cudaStream_t) { return cudaSuccess; }
}  // namespace vg
"""


def _run(tmp_path, main):
    """Compile api.cu and build.cpp with the fakes and `main`; its output."""
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    prog = tmp_path / "prog.cpp"
    prog.write_text(FAKE + main)
    exe = str(tmp_path / "prog")
    flags = ["-std=c++17", "-O1", "-g0", "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
             "-I", CSRC]
    # what no path of the test calls stays undefined
    subprocess.run(["g++", *flags, "-no-pie", "-fno-pie", "-Wl,--unresolved-symbols=ignore-all", str(prog), "-x", "c++",
                    os.path.join(CSRC, "api.cu"), os.path.join(CSRC, "build.cpp"), "-lpthread", "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    return r.stdout.split("\n")


@pytest.mark.parametrize("gpu_build", [0, 1])
def test_a_failing_layout_frees_each_buffer_once(tmp_path, gpu_build):
    """vgrid_create where the device arrays cannot be made: the error comes
    back, every device buffer is freed exactly once, and the next call works."""
    out = _run(tmp_path, r"""
int main() {
    const double sites[] = {0.1, 0.2, 0.3, -0.5, 0.25, 0.0, 0.5, -0.75, 0.125, 0.0, 0.0, -0.5};
    double S[12];
    for (int i = 0; i < 12; i++) S[i] = (double)(float)sites[i];
    const double box[] = {-1, -1, -1, 1, 1, 1};
    vgrid_opts o;
    vgrid_default_opts(&o);
    o.gpu_build = """ + str(gpu_build) + r""";
    for (int rc : {(int)vg::LAYOUT_NOMEM, (int)vg::LAYOUT_CUDA, (int)vg::LAYOUT_OK}) {
        layout_rc = rc;
        vgrid_t *g = nullptr;
        const int got = vgrid_create(S, 4, box, &o, &g);
        if (got == VGRID_OK) vgrid_destroy(g);
        printf("%d %d %zu\n", got, bad_frees, live().size());
    }
    printf("%d %d %d\n", VGRID_ERR_NOMEM, VGRID_ERR_CUDA, VGRID_OK);
    return 0;
}
""")
    nomem, cuda, ok = out[3].split()
    assert out[:3] == [f"{nomem} 0 0", f"{cuda} 0 0", f"{ok} 0 0"]
