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


SHAPES = r"""
// kernels are numbers: lanes, then row, then mode
namespace vg {
static void table(KernelSet &k, int lanes) {
    for (int r = 0; r < 3; r++)
        for (int m = 0; m < NUM_MODES; m++) k.fn[r][m] = (const void *)(uintptr_t)(1000 * lanes + 100 * r + m);
}
void kernel_table_lpr1(KernelSet &k) { table(k, 1); }
void kernel_table_lpr2(KernelSet &k) { table(k, 2); }
void kernel_table_lpr4(KernelSet &k) { table(k, 4); }
void kernel_table_lpr8(KernelSet &k) { table(k, 8); }
void count_launches(int64_t) {}
cudaError_t launch_locate(const LocateArgs &, int, int, cudaStream_t) { return cudaSuccess; }
}  // namespace vg
static int lanes, block;
extern "C" {
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *, int b, size_t) {
    *n = 1024 / b;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void *f, dim3, dim3 b, void **, size_t, cudaStream_t) {
    lanes = (int)((uintptr_t)f / 1000);
    block = b.x;
    return cudaSuccess;
}
}
static vgrid_t *g;
static void show(const char *what) {
    static double o[3], d[3], tau[1];
    printf("%s", what);
    for (int p : {VGRID_FP32_RECHECK, VGRID_FP32_EXACT, VGRID_FP64}) {
        vgrid_trace(g, o, d, 64, p, VGRID_TAU, tau, nullptr, nullptr, nullptr, 0, nullptr, nullptr, nullptr);
        printf(" %d/%d", lanes, block);
    }
    printf("\n");
}
static void set(int l, int b, int n, int l64, int order) {
    const vgrid_launch s = {l, b, n, l64, order};
    vgrid_set_launch(g, &s);
}
int main() {
    const double S[] = {0.125, 0.25, 0.375, -0.5, 0.25, 0.0}, box[] = {-1, -1, -1, 1, 1, 1};
    vgrid_opts o;
    vgrid_default_opts(&o);
    vgrid_create(S, 2, box, &o, &g);
    vgrid_launch was, now;
    show("new");
    vgrid_get_launch(g, &was);
    vgrid_set_launch(g, &was);
    show("set what get returned");
    set(4, 256, 2, 2, 0);
    show("4 and 2 lanes");
    set(was.lanes_per_ray, was.block, was.blocks_per_sm, was.fp64_lanes_per_ray, was.order);
    show("restored");
    set(was.lanes_per_ray, 256, 0, 4, was.order);
    show("float64 tuned");
    set(2, 256, 0, was.fp64_lanes_per_ray, was.order);
    show("float32 tuned");
    vgrid_set_launch(g, nullptr);
    show("reset");
    set(1, 128, 0, 1, -1);
    show("caller's order");
    set(1, 128, 8, 1, 0);
    show("one lane");
    vgrid_get_launch(g, &now);
    printf("%d %d\n", was.lanes_per_ray, now.blocks_per_sm);
    return 0;
}
"""


def test_launch_shape_read_and_set_again(tmp_path):
    """A call of few rays (64 of the 4096 resident ones) gets several lanes per
    ray: on a new grid, after its shape is read and set again or restored, and
    for the form whose lanes were left alone."""
    out = _run(tmp_path, SHAPES)
    auto = "8/128 8/128 8/32"
    assert out[:10] == ["new " + auto, "set what get returned " + auto, "4 and 2 lanes 4/256 4/256 2/256",
                        "restored " + auto, "float64 tuned 8/256 8/256 4/256", "float32 tuned 2/256 2/256 8/256",
                        "reset " + auto, "caller's order " + auto, "one lane 1/128 1/128 1/128", "1 8"]
