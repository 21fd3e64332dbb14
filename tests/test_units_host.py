"""The float64 form's units (host, g++): dtrunc(x, by) is dtrunc of x 2^by, and
unit_shift leaves ordinary boxes alone and brings others near one."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_1854_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROG = r"""
#include "fsplit.h"
#include "internal.h"
#include <cstdio>
int main() {
    double x;
    int by;
    while (scanf("%la %d", &x, &by) == 2) {
        const float f = vg::dtrunc(x, by), g = vg::dtrunc(std::ldexp(x, by));
        uint32_t a, b;
        memcpy(&a, &f, 4);
        memcpy(&b, &g, 4);
        printf("%d %d\n", a == b, x > 0 ? vg::unit_shift(x) : 0);
    }
    return 0;
}
"""


def test_scaled_truncation(tmp_path):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include", "vector_types.h")):
        pytest.skip("needs g++ and the CUDA headers")
    (tmp_path / "t.cpp").write_text(PROG)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, "-I", os.path.join(CUDA, "include"),
                           str(tmp_path / "t.cpp"), "-o", exe])
    rng = np.random.default_rng(5)
    by = np.concatenate([np.repeat([-120, -61, -41, 21, 80, 120], 500), [-120, 120, 21, 0]])
    # x 2^by from below float32's range to its largest values
    x = rng.standard_normal(by.size) * 2.0 ** (rng.uniform(-160, 125, by.size) - by)
    x[-4:] = [0.0, -0.0, 5e-324, 2.0 ** -1060]
    lines = "\n".join(f"{float(v).hex()} {b}" for v, b in zip(x, by))
    out = np.array(subprocess.run([exe], input=lines, capture_output=True, text=True, check=True).stdout.split(), int)
    assert np.all(out[0::2] == 1)
    boxes = 2.0 ** np.arange(-125, 126) * 1.5
    out = np.array(subprocess.run([exe], input="\n".join(f"{float(v).hex()} 0" for v in boxes), capture_output=True,
                                  text=True, check=True).stdout.split(), int)[1::2]
    e = np.arange(-125, 126)
    assert np.array_equal(out, np.where((e >= -20) & (e <= 40), 0, -np.clip(e, -120, 120)))
