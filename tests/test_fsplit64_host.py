"""Host checks of the integer conversions of the float64 traversal
(csrc/fsplit.h), compiled with g++ from the source the device compiles:
dtrunc cuts a float64 value to float32 towards zero, fexact widens a float32
value exactly."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1310_1854_gb300", "csrc")

PROG = r"""
#include "fsplit.h"
#include <cstdio>
int main() {
    unsigned long long b;
    while (scanf("%llx", &b) == 1) {
        double x;
        memcpy(&x, &b, 8);
        const float f = vg::dtrunc(x);
        uint32_t fb, g = (uint32_t)b;
        memcpy(&fb, &f, 4);
        float y;
        memcpy(&y, &g, 4);
        printf("%08x %016llx\n", fb, (unsigned long long)vg::dbits(vg::fexact(y)));
    }
    return 0;
}
"""


def test_conversions(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    (tmp_path / "t.cpp").write_text(PROG)
    exe = str(tmp_path / "t")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe])
    rng = np.random.default_rng(3)
    x = np.concatenate([
        rng.standard_normal(2000) * 10.0 ** rng.uniform(-60, 60, 2000),
        [0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, 2.0 ** -126, -(2.0 ** -126), np.nextafter(2.0 ** -126, 0.0), 2.0 ** -149,
         5e-324, 2.0 ** 127, np.nextafter(2.0 ** 128, 0.0), -(2.0 ** 128), 1.0 + 2.0 ** -24, 1e300]])
    low = rng.integers(0, 1 << 32, x.size, dtype=np.uint64)
    special = np.array([0, 1 << 31, 1, 0x7fffff, 0x800000, 0x807fffff, 0x7f7fffff, 0x7f800000, 0xff800000], np.uint64)
    bits = np.concatenate([x.view(np.uint64), (x.view(np.uint64) >> np.uint64(32) << np.uint64(32)) | low, special])
    out = subprocess.run([exe], input="\n".join(f"{int(b):x}" for b in bits), capture_output=True, text=True,
                         check=True).stdout.split()
    f = np.array([int(v, 16) for v in out[0::2]], np.uint32).view(np.float32)
    d = np.array([int(v, 16) for v in out[1::2]], np.uint64).view(np.float64)
    v = bits.view(np.float64)
    y = (bits & np.uint64(0xffffffff)).astype(np.uint32).view(np.float32)
    ok = ~np.isnan(y)
    assert np.array_equal(d[ok].view(np.uint64), y[ok].astype(np.float64).view(np.uint64))
    small = np.abs(v) < 2.0 ** -126
    assert np.all(f[small] == 0.0)
    fit = ~small & (np.abs(v) < 2.0 ** 128)
    e = v[fit] - f[fit].astype(np.float64)
    assert np.all(np.abs(e) < 2.0 ** -23 * np.abs(v[fit])) and np.all(np.abs(f[fit].astype(np.float64)) <= np.abs(v[fit]))
    with np.errstate(over="ignore"):
        assert np.array_equal(f[np.abs(v) >= 2.0 ** 128], v[np.abs(v) >= 2.0 ** 128].astype(np.float32))
