"""widen4's integer widening of FP32 to FP64 (csrc/common.cuh): exact for
every value that it says it takes (host build, no GPU)."""
import os
import subprocess

import numpy as np
import pytest

from paper_2509_08109_gb300 import build

PROGRAM = r'''
#include <stdio.h>
#include "common.cuh"
int main() {
    unsigned u;
    while (fread(&u, 4, 1, stdin) == 1) {
        const unsigned out[3] = {bmg::plain_f32(u), bmg::widen_lo(u), bmg::widen_hi(u)};
        fwrite(out, 4, 3, stdout);
    }
}
'''


@pytest.fixture(scope="module")
def widen(tmp_path_factory):
    d = tmp_path_factory.mktemp("widen")
    src, exe = d / "widen.cu", d / "widen"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.SRC, "-I",
                    os.path.join(build.ROOT, "include"), str(src), "-o", str(exe)], check=True, capture_output=True)

    def run(bits):
        out = subprocess.run([str(exe)], input=bits.astype(np.uint32).tobytes(), capture_output=True, check=True)
        v = np.frombuffer(out.stdout, dtype=np.uint32).reshape(-1, 3)
        return v[:, 0] != 0, np.ascontiguousarray(v[:, 1:]).view(np.uint64).ravel()
    return run


def test_widening_is_exact(widen):
    edges = np.array([0, 1, 0x7fffff, 0x800000, 0x800001, 0x3f800000, 0x7f7fffff, 0x7f800000, 0x7f800001, 0x7fc00000,
                      0x7fffffff], dtype=np.uint32)
    bits = np.concatenate([edges, edges | 0x80000000,
                           np.random.default_rng(0).integers(0, 1 << 32, 200000, dtype=np.uint32)])
    plain, got = widen(bits)
    f = bits.view(np.float32)
    tiny = np.finfo(np.float32).tiny
    assert np.array_equal(plain, np.isfinite(f) & ((f == 0) | (np.abs(f) >= tiny)))
    assert np.array_equal(got[plain], f[plain].astype(np.float64).view(np.uint64))
