"""The plans of the streamed and the FP32 products (host code, no GPU): splitting the
sources over SMs never takes more partial tiles than the bytes it is given, and an
FP32 plan keeps to the form it is allowed.  A small program linked with the library
prints the plans."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2312_09763_gb300")
SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include "zherk.h"
int main(int argc, char** argv) {
    const long long bytes = atoll(argv[1]);
    for (int i = 2; i + 2 < argc; i += 3) {
        const int N = atoi(argv[i]), n = atoi(argv[i + 1]);
        const double live = atof(argv[i + 2]);
        mv::ZherkPlan z;
        const bool ok = mv::zherk_plan(N, {}, 1, n, live, 152, 112ll << 20, bytes, z);
        const mv::Fp32Plan f = mv::herk_fp32_plan(N, 1, n, live, 152, true, bytes), r = mv::herk_fp32_plan(N, 1, n, live, 152, false, bytes);
        printf("%d %d %d %d %d %d %d %d\n", ok ? 1 : 0, z.S, (int)z.tiles.size(), f.split, (int)f.tiles.size(), f.form, r.form, r.rows);
    }
}
"""
CASES = [(9, 1, 25e3), (9, 256, 5e5), (12, 84, 35e3), (64, 200, 2e6), (128, 256, 2e6), (350, 19, 2e6), (350, 256, 5e4),
         (700, 256, 2e6), (1000, 256, 2e6), (1000, 1, 2e6), (1600, 7, 2e6)]


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    lib = os.path.join(PKG, "libmatvis_gb300.so")
    if not os.path.exists(nvcc) or not os.path.exists(lib):
        pytest.skip("needs nvcc and the built library")
    d = tmp_path_factory.mktemp("plans")
    src, exe = d / "plans.cu", d / "plans"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(PKG, "csrc"), str(src), lib, "-Xlinker", "-rpath=" + PKG, "-o", str(exe)], check=True)

    def run(split_bytes):
        args = [str(x) for c in CASES for x in c]
        out = subprocess.run([str(exe), str(split_bytes), *args], check=True, capture_output=True, text=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


@pytest.mark.parametrize("split_bytes", [0, 64 << 20, 1 << 30])
def test_split_sources_keep_to_their_bytes(plans, split_bytes):
    split = 0
    for (N, n, live), (ok, S, T, f_split, f_tiles, f_form, r_form, r_rows) in zip(CASES, plans(split_bytes), strict=True):
        tile = 128 * 128 * 4
        if ok:
            assert S == 1 or n * T * S * tile <= split_bytes, (N, n, live, S, T)
        assert f_split == 1 or f_tiles * f_split * tile <= split_bytes
        assert r_form == 0 and r_rows == 2 * N
        split += S > 1
    assert (split > 0) == (split_bytes > 0)
