"""Which form of the FP32 direct iteration a shape runs: the library's rule, compiled
for the host, against the bench's restatement of it, and on shapes where the split
form is slower than the halo-exchange kernel (100 tiles of 64 x 128 and more without
a launch of 500 items)."""
import os
import shutil
import subprocess

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2302_05804_gb300")

SOURCE = """
#include <cstdio>
#include <cstdlib>
#include "emd_taps.cuh"
int main(int, char** v) {
  emd::Shape s;
  const char* why = "";
  if (!emd::make_shape(atoi(v[1]), atoi(v[2]), atoi(v[3]), atoi(v[4]), atoi(v[5]), &s, &why))
    return 1;
  for (int student = 0; student < 2; ++student) {
    const emd::DirectPlan p = emd::direct_plan(s, student != 0);
    std::printf("%d %d %d ", p.form, p.chunk, p.parts);
  }
}
"""

HALO, TAPS, SPLIT = 0, 1, 2


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_2302_05804_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", cuda, "-I",
                    os.path.join(PKG, "csrc"), str(d / "plan.cpp"), lib,
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(d / "plan")], check=True)

    def run(*shape):
        out = subprocess.run([str(d / "plan"), *map(str, shape)], check=True,
                             capture_output=True, text=True)
        return [int(x) for x in out.stdout.split()]
    return run


@pytest.mark.parametrize("shape,form", [
    ((900, 1000, 10, 43, 1), HALO), ((1100, 1150, 20, 47, 1), HALO),
    ((1000, 1000, 31, 47, 8), HALO), ((1000, 1000, 31, 85, 4), HALO),
    ((900, 900, 12, 93, 2), HALO), ((2047, 2040, 2, 3, 1), HALO),
    ((700, 700, 24, 43, 1), SPLIT), ((128, 128, 4, 15, 1), SPLIT), ((1200, 1200, 12, 3, 1), SPLIT),
    ((512, 512, 100, 15, 4), SPLIT), ((1021, 1009, 33, 43, 1), TAPS), ((4096, 4096, 33, 43, 1), TAPS),
    ((2048, 2048, 33, 85, 2), TAPS), ((1000, 1010, 17, 15, 1), TAPS)])
def test_form_of_a_shape(plan, shape, form):
    got = plan(*shape)
    assert got[0] == form and got[3] == form
    n = shape[2]
    for nu in (0.0, 3.0):
        _, chunk, parts = got[:3] if nu == 0 else got[3:]
        names, launches = bench.direct_form(*shape, nu, None)
        if form == TAPS:
            assert names.startswith("taps_forward_kernel")
            assert ("taps_sum_kernel" in names) == bool(parts)
            assert launches == -(-n // chunk) * (3 if parts else 2)
        else:
            assert (names, launches) == (("halo_kernel", "split_kernel")[form == SPLIT], 1)
