"""The FFT buffer's parts hold what its kernels put there, on devices with any
number of SMs: a shape may take the split launch alone (one slot per SM) and
exposure groups in a batch (one slot per tile and group). Compiled for the host
against the library."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2302_05804_gb300")

SOURCE = """
#include <cstdio>
#include <cstdlib>
#include "emd_fft.cuh"
int main(int, char** v) {
  emd::Shape s;
  const char* why = "";
  if (!emd::make_shape(atoi(v[1]), atoi(v[2]), atoi(v[3]), atoi(v[4]), 1, &s, &why)) return 1;
  const emd::FftLayout L = emd::fft_layout(s, atoi(v[6]) != 0, atoi(v[5]));
  std::printf("%d %d %zu %zu\\n", emd::fft_tiles_total(s), emd::fft_groups(s),
              L.counters - L.partials, L.total - L.counters);
}
"""


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    from paper_2302_05804_gb300 import build
    lib = build.build()
    d = tmp_path_factory.mktemp("layout")
    (d / "layout.cpp").write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", cuda, "-I",
                    os.path.join(PKG, "csrc"), str(d / "layout.cpp"), lib,
                    "-Wl,-rpath," + os.path.dirname(lib), "-o", str(d / "layout")], check=True)

    def run(*a):
        out = subprocess.run([str(d / "layout"), *map(str, a)], check=True, capture_output=True,
                             text=True)
        return [int(x) for x in out.stdout.split()]
    return run


@pytest.mark.parametrize("sms", [0, 18, 40, 76, 132, 152])
@pytest.mark.parametrize("student", [0, 1])
def test_partials_hold_groups_and_split_slots(layout, sms, student):
    for H, W, n, K in ((200, 150, 9, 21), (500, 430, 24, 31), (900, 640, 17, 43),
                       (1100, 900, 40, 43), (2048, 2048, 33, 43)):
        tiles, groups, partials, counters = layout(H, W, n, K, sms, student)
        slot = (2 * 64 * 128 if student else 64 * 128 + 128) * 8
        if groups > 1:  # emd_batch_step, and emd_iterate below one tile per SM
            assert partials >= tiles * groups * slot
        if sms and tiles >= sms and not student:  # the split launch
            assert partials >= sms * slot
        if groups > 1 or (sms and tiles >= sms and not student):
            assert counters >= tiles * 4
