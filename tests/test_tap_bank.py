"""The taps in a launch's parameters are read as 16-byte words, so their bank must
start 16-byte aligned whatever parameters come before it. Compiled for the host
from the library's own header; parameters are laid out like a struct's members."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = """
#include <cstdio>
#include <cstddef>
#include "emd_taps.cuh"
template <int N> struct Before { emd::Shape s; char more[N]; emd::TapBank bank; };
int main() {
  std::printf("%zu %d %zu %zu %zu %zu\\n", alignof(emd::TapBank), emd::kTapFloats % 4,
              offsetof(Before<4>, bank) % 16, offsetof(Before<8>, bank) % 16,
              offsetof(Before<12>, bank) % 16, offsetof(Before<16>, bank) % 16);
}
"""


def test_the_bank_is_16_byte_aligned_behind_any_parameters(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    src = tmp_path / "layout.cpp"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", cuda, "-I",
                    os.path.join(ROOT, "paper_2302_05804_gb300", "csrc"), str(src), "-o",
                    str(tmp_path / "layout")], check=True)
    out = subprocess.run([str(tmp_path / "layout")], check=True, capture_output=True, text=True)
    assert out.stdout.split() == ["16", "0", "0", "0", "0", "0"]
