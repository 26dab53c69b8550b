"""Host rules of the Legendre dispatch, called in the built library from a
small C++ program (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1308_5299_gb300")


def run(tmp_path, body):
    import __graft_entry__

    __graft_entry__.build()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text('#include "kernels.h"\n#include <cstdio>\nusing namespace cr;\nint main() {\n%s\n}\n' % body)
    subprocess.run(["g++", "-std=c++17", "-I" + os.path.join(PKG, "csrc"), "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(cuda, "include"), str(src), "-o", str(exe), "-L" + PKG, "-l:libcrgb300.so",
                    "-Wl,-rpath," + PKG, "-L" + os.path.join(cuda, "lib64"), "-lcudart",
                    "-Wl,-rpath," + os.path.join(cuda, "lib64")], check=True, capture_output=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()


@pytest.mark.parametrize("pairs,lmax,df,expect", [(64, 64, 0, 1), (63, 64, 0, 0), (64, 63, 0, 0), (64, 64, 1, 0)])
def test_digit_slices_by_the_grid_whatever_the_mask(tmp_path, pairs, lmax, df, expect):
    """A mask that leaves few ring pairs changes how many take part, not the
    kernels they run on."""
    out = run(tmp_path, """
  DsTab t;
  LegArgs<double> a;
  a.ds = &t;
  a.df = %d;
  a.L = %d;
  a.nring = %d;
  for (int n : {%d, 55, 1}) {
    a.npairs = n;
    std::printf("%%d\\n", (int)ds_use(a));
  }""" % (df, lmax, 2 * pairs - 1, pairs))
    assert out == [str(expect)] * 3
