"""Row classes that the row kernels know (csrc/layout_types.h), on the CPU.

The kernels leave out rows of a width they have no code for, so lp_create refuses
such a layout.  A layout without widening has none; one with it (rows of 2 and 8
lanes) is refused.
"""
import os
import shutil
import subprocess

import pytest

from tests.conftest import ROOT

SOURCE = r'''
#include <cstdio>
#include "layout_types.h"
using namespace lpop;
int main() {
  for (int widen = 1; widen <= 8; widen *= 2) {
    int bad = 0;
    for (long long len = 0; len <= 5000; ++len) {
      BinTable t{};
      t.nbins = 1;
      const int w = width_for_length(len, widen);
      t.bin[0].width = w == 1 ? kSell : w;  // (one lane: the sliced copy)
      bad += !check_row_classes(t);
    }
    std::printf("%d ", bad);
  }
}
'''


def test_classes_of_a_layout_are_those_of_the_kernels(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    src, exe = tmp_path / "classes.cpp", str(tmp_path / "classes")
    src.write_text(SOURCE)
    subprocess.run([gxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2506_17650_gb300", "csrc"), str(src), "-o", exe],
                   check=True)
    plain, *widened = (int(x) for x in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert plain == 0 and widened[0] > 0 and widened[2] > 0
