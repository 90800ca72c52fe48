"""The attention's rule for how many CTAs share a unit (csrc/jf_attn_form.h), compiled for the host.

The cluster counts are a GB300's (152 single CTAs, 76 pairs, 36 clusters of 4, 15 of 8); the unit
counts are the 7B shape's at the points where the forms were timed against each other, and the edges
of each form's one-wave range.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_14681_gb300", "csrc")


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_ctas_per_unit(tmp_path):
    expect = {1: 8, 8: 8, 15: 8, 16: 4, 28: 4, 36: 4, 37: 2, 56: 2, 76: 2, 77: 1, 112: 1, 152: 1, 153: 2, 220: 2, 300: 1}
    src = tmp_path / "ctas.cpp"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "jf_attn_form.h"\nint main(int n, char** v) {\n'
                   "  const int mc[4] = {152, 76, 36, 15};\n"
                   '  for (int i = 1; i < n; ++i) std::printf("%d ", jf::attn_ctas_per_unit(std::atoi(v[i]), mc));\n}\n')
    exe = tmp_path / "ctas"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe), *map(str, expect)], capture_output=True, text=True, check=True).stdout.split()
    assert dict(zip(expect, map(int, out))) == expect
