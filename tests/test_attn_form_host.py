"""The attention's launch rule (csrc/jf_attn_form.h), from rows and chains to CTAs per unit, on the host.

A unit (chain, KV head, tile of up to 128 query rows of whole tokens) runs on a cluster of 8, 4 or 2 CTAs or on
one. The cases are the 7B shape (4 KV heads, 7 query heads each: tiles of 126 rows) at the row and chain
counts of the window sweep, and the small model (2 KV heads, 4 query heads each: tiles of 128) at those of the
GPU tests that compare its forms. A GB300 holds 152 single CTAs, 76 pairs, 36 clusters of 4 and 15 of 8.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2512_14681_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "jf_attn_form.h"

#define CHECK(c) do { if (!(c)) { std::printf("FAIL line %d: %s\n", __LINE__, #c); return 1; } } while (0)

static int ctas(int M, int chains, int Hkv, int G) {
  const int tile = 128 / G * G, bound = Hkv * ((M * G + tile - 1) / tile + chains);
  const int mc[4] = {152, 76, 36, 15};
  return jf::attn_ctas_per_unit(jf::attn_units_estimate(M, chains, bound, Hkv, G, tile), mc);
}

int main() {
  // unit estimates: rows spread over the chains, whole tiles per chain and KV head
  CHECK(jf::attn_units_estimate(32, 1, 12, 4, 7, 126) == 8);      // 224 query rows: 2 tiles x 4 heads
  CHECK(jf::attn_units_estimate(64, 4, 32, 4, 7, 126) == 16);     // 4 windows of 16 rows: 1 tile each
  CHECK(jf::attn_units_estimate(128, 4, 44, 4, 7, 126) == 32);    // 4 windows of 32 rows: 2 tiles each
  CHECK(jf::attn_units_estimate(512, 4, 132, 4, 7, 126) == 128);  // 4 windows of 128 rows: 8 tiles each
  CHECK(jf::attn_units_estimate(512, 4, 100, 4, 7, 126) == 100);  // capped by the launch bound
  CHECK(jf::attn_units_estimate(5, 0, 8, 2, 4, 128) == 2);        // no chain count: one chain
  // no residency known: one cluster at a time
  const int none[4] = {0, 0, 0, 0};
  CHECK(jf::attn_ctas_per_unit(3, none) == 8);
  // the 7B shape: one wave of the widest clusters that fit
  CHECK(ctas(32, 1, 4, 7) == 8);    // 8 units
  CHECK(ctas(64, 1, 4, 7) == 4);    // 16
  CHECK(ctas(128, 1, 4, 7) == 4);   // 32
  CHECK(ctas(192, 1, 4, 7) == 2);   // 44
  CHECK(ctas(384, 1, 4, 7) == 1);   // 88
  CHECK(ctas(512, 1, 4, 7) == 1);   // 116
  CHECK(ctas(64, 4, 4, 7) == 4);    // four sequences: 16
  CHECK(ctas(128, 4, 4, 7) == 4);   // 32
  CHECK(ctas(512, 4, 4, 7) == 1);   // 128
  // the small model: 16 units of a 256-row window on clusters of 4, one row on clusters of 8; prefills of 64,
  // 300, 700 and 1,300 rows
  CHECK(ctas(256, 1, 2, 4) == 4);
  CHECK(ctas(1, 1, 2, 4) == 8);
  CHECK(ctas(64, 1, 2, 4) == 8);
  CHECK(ctas(300, 1, 2, 4) == 4);
  CHECK(ctas(700, 1, 2, 4) == 2);
  CHECK(ctas(1300, 1, 2, 4) == 1);
  std::printf("ok\n");
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_attention_form_rule(tmp_path):
    src = tmp_path / "form.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "form"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
