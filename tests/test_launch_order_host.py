"""Launch attributes and grids of the forward's small kernels, recorded on the host.

The launch helpers of the forward's small kernels are compiled with a recorder in the place of
cudaLaunchKernelEx and called without a GPU. Kernels of a forward read what was written before it (rows,
positions, the chain table) ahead of their own dependency wait, and every kernel lets the next one in at its
entry; so the first one, the embedding, must not be launched programmatically. The last test reads the source
for an order that no run can show.
"""
import os
import subprocess

import pytest

from paper_2512_14681_gb300 import build as B

PRELUDE = r"""
#include <cstdio>
#include <cuda_runtime.h>
struct Launch { int programmatic; dim3 grid; };
static Launch g_last;
static int g_launches;
template <typename... E, typename... A>
cudaError_t record_launch(const cudaLaunchConfig_t* c, void (*)(E...), A&&...) {
  g_last = {0, c->gridDim};
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization)
      g_last.programmatic = c->attrs[i].val.programmaticStreamSerializationAllowed;
  ++g_launches;
  return cudaSuccess;
}
#define cudaLaunchKernelEx record_launch
"""


def run_host(tmp_path, source, body):
    """Output lines of `body` (a main) compiled behind csrc/`source` and the recorder."""
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("needs nvcc")
    src = tmp_path / "host.cu"
    src.write_text(PRELUDE + f'#include "{os.path.join(B.CSRC, source)}"\n' + body)
    exe = tmp_path / "host"
    r = subprocess.run([nvcc, *B.ARCH, "-std=c++17", "-O0", "-Xcicc", "-O0", "-Xptxas", "-O0", "--expt-relaxed-constexpr",
                        "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"), str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return subprocess.run([str(exe)], capture_output=True, text=True, check=True, env=dict(os.environ, CUDA_VISIBLE_DEVICES="")).stdout.split()


def test_the_first_kernel_of_a_forward_is_a_full_boundary(tmp_path):
    out = run_host(tmp_path, "jf_elementwise.cu", r"""
int main() {
  for (int bf16 = 0; bf16 < 2; ++bf16) {
    g_launches = g_last.programmatic = 0;
    jf::launch_embed(nullptr, bf16, nullptr, nullptr, 4, 256, 512, nullptr, 0);
    std::printf("%d ", g_launches ? g_last.programmatic : 0);
    jf::launch_rmsnorm(nullptr, nullptr, nullptr, bf16, 4, 256, 1e-6f, nullptr, 0, 0);
    std::printf("%d ", g_last.programmatic);
  }
}
""")
    assert out == ["0", "1", "0", "1"]  # embedding, norm; fp32, bf16


def test_the_commit_grid_follows_what_one_sequence_commits(tmp_path):
    """16 sequences of 32 rows, 28 layers of 4 KV heads: 2,048 pieces of 16 bytes a sequence, two blocks; where
    prompts join in chunks of 64 rows, four. One sequence of 4 rows: one block."""
    out = run_host(tmp_path, "jf_decode.cu", r"""
int main() {
  jf::GenCfg g = {};
  const int cfg[3][4] = {{32, 0, 512, 16}, {32, 64, 512, 16}, {32, 0, 4, 1}};  // block, chunk, rows in flight, sequences
  for (auto& c : cfg) {
    g.n = c[0];
    g.prefill_chunk = c[1];
    jf::launch_commit(nullptr, c[3], jf::commit_rows(g, c[2]), 28, nullptr, nullptr, nullptr, nullptr, nullptr, 64, 64, 512, 4,
                      128, 2, nullptr, nullptr, 0);
    std::printf("%u,%u,%u ", g_last.grid.x, g_last.grid.y, g_last.grid.z);
  }
}
""")
    assert out == ["28,16,2", "28,16,4", "28,1,1"]


def test_copied_rows_are_ordered_before_the_arrival():
    """The attention's loaders: what 32 lanes copied is published by lane 0's arrival, so the lanes meet between."""
    text = open(os.path.join(B.CSRC, "jf_attention.cu")).read()
    text = text[text.index("JF_DEV bool load_steps("):]
    copied, arrival = text.index("cp_async_wait<0>();"), text.index("mbar_arrive_expect_tx(")
    fence = text.index("fence_proxy_async_smem();", copied)
    assert copied < fence < text.index("__syncwarp();", fence) < arrival
