"""jf_op_gemm and jf_op_gemm_noalloc read what the kernel just before them on the stream writes.

The kernel ahead lets its successor start at its entry, waits a while and then writes W and X (all ones over
zeros). The GEMM kernels may start early, but must wait for it before they request a tile of W: every element
of Y is K.
"""
import ctypes as C
import subprocess

import pytest

from paper_2512_14681_gb300 import build as B
from tests.parity import need_gpu

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cuda_runtime.h>
template <typename T>
__global__ void k_late(T* w, T* x, long long nw, long long nx, T one, unsigned long long delay_ns) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (int i = 0; i < 1000000; ++i) {  // the timer's limit, or this many rounds
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > delay_ns) break;
  }
  for (long long i = threadIdx.x; i < nw; i += blockDim.x) w[i] = one;
  for (long long i = threadIdx.x; i < nx; i += blockDim.x) x[i] = one;
}
extern "C" int late(void* w, void* x, long long nw, long long nx, int bf16, unsigned long long delay_ns, void* st) {
  if (bf16) k_late<<<1, 1024, 0, (cudaStream_t)st>>>((unsigned short*)w, (unsigned short*)x, nw, nx, (unsigned short)0x3f80, delay_ns);
  else k_late<<<1, 1024, 0, (cudaStream_t)st>>>((float*)w, (float*)x, nw, nx, 1.0f, delay_ns);
  return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def late(tmp_path_factory):
    need_gpu()
    d = tmp_path_factory.mktemp("late")
    (d / "late.cu").write_text(PROGRAM)
    r = subprocess.run([B.nvcc(), *B.ARCH, "-shared", "-Xcompiler", "-fPIC", str(d / "late.cu"), "-o", str(d / "late.so")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    fn = C.CDLL(str(d / "late.so")).late
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_longlong, C.c_longlong, C.c_int, C.c_ulonglong, C.c_void_p]
    return fn


@pytest.mark.parametrize("M,splits", [(32, 1), (32, 4), (200, 2)])  # one CTA a tile, split, pairs
@pytest.mark.parametrize("call", ["bf16", "noalloc", "f32"])
def test_a_call_waits_for_the_kernel_that_writes_its_inputs(late, call, M, splits):
    import torch

    from paper_2512_14681_gb300 import _lib as J

    lib, N, K = J.load(), 300, 2048
    dt = torch.float32 if call == "f32" else torch.bfloat16
    W, X = torch.zeros(N, K, device="cuda", dtype=dt), torch.zeros(M, K, device="cuda", dtype=dt)
    Y = torch.empty(M, N, device="cuda")
    ws, err = torch.zeros(4 << 20, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()

    def gemm():
        p = [t.data_ptr() for t in (W, X, Y)] + [N, K, M, splits]
        if call == "noalloc":
            return lib.jf_op_gemm_noalloc(*p, err.data_ptr(), st.cuda_stream)
        return lib.jf_op_gemm(J.JF_F32 if call == "f32" else J.JF_BF16, *p, ws.data_ptr(), ws.numel(), err.data_ptr(),
                              st.cuda_stream)

    torch.cuda.synchronize()
    assert gemm() == J.JF_OK  # sets the kernels up
    torch.cuda.synchronize()
    assert not Y.any()
    assert late(W.data_ptr(), X.data_ptr(), W.numel(), X.numel(), call != "f32", 200_000, st.cuda_stream) == 0
    assert gemm() == J.JF_OK
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert (Y == K).all()
