"""jf_op_gemm and jf_op_gemm_noalloc start after the work ahead of them on the stream is complete.

W may be what the kernel just before wrote, and the bf16 kernel requests its first weight tiles before its
dependency wait, so the public calls must not be launched programmatically. Two calls are captured (nothing
runs) and the captured graph's edges are looked at: none may be a programmatic one.
"""
import ctypes as C

import pytest

from tests.parity import need_gpu

pytestmark = pytest.mark.gpu


class EdgeData(C.Structure):  # CUgraphEdgeData
    _fields_ = [("from_port", C.c_ubyte), ("to_port", C.c_ubyte), ("type", C.c_ubyte), ("reserved", C.c_ubyte * 5)]


def _captured_edges(stream, calls):
    """Types of the edges of the graph that `calls` leave on `stream`."""
    cuda = C.CDLL("libcuda.so.1")
    st, graph, n = C.c_void_p(stream), C.c_void_p(), C.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(st, 1) == 0  # thread-local
    calls()
    assert cuda.cuStreamEndCapture(st, C.byref(graph)) == 0
    try:
        assert cuda.cuGraphGetEdges_v2(graph, None, None, None, C.byref(n)) == 0
        a, b, data = (C.c_void_p * n.value)(), (C.c_void_p * n.value)(), (EdgeData * n.value)()
        assert cuda.cuGraphGetEdges_v2(graph, a, b, data, C.byref(n)) == 0
        return [d.type for d in data]
    finally:
        cuda.cuGraphDestroy(graph)


@pytest.mark.parametrize("M", [32, 200])  # one CTA a tile; pairs
@pytest.mark.parametrize("noalloc", [False, True])
def test_calls_are_full_boundaries(noalloc, M):
    torch = need_gpu()
    from paper_2512_14681_gb300 import _lib as J

    lib, N, K = J.load(), 256, 512
    W, X = (torch.randn(r, K, device="cuda").bfloat16() for r in (N, M))
    Y = torch.empty(M, N, device="cuda")
    ws, err = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    st = torch.cuda.Stream()

    def call():
        p = [t.data_ptr() for t in (W, X, Y)] + [N, K, M, 1]
        if noalloc:
            assert lib.jf_op_gemm_noalloc(*p, err.data_ptr(), st.cuda_stream) == J.JF_OK
        else:
            assert lib.jf_op_gemm(J.JF_BF16, *p, ws.data_ptr(), ws.numel(), err.data_ptr(), st.cuda_stream) == J.JF_OK

    st.wait_stream(torch.cuda.current_stream())
    call()  # sets the kernels up
    torch.cuda.synchronize()
    types = _captured_edges(st.cuda_stream, lambda: (call(), call()))
    assert types and not any(types)
