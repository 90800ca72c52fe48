"""The fp32 kernels at the edges of their tiles, against the oracle.

Projection: 16- and 32-token tiles, the cluster's K shares (1, 2, 4, 8 CTAs), feature counts and K that
are no multiple of a tile or of four, and buffers that are not 16-byte aligned (4-byte copies). The
bound is the fp32 sum's: K * 2^-24 of the sum of absolute products, which it stays far below.
Attention: heads of 64 and of 128 dims; drafts that end inside a 32-key group, and that leave its four
warps one group each, fewer, or several.
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2512_14681_gb300 import inputs as I
from tests.parity import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,offset", [(1, 1, 1, 0), (128, 64, 16, 0), (300, 130, 17, 0), (257, 515, 33, 1),
                                          (2048, 256, 8, 0), (256, 1024, 5, 0), (256, 1028, 40, 1), (4096, 1024, 40, 0),
                                          (20000, 100, 65, 0)])
def test_gemm_f32_edges(N, K, M, offset):
    torch = need_gpu()
    from paper_2512_14681_gb300.jacobi import op_gemm

    W, X = I.random_array((N, K), seed=N + K, scale=0.5), I.random_array((M, K), seed=M, scale=0.5)

    def place(a):
        buf = torch.empty(a.size + offset, dtype=torch.float32, device="cuda")
        buf[offset:] = torch.from_numpy(a).cuda().reshape(-1)
        return buf[offset:].view(*a.shape)

    Y, err, _ = op_gemm(place(W), place(X))
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    ref = O.linear(X.astype(np.float64), W.astype(np.float64))
    bound = K * 2.0**-24 * (np.abs(X).astype(np.float64) @ np.abs(W).astype(np.float64).T)
    assert (np.abs(Y.cpu().numpy() - ref) <= bound + 1e-30).all()
    # a row's sums do not depend on the rows in flight
    one, _, _ = op_gemm(place(W), place(X[-1:].copy()))
    torch.cuda.synchronize()
    assert torch.equal(one[0], Y[-1])


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("prompt,rows", [(1, 1), (31, 2), (45, 20), (96, 32), (127, 2), (255, 9)])
def test_attention_f32_head_dims(head_dim, prompt, rows):
    need_gpu()
    from paper_2512_14681_gb300.jacobi import Context

    shape = dataclasses.replace(I.TINY_F32, name=f"tiny-f32-hd{head_dim}", head_dim=head_dim)
    toks = I.prompt_tokens(shape.vocab, prompt + rows, seed=head_dim + prompt)
    ctx = Context(shape, max_ctx=320, max_rows=64, logits_rows=32)
    try:
        ctx.init_random_weights(I.WEIGHT_SEED, I.WEIGHT_STD)
        ctx.prefill(0, toks[:prompt])
        logits, _, _ = ctx.forward_logits(0, toks[prompt:])
    finally:
        ctx.close()
    model = O.Model(O.ModelConfig(**shape.oracle_kwargs())).init_random(I.WEIGHT_SEED, I.WEIGHT_STD)
    n = prompt + rows
    ref = O.forward(model, O.Cache(model, 320, n), toks, np.arange(n), want_logits=True).logits[prompt:]
    assert np.abs(logits - ref).max() < 1e-4
