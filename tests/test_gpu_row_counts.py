"""The bf16 projections, the LM head's argmax and the norms at the row counts where their forms change.

Projection: 16-token tiles up to 16 rows, CTA pairs on tiles of 160 to 256 tokens above 160 rows (an
odd number of 128-feature tiles leaves a pair's second CTA without one), reductions that end inside a 128-k stage pair.
Inputs are bf16 values and the reference multiplies them in fp64, so the difference is the fp32 sum's:
K * 2^-23 of the sum of absolute products (one unit per addition, whichever way it rounds).
Argmax: in shared memory up to 512 rows, in the CTAs' global slots above; against the stored logits of the
same rows, bit for bit, and the lowest index when every logit is equal.
Hand-over of a call's inputs and results through pinned memory: prompts and steps that fill it.
Norm: 1024 threads a row up to 152 rows, 256 above, the same sums: a row's bits do not depend on the rows
beside it.
"""
import dataclasses

import numpy as np
import pytest

from paper_2512_14681_gb300 import inputs as I
from tests.parity import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 15, 16, 17, 161, 192, 193, 224, 225, 256, 257, 320, 321, 384, 385, 449])
@pytest.mark.parametrize("N,K,splits", [(1, 8, 0), (129, 64, 0), (384, 192, 0), (128, 72, 0), (640, 1096, 3), (257, 320, 5)])
def test_gemm_tile_edges(N, K, splits, M):
    torch = need_gpu()
    from paper_2512_14681_gb300.jacobi import op_gemm

    W = torch.from_numpy(I.random_array((N, K), seed=N + K, scale=0.5)).to(torch.bfloat16).cuda()
    X = torch.from_numpy(I.random_array((M, K), seed=M, scale=0.5)).to(torch.bfloat16).cuda()
    Y, err, _ = op_gemm(W, X, k_splits=splits)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    Wd, Xd = W.double().cpu().numpy(), X.double().cpu().numpy()
    bound = K * 2.0**-23 * (np.abs(Xd) @ np.abs(Wd).T)
    assert (np.abs(Y.cpu().numpy() - Xd @ Wd.T) <= bound + 1e-30).all()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("vocab", [2, 129, 1000, 8193])
def test_argmax_matches_the_stored_logits(bf16, vocab):
    need_gpu()
    from paper_2512_14681_gb300._lib import JF_BLOCK_RA
    from paper_2512_14681_gb300.jacobi import Context

    shape = dataclasses.replace(I.SMALL_BF16 if bf16 else I.TINY_F32, name=f"argmax-{vocab}", n_layers=1, vocab=vocab)
    ctx = Context(shape, max_ctx=768, max_rows=640, logits_rows=640)
    try:
        ctx.init_random_weights(I.WEIGHT_SEED, I.WEIGHT_STD)
        for n in (1, 16, 33, 161, 512, 513, 600):
            if ctx.seq_len(0):
                ctx.truncate(0, 0)
            ctx.prefill(0, I.prompt_tokens(vocab, 3, seed=1))
            draft = I.prompt_tokens(vocab, n, seed=n)
            logits, _, am = ctx.forward_logits(0, draft)
            assert np.array_equal(am, logits.argmax(1))
            if n <= 513:
                out = ctx.jacobi_step(0, [(JF_BLOCK_RA, 3, n, -1)], draft)
                assert np.array_equal(out["predictions"], am)
                assert np.array_equal(out["top2"], -np.sort(-logits, axis=1)[:, :2])
        ctx.init_random_weights(0, 0.0)  # every logit equal: the lowest index
        for n in (1, 33, 600):
            ctx.truncate(0, 3)
            assert not ctx.forward_logits(0, I.prompt_tokens(vocab, n, seed=n), want_logits=False)[2].any()
    finally:
        ctx.close()


@pytest.mark.parametrize("d,heads", [(512, 4), (4608, 8)])
def test_norm_rows_agree_bit_for_bit(d, heads):
    need_gpu()
    from paper_2512_14681_gb300.jacobi import Context

    shape = dataclasses.replace(I.SMALL_BF16, name=f"norm-{d}", d_model=d, n_heads=heads, vocab=512)
    toks = I.prompt_tokens(shape.vocab, 153, seed=d)
    ctx = Context(shape, max_ctx=256, max_rows=160)
    try:
        ctx.init_random_weights(I.WEIGHT_SEED, I.WEIGHT_STD)
        rows = {n: ctx.forward_logits(0, toks[:n], want_logits=False)[1] for n in (1, 152, 153)}
    finally:
        ctx.close()
    assert np.array_equal(rows[152], rows[153][:152])
    assert np.array_equal(rows[1], rows[153][:1])


@pytest.mark.parametrize("bf16", [False, True])
def test_calls_that_fill_the_staging_memory(bf16):
    need_gpu()
    from paper_2512_14681_gb300._lib import JF_BLOCK_CAND, JF_BLOCK_RA
    from paper_2512_14681_gb300.jacobi import Context

    shape = I.SMALL_BF16 if bf16 else I.TINY_F32
    toks = I.prompt_tokens(shape.vocab, 64, seed=3)
    got = []
    for rows in (64, 7):  # one forward, or ten with a last one of one row
        ctx = Context(shape, max_ctx=64, max_rows=rows)
        try:
            ctx.init_random_weights(I.WEIGHT_SEED, I.WEIGHT_STD)
            q0 = ctx.prefill(0, toks)  # the whole context
            ctx.truncate(0, 57)
            draft = toks[57:]
            _, hidden, am = ctx.forward_logits(0, draft, want_logits=False)
            blocks = [(JF_BLOCK_RA, 57, 3, -1), (JF_BLOCK_CAND, 57, 4, -1)]
            out = ctx.jacobi_step(0, blocks, np.concatenate([draft[:3], draft[:4]]))
            assert np.array_equal(out["predictions"], np.concatenate([am[:3], am[:4]]))
            got.append((q0, hidden, am, out["counts"], out["committed"], out["top2"]))
        finally:
            ctx.close()
    assert got[0][0] == got[1][0] == got[0][2][-1]
    for a, b in zip(got[0][1:], got[1][1:]):
        assert np.array_equal(a, b)
