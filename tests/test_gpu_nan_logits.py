"""Rows whose logits hold no number (weights that overflowed) are reported, not decoded as token 0.

Infinite weights make every logit NaN. The argmax then is 0x7fffffff with -infinity for the best two
logits, prefill and the forward show it to the caller, a generation ends with JF_EDEVICE at the forward that
would read that token, and the context works again with finite weights.
"""
import math

import numpy as np
import pytest

from paper_2512_14681_gb300 import inputs as I
from tests.parity import need_gpu

pytestmark = pytest.mark.gpu

NO_TOKEN = 0x7FFFFFFF


@pytest.mark.parametrize("bf16", [False, True])
def test_rows_without_a_number_are_reported(bf16):
    need_gpu()
    from paper_2512_14681_gb300._lib import JF_BLOCK_RA, JF_EDEVICE, JfError
    from paper_2512_14681_gb300.jacobi import Context, Gen

    shape = I.SMALL_BF16 if bf16 else I.TINY_F32
    prompt = I.prompt_tokens(shape.vocab, 20, seed=5)
    ctx = Context(shape, max_ctx=128, max_rows=32, logits_rows=8)
    try:
        ctx.init_random_weights(0, math.inf)
        assert ctx.prefill(0, prompt) == NO_TOKEN
        logits, _, am = ctx.forward_logits(0, prompt[:5])
        assert np.isnan(logits).all() and (am == NO_TOKEN).all()
        out = ctx.jacobi_step(0, [(JF_BLOCK_RA, 20, 5, -1)], prompt[:5])
        assert (out["predictions"] == NO_TOKEN).all() and (out["top2"] == -np.inf).all()
        ctx.truncate(0, 0)
        with pytest.raises(JfError) as e:
            ctx.generate([prompt], Gen(block_size=4, max_new=8))
        assert e.value.status == JF_EDEVICE
        # reading the error cleared it
        ctx.init_random_weights(I.WEIGHT_SEED, I.WEIGHT_STD)
        ctx.truncate(0, 0)
        assert 0 <= ctx.prefill(0, prompt) < shape.vocab
    finally:
        ctx.close()
