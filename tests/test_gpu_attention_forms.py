"""Every form of the bf16 attention gives a row the same bits.

A unit's 8 key lanes run on a cluster of 8, 4 or 2 CTAs or on one CTA, by the number of units of the
forward. A prompt prefilled in one forward of 300, 700 or 1,300 rows (18, 44 and 82 units on the small
model: clusters of 4, of 2 and single CTAs) must leave the K/V that 64-row forwards (4 units, clusters
of 8) leave, so that the rows after it come out bit for bit the same. The committed lengths put the
page of the last cached and first in-flight key, and the partly filled last page, at every kind of
offset.
"""
import numpy as np
import pytest

from paper_2512_14681_gb300 import inputs as I
from tests.parity import need_gpu

pytestmark = pytest.mark.gpu


def _rows_after(max_rows, lengths, prompt, draft):
    from paper_2512_14681_gb300.jacobi import Context

    ctx = Context(I.SMALL_BF16, max_ctx=len(prompt) + 64, max_rows=max_rows)
    try:
        ctx.init_random_weights(I.WEIGHT_SEED, I.WEIGHT_STD)
        at = 0
        for n in lengths:
            ctx.prefill(0, prompt[at:at + n])
            at += n
        return ctx.forward_logits(0, draft, want_logits=False)[1]
    finally:
        ctx.close()


@pytest.mark.parametrize("rows", [300, 700, 1300])
@pytest.mark.parametrize("start", [0, 1, 16, 37, 1023])
def test_forms_agree_bit_for_bit(rows, start):
    need_gpu()
    prompt = I.prompt_tokens(I.SMALL_BF16.vocab, start + rows, seed=rows + start)
    draft = I.prompt_tokens(I.SMALL_BF16.vocab, 5, seed=7)
    head = [start] if start else []
    wide = _rows_after(max(rows, start), head + [rows], prompt, draft)
    narrow = _rows_after(64, head + [rows], prompt, draft)
    assert np.array_equal(wide, narrow)
