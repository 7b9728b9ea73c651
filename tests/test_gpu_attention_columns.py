"""Attention of row passes in steps of eight columns, a column being a (row, query head of the group) pair: groups of 1 to 12 heads and 1 to
9 rows on both sides of a step's end, one or two columns (the terms of P share a product), key counts around a block of 16 and a chunk
of 128. Rows equal one-row passes bit for bit, and the one-row passes and the 16-row passes of the prompt agree with the oracle."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_logits_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,heads,kv_heads,prompt_len", [(128, 2, 2, 15), (128, 4, 2, 127), (64, 8, 2, 112), (64, 3, 1, 129), (256, 2, 1, 30), (256, 2, 2, 247),
                                                              (32, 10, 2, 128), (16, 24, 2, 31)])
def test_rows_and_heads_share_steps(head_dim, heads, kv_heads, prompt_len):
    import paper_2410_01028_b200 as asd
    shape = synth.DecoderShape(n_layers=2, d_model=head_dim * heads, n_heads=heads, head_dim=head_dim, d_ffn=344, vocab=515, n_kv_heads=kv_heads)
    model = synth.make_model(shape, seed=head_dim + heads, std=0.08)
    dec = asd.Decoder(shape, max_seq=prompt_len + 16, max_draft=8)
    dec.load_weights_host(model)
    dec.set_debug(True)
    dec.set_prefill_mode(asd.PREFILL_ROWS)
    orc = oracle.Oracle(model, max_seq=prompt_len + 16)
    prompt = synth.make_prompt(shape.vocab, prompt_len, seed=17)
    rows = [int(t) for t in synth.make_prompt(shape.vocab, 9, seed=18)]
    dec.prefill(prompt)
    orc.prefill(prompt)
    single = []
    for t in rows:
        dec.decode_step(t)
        orc.decode_step(t)
        single.append(dec.get_last_logits()[0].copy())
        assert_logits_close(single[-1][None], orc.last()["logits"])
    for M in (2, 3, 4, 5, 8, 9):
        dec.reset()
        dec.prefill(prompt)
        dec.verify(rows[:M])
        np.testing.assert_array_equal(dec.get_last_logits(), np.stack(single[:M]), err_msg="M=%d" % M)
