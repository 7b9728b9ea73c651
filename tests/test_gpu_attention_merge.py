"""Attention of row passes over many 128-key chunks: the merge of the chunks in batches of 16 and 32 (positions on both sides of
a batch's end), for head sizes with code of their own and one without, grouped queries, one row (chunks handed over by tags) and
several (grid barrier). Rows equal one-row passes bit for bit, and the one-row passes agree with the oracle."""
import numpy as np
import pytest

import oracle
import synth
from helpers import assert_logits_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("head_dim,heads,kv_heads,prompt_len", [(128, 2, 2, 2043), (64, 4, 2, 4091), (32, 4, 4, 2044), (16, 16, 8, 127)])
def test_rows_over_many_chunks(head_dim, heads, kv_heads, prompt_len):
    import paper_2410_01028_b200 as asd
    shape = synth.DecoderShape(n_layers=1, d_model=head_dim * heads, n_heads=heads, head_dim=head_dim, d_ffn=344, vocab=515, n_kv_heads=kv_heads)
    model = synth.make_model(shape, seed=head_dim, std=0.08)
    dec = asd.Decoder(shape, max_seq=prompt_len + 16, max_draft=8)
    dec.load_weights_host(model)
    dec.set_debug(True)
    orc = oracle.Oracle(model, max_seq=prompt_len + 16)
    prompt = synth.make_prompt(shape.vocab, prompt_len, seed=7)
    rows = [int(t) for t in synth.make_prompt(shape.vocab, 9, seed=8)]
    dec.prefill(prompt)
    orc.prefill(prompt)
    single = []
    for t in rows:
        dec.decode_step(t)
        orc.decode_step(t)
        single.append(dec.get_last_logits()[0].copy())
        assert_logits_close(single[-1][None], orc.last()["logits"])
    for M in (2, 5, 9):
        dec.reset()
        dec.prefill(prompt)
        dec.verify(rows[:M])
        np.testing.assert_array_equal(dec.get_last_logits(), np.stack(single[:M]), err_msg="M=%d" % M)
