"""Results that a pass itself leaves in pinned host memory: recorded logits up to 256 KB (beyond, they are copied when asked for) and the
similarity sums. Row m of a verify pass is the same whatever the number of rows, so both ways have to give the same bits."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab,m_host,m_copy", [(16384, 4, 5), (9362, 7, 8), (16381, 1, 9)])
def test_logits_on_both_sides_of_the_limit(vocab, m_host, m_copy):
    import paper_2410_01028_b200 as asd
    assert m_host * vocab * 4 <= 256 * 1024 < m_copy * vocab * 4
    shape = synth.DecoderShape(n_layers=2, d_model=256, n_heads=4, head_dim=64, d_ffn=344, vocab=vocab)
    dec = asd.Decoder(shape, max_seq=128, max_draft=8)
    dec.load_weights_host(synth.make_model(shape, seed=3, std=0.08))
    dec.set_debug(True)
    prompt = synth.make_prompt(vocab, 40, seed=4)  # the dense prompt path; its LM head leaves one row
    rows = [int(t) for t in synth.make_prompt(vocab, 9, seed=5)]

    def logits(m):
        dec.reset()
        dec.prefill(prompt)
        first = dec.get_last_logits()
        dec.verify(rows[:m])
        got = dec.get_last_logits()
        assert got.shape == (m, vocab)
        np.testing.assert_array_equal(dec.get_last_logits(), got)  # asked for twice
        return first, got

    first_a, a = logits(m_host)
    first_b, b = logits(m_copy)
    np.testing.assert_array_equal(first_a, first_b)
    n = min(m_host, m_copy)
    np.testing.assert_array_equal(a[:n], b[:n])
    assert not np.array_equal(a[0], first_a[0])


@pytest.mark.parametrize("prompt_len", [5, 21, 90])
def test_similarity_is_the_mean_of_the_reported_rows(prompt_len):
    import paper_2410_01028_b200 as asd
    shape = synth.DecoderShape(n_layers=3, d_model=256, n_heads=4, head_dim=64, d_ffn=344, vocab=515)
    dec = asd.Decoder(shape, max_seq=256, max_draft=8)
    dec.load_weights_host(synth.make_model(shape, seed=6, std=0.08))
    tokens = synth.make_prompt(515, prompt_len, seed=7)
    sums = np.zeros((2, 3))
    for i, t in enumerate(tokens):  # one row at a time, its cosines read back
        dec.prefill(np.array([t], np.int32))
        ca, cm = dec.get_last_cosines()
        sums += np.stack([ca[:, 0], cm[:, 0]])
        if i in (0, 3):
            np.testing.assert_allclose(np.stack(dec.get_similarity()[:2]), sums / (i + 1), rtol=1e-6)
    np.testing.assert_allclose(np.stack(dec.get_similarity()[:2]), sums / prompt_len, rtol=1e-6)
    dec.reset()
    dec.prefill(tokens)  # all at once: 16-row passes or dense products, other orders of the same sums
    np.testing.assert_allclose(np.stack(dec.get_similarity()[:2]), sums / prompt_len, atol=1e-3)
