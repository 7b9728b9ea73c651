"""The timeline of a pass: every CTA enters a stage, finds its inputs ready and leaves it, in this order, and enters no stage before it
has left the one in front; for every kind of pass, stages without anything to wait for among them."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,tagged", [(1, True), (1, False), (2, True), (5, True), (16, True)])
def test_stages_of_every_cta_follow_one_another(tiny_model, rows, tagged):
    import paper_2410_01028_b200 as asd
    dec = asd.Decoder(synth.TINY, max_seq=64, max_draft=8)
    dec.load_weights_host(tiny_model)
    dec.set_prefill_mode(asd.PREFILL_ROWS)
    tokens = synth.make_prompt(synth.TINY.vocab, 16, seed=13)
    dec.set_debug(record_logits=False, trace=True, no_tagged_handoff=not tagged)
    for _ in range(2):  # the second pass must not show what the first one left
        if rows == 16:
            dec.prefill(tokens)
        else:
            dec.reset()
            dec.prefill(tokens[:3])
            dec.verify(tokens[:rows]) if rows > 1 else dec.decode_step(int(tokens[0]))
        t = dec.get_last_trace()
        entered, ready, left = t[:, 0], t[:, 1], t[:, 3]
        assert len(t) == 3 + 5 * synth.TINY.n_layers  # embedding, five a layer, finish, LM head
        assert (entered > 0).all() and (entered <= ready).all() and (ready <= left).all(), np.argwhere((entered > ready) | (ready > left))
        assert (left[:-1] <= entered[1:]).all()
