"""The wait in front of the stage that finishes a pass's cosines, told to expect an arrival that never comes, runs out for every kind of
pass: in the producer warp (one row with tags) and in the consumer warps (all others). The call reports it, and after a reset the
context gives what it gave before."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,rows,tagged", [("decode", 1, True), ("decode", 1, False), ("verify", 2, True), ("verify", 3, True), ("verify", 5, True),
                                              ("verify", 9, True), ("prompt", 2, True), ("prompt", 16, True)])
def test_missing_arrival_ends_every_kind_of_pass(tiny_model, kind, rows, tagged):
    import paper_2410_01028_b200 as asd
    dec = asd.Decoder(synth.TINY, max_seq=128, max_draft=8)
    dec.load_weights_host(tiny_model)
    dec.set_prefill_mode(asd.PREFILL_ROWS)
    tokens = synth.make_prompt(synth.TINY.vocab, 24, seed=12)

    def run(**flags):
        dec.reset()
        dec.set_debug(no_tagged_handoff=not tagged)
        if kind != "prompt":
            dec.prefill(tokens[:7])
        dec.set_debug(no_tagged_handoff=not tagged, **flags)
        if kind == "decode":
            dec.decode_step(int(tokens[7]))
        elif kind == "verify":
            dec.verify(tokens[7:7 + rows])
        else:
            dec.prefill(tokens[:rows])
        return dec.get_last_logits()

    want = run()
    np.testing.assert_array_equal(run(short_waits=True), want)  # a short budget alone changes nothing
    with pytest.raises(asd.AsdError) as e:
        run(short_waits=True, missing_arrival=True)
    assert e.value.code == asd.binding.ERR_DEVICE_TIMEOUT
    assert "grid barrier" in str(e.value) and "stage" in str(e.value)
    np.testing.assert_array_equal(run(), want)
