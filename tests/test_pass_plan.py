"""The shared-memory plan of a pass (no GPU needed): scratch is set aside for the groups of attention warps that the ring feeds, and a decoder
is refused only where one group and the shortest window leave the ring too few slots."""
import collections
import ctypes
import functools
import os
import random
import subprocess
import tempfile

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_01028_b200", "csrc")
SMS, SMEM = 148, 232448
Plan = collections.namedtuple("Plan", "ns groups xs psum reg_a smem scratch")


@functools.lru_cache(None)
def _lib():
    with tempfile.TemporaryDirectory() as tmp:
        src, lib = os.path.join(tmp, "plan.cpp"), os.path.join(tmp, "plan.so")
        with open(src, "w") as f:
            f.write('#include "pass_plan.h"\nextern "C" int plan(int sms, int smem, const asd_config* c, int M, int* o) {\n'
                    "    asd::PassPlan p{};\n    const bool ok = asd::plan_pass(sms, smem, *c, M, &p);\n"
                    "    o[0] = p.ns, o[1] = p.attn_groups, o[2] = p.xs_bytes, o[3] = p.off_reg_a - p.off_psum, o[4] = (int)p.smem - 1024 - p.off_reg_a, o[5] = (int)p.smem;\n"
                    "    o[6] = asd::attn_scratch_bytes(M, c->n_heads / c->n_kv_heads, c->head_dim);\n    return ok;\n}\n")
        subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
        return ctypes.CDLL(lib)


def _plan(head_dim, heads, kv_heads, d_ffn, vocab, M):
    from paper_2410_01028_b200.binding import Config
    cfg = Config(n_layers=2, d_model=heads * head_dim, n_heads=heads, n_kv_heads=kv_heads, head_dim=head_dim, d_ffn=d_ffn, vocab=vocab, max_seq=1024)
    out = (ctypes.c_int * 7)()
    ok = _lib().plan(SMS, SMEM, ctypes.byref(cfg), M, out)
    return (Plan(*out) if ok else None), out[6]


@pytest.mark.parametrize("vocab", [128256, 141500, 151936, 161000])
@pytest.mark.parametrize("M", [1, 5, 9, 16])
def test_large_vocabularies_at_head_size_256(vocab, M):
    plan, _ = _plan(256, 8, 1, 16384, vocab, M)
    assert plan is not None and plan.ns >= 16 and plan.groups == 1


def test_groups_have_scratch_and_slots_and_nothing_fits_that_is_refused():
    rng, seen, refused = random.Random(4), collections.Counter(), 0
    for _ in range(20000):
        hd, kv = rng.choice([16, 32, 64, 128, 256]), rng.choice([1, 2, 4, 8, rng.randint(1, 40)])
        heads = kv * rng.choice([1, 1, 2, 4, 8, rng.randint(1, 12)])
        if heads * hd > 16384:
            continue
        d_ffn, vocab, M = 8 * int(2 ** rng.uniform(3, 13)), int(2 ** rng.uniform(5, 18.7)), rng.choice([1, 2, 5, 9, 16])
        tile_slots, least = 2 * max(1, hd // 64), max(8, 4 * max(1, hd // 64))  # slots of a K (or V) tile; the shortest ring
        plan, scratch = _plan(hd, heads, kv, d_ffn, vocab, M)
        if plan is None:
            refused += 1
            pairs = (max(vocab, 2 * d_ffn, (heads + 2 * kv) * hd) + 1) // 2
            psum = max(-(-pairs // SMS) + 2, 120) * 2 * M * 4
            if pairs * SMS < 1 << 31:
                # 1 KB of alignment, 4 to 6 KB of barriers and reduction scratch, a window of one segment of 256 inputs
                assert SMEM - 1024 - 4096 - psum - max(scratch, M * (256 + 32) * 2) < least * 8192 + 2048, (hd, heads, kv, d_ffn, vocab, M)
            continue
        seen[plan.groups] += 1
        assert plan.smem <= SMEM and plan.ns >= least and plan.ns <= 48
        assert plan.groups == 1 or (plan.ns >= plan.groups * 2 * tile_slots and plan.groups * scratch <= 40960)
        assert plan.reg_a >= plan.groups * scratch and plan.reg_a >= min(plan.xs, M * (256 + 32) * 2)
        if plan.groups < 3 and (plan.groups + 1) * scratch <= 40960:  # the next group's scratch would leave it no tiles
            more = max(0, (plan.groups + 1) * scratch - plan.reg_a)
            assert plan.ns + (SMEM - plan.smem - more) // 8192 < (plan.groups + 1) * 2 * tile_slots
    assert all(seen[g] > 100 for g in (1, 2, 3)) and refused > 50


@pytest.mark.gpu
def test_decoder_of_head_size_256_with_a_large_vocabulary():
    """Row passes of 16, 9 and one row with their plans' rings; the prompt's last row and a decode step against the oracle."""
    import oracle
    import paper_2410_01028_b200 as asd
    import synth
    from helpers import assert_logits_close
    shape = synth.DecoderShape(n_layers=1, d_model=2048, n_heads=8, head_dim=256, d_ffn=512, vocab=151936, n_kv_heads=1)
    model = synth.make_model(shape, seed=9)
    dec = asd.Decoder(shape, max_seq=64, max_draft=8)
    dec.load_weights_host(model)
    dec.set_debug(True)
    orc = oracle.Oracle(model, max_seq=64)
    prompt = synth.make_prompt(shape.vocab, 25, seed=10)
    dec.prefill(prompt)
    orc.prefill(prompt)
    assert_logits_close(dec.get_last_logits()[-1:], orc.last()["logits"][-1:])
    dec.decode_step(7)
    orc.decode_step(7)
    one = dec.get_last_logits()
    assert_logits_close(one, orc.last()["logits"])
    dec.reset()
    dec.prefill(prompt)
    dec.verify([7, 1, 2])
    np.testing.assert_array_equal(dec.get_last_logits()[:1], one)
