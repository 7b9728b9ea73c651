"""GPU parity of the prompt attention kernel at the edges of its tiles (128 query rows x 64 keys): prompts that end one
row before, at and one row behind a tile border, and prompts appended to a cache whose length is not a multiple of a
tile, against the CPU oracle; with weights large enough that the running maximum has to move between tiles."""
import numpy as np
import pytest

import oracle
import synth
from helpers import COS_TOL

pytestmark = pytest.mark.gpu

HD128 = synth.DecoderShape(n_layers=2, d_model=256, n_heads=2, head_dim=128, d_ffn=264, vocab=97, n_kv_heads=1)
HD64 = synth.DecoderShape(n_layers=2, d_model=256, n_heads=4, head_dim=64, d_ffn=264, vocab=97, n_kv_heads=2)


@pytest.mark.parametrize("shape", [HD128, HD64], ids=["hd128", "hd64"])
@pytest.mark.parametrize("std", [0.02, 0.15])  # 0.15: scores of several units, the maximum of a row grows by more than 2^8
@pytest.mark.parametrize("parts", [(2,), (63,), (64,), (65,), (127,), (128, 1), (129,), (33, 96), (61, 131), (192, 65), (257, 300)])
def test_prompt_attention_at_tile_edges(shape, std, parts):
    import paper_2410_01028_b200 as asd
    model = synth.make_model(shape, seed=7, std=std)
    n = sum(parts)
    dec = asd.Decoder(shape, max_seq=n, max_draft=1)
    dec.load_weights_host(model)
    dec.set_prefill_mode(asd.PREFILL_GEMM)
    orc = oracle.Oracle(model, max_seq=n)
    prompt = synth.make_prompt(shape.vocab, n, seed=11)
    at = 0
    for part in parts:
        if part == 1:
            dec.set_prefill_mode(asd.PREFILL_AUTO)  # a single row takes the row passes
        dec.prefill(prompt[at:at + part])
        orc.prefill(prompt[at:at + part])
        at += part
    ca_g, cm_g, rows = dec.get_similarity()
    ca_o, cm_o, _ = orc.similarity()
    assert rows == n
    assert np.abs(ca_g - ca_o).max() <= COS_TOL and np.abs(cm_g - cm_o).max() <= COS_TOL
    # the second layer's K and V rows carry the first layer's attention output of the same position. A flipped bf16
    # rounding upstream moves them by about 1e-3 of their scale; the bound is one ulp plus 1e-2 of the row's scale
    for p in range(n):
        for g, o in zip(dec.get_kv(1, p), orc.kv(1, p)):
            g = synth.bf16_to_f32(g)
            assert np.all(np.abs(g - o) <= 2 ** -7 * np.abs(o) + 1e-2 * np.abs(o).max()), (p, np.abs(g - o).max(), np.abs(o).max())


# A row's arithmetic depends on the keys it sees alone: not on later rows, and not on what an earlier prompt left in the
# buffers behind the last row. A changed order of fp32 operations flips a bf16 rounding in about 3e-5 of the elements of the
# attention output, of which the rows that share a warp with the changed ones have 40000 per prompt.
@pytest.mark.parametrize("head_dim", [128, 64])
def test_rows_depend_neither_on_later_rows_nor_on_earlier_prompts(head_dim):
    import paper_2410_01028_b200 as asd
    shape = synth.DecoderShape(n_layers=2, d_model=2048, n_heads=2048 // head_dim, head_dim=head_dim, d_ffn=264, vocab=97,
                               n_kv_heads=1024 // head_dim)
    n, cut = 507, 500  # 507 rows: five rows of the last warp lie behind the prompt
    dec = asd.Decoder(shape, max_seq=640, max_draft=1)
    dec.load_weights_host(synth.make_model(shape, seed=7, std=0.05))
    dec.set_prefill_mode(asd.PREFILL_GEMM)
    prompt = synth.make_prompt(shape.vocab, n, seed=11)

    def rows_of(tokens):
        dec.reset()
        dec.prefill(tokens)
        return [a.copy() for p in range(384, cut) for a in dec.get_kv(1, p)]

    first = rows_of(prompt)
    for seed in range(12):
        other = synth.make_prompt(shape.vocab, 640, seed=100 + seed)
        changed = prompt.copy()
        changed[cut:] = other[cut:n]
        assert all(np.array_equal(a, b) for a, b in zip(first, rows_of(changed))), "later rows"
        rows_of(other)  # leaves its queries in rows 507 to 639
        assert all(np.array_equal(a, b) for a, b in zip(first, rows_of(prompt))), "an earlier prompt"


# nothing in the kernel may depend on when its products, copies and warps get their turn: many blocks per SM over many
# key tiles, and every repetition gives the same bits
@pytest.mark.parametrize("shape", [HD128, HD64], ids=["hd128", "hd64"])
def test_repeated_prompts_give_the_same_bits(shape):
    import paper_2410_01028_b200 as asd
    n = 2500  # two chunks; up to 40 key tiles per block
    dec = asd.Decoder(shape, max_seq=n, max_draft=1)
    dec.load_weights_host(synth.make_model(shape, seed=7, std=0.15))
    dec.set_prefill_mode(asd.PREFILL_GEMM)
    dec.set_debug(True)
    prompt = synth.make_prompt(shape.vocab, n, seed=11)

    def outputs():
        dec.reset()
        dec.prefill(prompt)
        kv = [a.copy() for p in range(0, n, 7) for a in dec.get_kv(1, p)]
        return kv + [dec.get_last_logits().copy(), *(c.copy() for c in dec.get_similarity()[:2])]

    first = outputs()
    for _ in range(5):
        assert all(np.array_equal(a, b) for a, b in zip(first, outputs()))
