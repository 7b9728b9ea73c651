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


# Long chains of products must not lose what they add up. Tokens share most of their embedding, so that the values of a head
# have a mean and the rows' sums grow with every key; the attention output is as large as the hidden state it is added to.
# A sum that has lost the share e of itself moves the mean cosine before and after by about e / 2. Rounded to nearest, the
# sums of 8192 keys lose far below 1e-6. An MMA cuts every sum off by half an ulp on average: a chain over half of the keys
# of a row (768 steps on the longest row, counted by half of the sum, at a mean size of half) loses up to 768 * 2^-24 / 4 = 1.1e-5
# and the shorter ones before it as much again over all rows: a cosine off by at most 6e-6. Left to grow over
# all keys, a chain loses up to 4.6e-5 (measured: 1e-5 in the mean cosine).
@pytest.mark.parametrize("head_dim", [128, 64])
def test_attention_over_many_keys_keeps_its_sums(head_dim):
    import torch
    import paper_2410_01028_b200 as asd
    d, S, H = 256, 8192, 256 // head_dim
    shape = synth.DecoderShape(n_layers=1, d_model=d, n_heads=H, head_dim=head_dim, d_ffn=64, vocab=499)
    model = synth.make_model(shape, seed=3, std=0.0625, scale_lo=1.0)
    base, noise = synth.make_array_f32((1, d), seed=5, stream=1), synth.make_array_f32((499, d), seed=5, stream=2)
    model.embed = synth.f32_to_bf16(base + 0.5 * noise)
    prompt = synth.make_prompt(shape.vocab, S, seed=11)
    dec = asd.Decoder(shape, max_seq=S, max_draft=1)
    dec.load_weights_host(model)
    dec.prefill(prompt)
    got = float(dec.get_similarity()[0][0])

    def w(a):
        return torch.from_numpy(synth.bf16_to_f32(a)).cuda().double()

    def bf(t):
        return t.float().to(torch.bfloat16).double()

    x = w(model.embed)[torch.from_numpy(prompt).cuda().long()]
    xn = bf(x * torch.rsqrt((x * x).mean(-1, keepdim=True) + dec.cfg.rms_eps) * w(model.attn_norm[0]))
    ang = torch.arange(S, device="cuda").double()[:, None] * torch.exp(
        -np.log(dec.cfg.rope_theta) * 2.0 * torch.arange(head_dim // 2, device="cuda").double() / head_dim)
    cos, sin = torch.cos(ang).float().double()[:, None], torch.sin(ang).float().double()[:, None]

    def rope(t):
        a, b = t.view(S, H, head_dim).chunk(2, -1)
        return bf(torch.cat([a * cos - b * sin, b * cos + a * sin], -1))

    q, k, v = rope(xn @ w(model.wq[0]).T), rope(xn @ w(model.wk[0]).T), bf(xn @ w(model.wv[0]).T).view(S, H, head_dim)
    o = torch.empty(S, H, head_dim, dtype=torch.float64, device="cuda")
    later = torch.ones(S, S, dtype=torch.bool, device="cuda").triu_(1)
    for h in range(H):
        o[:, h] = torch.softmax((q[:, h] @ k[:, h].T / head_dim ** 0.5).masked_fill_(later, -np.inf), -1) @ v[:, h]
    y = x + bf(o).view(S, d) @ w(model.wo[0]).T
    ref = float(((x * y).sum(-1) / (x.norm(dim=-1) * y.norm(dim=-1))).mean())
    assert abs(got - ref) <= 6e-6, (got, ref, got - ref)


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
