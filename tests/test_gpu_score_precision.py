"""How far attention scores of a row pass are from 64 bits. Two keys have the same score in exact arithmetic (the second is the first one
permuted, the query is the same on permuted dimensions), scores are millions, and the weight that the first key gets shows the difference of
the two rounding errors: 1 / (1 + exp(-difference))."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

D = 1024  # a one-hot embedding has a normalised entry of sqrt(D) = 32: weights and activations are exact


def _bf16(a):
    bits = np.ascontiguousarray(a, np.float32).view(np.uint32)
    assert not np.any(bits & 0xFFFF), "not a bf16 value"
    return (bits >> 16).astype(np.uint16)


@pytest.mark.parametrize("head_dim", [128, 256])
def test_scores_are_as_exact_as_sums_in_fp32(head_dim):
    """In units of 2^-24 of the score S. An addition in fp32 whose result is v adds 0.29 to 0.58 of v (rms; 0.41 on average). Sums of 16 products
    are added in a tree: heads of 128 0.41 sqrt(4 / 4^2 + 2 / 2^2 + 1) = 0.54, heads of 256 0.41 sqrt(8 / 8^2 + 4 / 4^2 + 2 / 2^2 + 1) = 0.56. In a chain
    of 8 or 16, with the product with the scale behind it (heads of 128), it would be 0.84 and 0.99. The bound is 15 % above the tree: the
    values behind an addition are not spread evenly, the number of scores leaves 2 to 3 %."""
    import paper_2410_01028_b200 as asd
    rng = np.random.default_rng(head_dim)
    heads, half, n_pairs = D // head_dim, head_dim // 2, 200
    # rotary pairs whose angle is below 1e-4 at position 1 leave bf16 values as they are; the others are not used
    j0 = next(j for j in range(half) if 1e38 ** (-j / half) < 1e-4)
    active = np.concatenate([np.arange(j0, half), half + np.arange(j0, half)])
    q, k_a, k_b = (np.zeros((n_pairs, heads, head_dim), np.float32) for _ in range(3))
    for i in range(n_pairs):
        for h in range(heads):
            order = rng.permutation(active)
            left, right = order[0::2], order[1::2]
            v, *k = rng.integers(128, 256, (3, len(left))) * 2.0 ** rng.integers(0, 4, (3, len(left)))  # bf16; sums have more bits than fp32
            q[i, h, left] = q[i, h, right] = v
            k_a[i, h, left], k_a[i, h, right] = k
            k_b[i, h, right], k_b[i, h, left] = k
    score = (q.astype(np.float64) * k_a).sum(-1) / np.sqrt(head_dim)
    np.testing.assert_array_equal(score, (q.astype(np.float64) * k_b).sum(-1) / np.sqrt(head_dim))

    # tokens 2 i and 2 i + 1 are the two keys of pair i, the query belongs to the second one
    shape = synth.DecoderShape(n_layers=1, d_model=D, n_heads=heads, head_dim=head_dim, d_ffn=64, vocab=D)
    model = synth.make_model(shape, seed=1)
    w = {n: np.zeros((D, D), np.float32) for n in ("wq", "wk", "wv")}
    for i in range(n_pairs):
        w["wk"][:, 2 * i], w["wk"][:, 2 * i + 1], w["wq"][:, 2 * i + 1] = k_a[i].ravel() / 32, k_b[i].ravel() / 32, q[i].ravel() / 32
    w["wv"][0::head_dim, 0::2] = 1 / 32          # dimension 0 of a head: 1 from the first key, 0 from the second
    w["wv"][1::head_dim, :] = 1 / 32             # dimension 1: 1 from both
    for name, a in w.items():
        getattr(model, name)[0] = _bf16(a)
    eye = _bf16(np.eye(D))
    model.embed[:], model.lm_head[:], model.wo[0] = eye, eye, eye
    for gain in (model.attn_norm, model.mlp_norm, model.final_norm):
        gain[:] = 0x3F80
    model.wd[:] = 0
    dec = asd.Decoder(shape, max_seq=16, max_draft=8, rms_eps=1e-9, rope_theta=1e38)
    dec.load_weights_host(model)
    dec.set_debug(True)
    errors = []
    for i in range(n_pairs):
        dec.reset()
        dec.prefill([2 * i])
        dec.decode_step(2 * i + 1)
        for pos, want in ((0, k_a[i]), (1, k_b[i])):
            np.testing.assert_array_equal(dec.get_kv(0, pos)[0], _bf16(want.ravel()))
        logits = dec.get_last_logits()[0].astype(np.float64)
        own = (2 * i + 1) // head_dim if (2 * i + 1) % head_dim == 1 else -1  # the head whose entries the residual stream's own one is among
        keep = np.arange(heads) != own
        ratio = (logits[0::head_dim] / logits[1::head_dim])[keep]
        errors.append(np.log(ratio / (1 - ratio)) / score[i][keep])
    errors = np.concatenate(errors)
    rms = float(np.sqrt(np.mean(errors ** 2) / 2)) * 2.0 ** 24  # of one score
    print("rms error of a score: %.3f x 2^-24, %d scores" % (rms, len(errors)))
    assert 0.1 < rms < 0.65
