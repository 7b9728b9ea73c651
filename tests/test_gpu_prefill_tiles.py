"""GPU parity of the prompt products for every kind of tile (pairs of SMs on 256-, 224- and 192-column tiles, single SMs on
tiles of 32 to 256 columns) at ragged edges, and for products cut into parts of their reduction dimension."""
import numpy as np
import pytest

import oracle
import synth
from helpers import COS_TOL, argmax_rows_agree, assert_cos_close, assert_logits_close

pytestmark = pytest.mark.gpu


# fp32 sums of K <= 136 products: an error of at most K 2^-24 of the sum of magnitudes, below 1e-5 of the largest output
@pytest.mark.parametrize("M,N,K", [(129, 12289, 72), (1300, 2100, 136),             # 192-column pair tiles
                                   (257, 9401, 136), (640, 6001, 72),               # 256-column pair tiles, several rounds
                                   (640, 5000, 136), (640, 9473, 72),               # 224-column pair tiles
                                   (3, 40, 72), (129, 1000, 136), (1, 6001, 72),    # single SMs: 32, 64,
                                   (3, 9473, 136), (130, 9401, 72), (3, 18945, 136),  # 96, 128, 160,
                                   (383, 12289, 72)])                               # 256 columns
def test_every_kind_of_tile(M, N, K):
    import torch
    import paper_2410_01028_b200 as asd
    dev = torch.device("cuda:0")
    A = synth.make_matrix_bf16((M, K), seed=M + N + K, stream=1, std=1.0)
    W = synth.make_matrix_bf16((N, K), seed=M + N + K, stream=2, std=0.05)
    A_d = torch.from_numpy(A.view(np.int16)).to(dev).view(torch.bfloat16)
    W_d = torch.from_numpy(W.view(np.int16)).to(dev).view(torch.bfloat16)
    guard = torch.full((M * N + 64,), float("nan"), dtype=torch.float32, device=dev)
    C = guard[:M * N].view(M, N)
    status = torch.ones(8, dtype=torch.int32, device=dev)
    asd.gemm_bf16(A_d, W_d, C, status)
    torch.cuda.synchronize()
    assert status.tolist() == [0] * 8
    ref = synth.bf16_to_f32(A).astype(np.float64) @ synth.bf16_to_f32(W).astype(np.float64).T
    assert np.all(np.abs(C.cpu().numpy() - ref) <= 1e-5 * np.abs(ref).max())
    assert bool(torch.isnan(guard[M * N:]).all())  # nothing behind the last row


WIDE = synth.DecoderShape(n_layers=1, d_model=1024, n_heads=8, head_dim=128, d_ffn=2056, vocab=301, n_kv_heads=4)


# W_o in two parts of 8 blocks of 64, W_d in up to four parts of 8 or 9 (33 blocks, the last one ragged); cosines,
# hidden state (logits) and the mean similarities see the sum of the parts
@pytest.mark.parametrize("S", [33, 128, 129, 300])
def test_products_in_parts(S):
    import paper_2410_01028_b200 as asd
    model = synth.make_model(WIDE, seed=5, std=0.03)
    prompt = synth.make_prompt(WIDE.vocab, S, seed=3)
    dec = asd.Decoder(WIDE, max_seq=S + 1, max_draft=1)
    dec.load_weights_host(model)
    dec.set_debug(True)
    dec.set_prefill_mode(asd.PREFILL_GEMM)
    orc = oracle.Oracle(model, max_seq=S + 1)
    orc.prefill(prompt)
    dec.prefill(prompt)
    last = orc.last()
    assert_logits_close(dec.get_last_logits(), last["logits"][-1:])
    argmax_rows_agree(dec.get_last_logits(), last, slice(-1, None))
    ca, cm = dec.get_last_cosines()
    assert_cos_close(ca, last["cos_attn"][:, -1:])
    assert_cos_close(cm, last["cos_mlp"][:, -1:])
    for g, o in zip(dec.get_similarity()[:2], orc.similarity()[:2]):
        assert np.abs(g - o).max() <= COS_TOL
