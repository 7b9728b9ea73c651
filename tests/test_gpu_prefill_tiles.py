"""GPU parity of the prompt products for every kind of tile (pairs of SMs on 256-, 224- and 192-column tiles, single SMs on
tiles of 32, 64, 96, 128, 160 and 256 columns) at ragged edges and over several rounds, and for products cut into parts of
their reduction dimension. Every case says which tile it is there for, and the library's own rule has to agree."""
import numpy as np
import pytest

import oracle
import synth
from helpers import COS_TOL, argmax_rows_agree, assert_cos_close, assert_logits_close, gemm_plan

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


# (columns of a tile, SMs of a unit)
TILES = {(129, 12289, 72): (192, 2), (1300, 2100, 136): (192, 2), (257, 9401, 136): (256, 2), (640, 6001, 72): (256, 2),
         (640, 5000, 136): (224, 2), (640, 9473, 72): (224, 2), (3, 40, 72): (32, 1), (129, 1000, 136): (32, 1), (1, 6001, 72): (64, 1),
         (3, 9473, 136): (96, 1), (130, 9401, 72): (128, 1), (3, 18945, 136): (160, 1), (383, 12289, 72): (256, 1)}


# 17 blocks of 64 inputs, the last one ragged: more than any tile has stages (4 to 8), so that every stage is filled again;
# and at least three tiles per unit, so that both accumulators are used again. (The narrow tiles are chosen for one round only.)
# fp32 sums of 1032 products: below 1e-5 of the largest output, as in test_gpu_prefill_dense.py.
@pytest.mark.parametrize("M,N,tile,rounds", [(258, 25236, (256, 2), 3), (515, 15180, (224, 2), 3), (385, 18964, (192, 2), 3),
                                             (514, 18989, (256, 1), 3), (257, 28555, (160, 1), 4), (257, 16641, (128, 1), 3),
                                             (3, 9473, (96, 1), 1), (1, 6001, (64, 1), 1), (3, 40, (32, 1), 1)])
def test_stages_and_accumulators_in_several_rounds(M, N, tile, rounds):
    import torch
    import paper_2410_01028_b200 as asd
    K, sms = 1032, _sms()
    plan = gemm_plan(M, N, K, sms=sms)
    assert plan[:2] == tile and -(-plan.tiles // (sms // plan.cg)) == rounds
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(M + N)
    A = torch.randn((M, K), generator=gen, device=dev).to(torch.bfloat16)
    W = (0.05 * torch.randn((N, K), generator=gen, device=dev)).to(torch.bfloat16)
    guard = torch.full((M * N + 64,), float("nan"), dtype=torch.float32, device=dev)
    C = guard[:M * N].view(M, N)
    status = torch.ones(8, dtype=torch.int32, device=dev)
    asd.gemm_bf16(A, W, C, status)
    assert status.tolist() == [0] * 8
    ref = A.double() @ W.double().T
    assert bool(((C.double() - ref).abs() <= 1e-5 * ref.abs().max()).all())
    assert bool(torch.isnan(guard[M * N:]).all())


# fp32 sums of K <= 136 products: an error of at most K 2^-24 of the sum of magnitudes, below 1e-5 of the largest output
@pytest.mark.parametrize("M,N,K", [(129, 12289, 72), (1300, 2100, 136),             # 192-column pair tiles
                                   (257, 9401, 136), (640, 6001, 72),               # 256-column pair tiles
                                   (640, 5000, 136), (640, 9473, 72),               # 224-column pair tiles, one and two rounds
                                   (3, 40, 72), (129, 1000, 136), (1, 6001, 72),    # single SMs: 32, 32, 64,
                                   (3, 9473, 136), (130, 9401, 72), (3, 18945, 136),  # 96, 128, 160,
                                   (383, 12289, 72)])                               # 256 columns
def test_every_kind_of_tile(M, N, K):
    assert gemm_plan(M, N, K, sms=_sms())[:2] == TILES[M, N, K]
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


# W_o in parts of its 16 blocks of 64, W_d in parts of its 33 (the last one ragged); cosines, hidden state (logits)
# and the mean similarities see the sum of the parts. The buffer of the parts has room for 1024 rows.
@pytest.mark.parametrize("S,parts_o,parts_d", [(33, 2, 4), (128, 2, 4), (129, 2, 4), (300, 2, 3)])
def test_products_in_parts(S, parts_o, parts_d):
    import paper_2410_01028_b200 as asd
    most, d = min(8, 1024 // S), WIDE.d_model
    assert gemm_plan(S, d, d, most, _sms()).parts == parts_o and gemm_plan(S, d, WIDE.d_ffn, most, _sms()).parts == parts_d
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
