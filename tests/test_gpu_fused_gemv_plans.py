"""GPU parity of the stand-alone fused product over its launch plans: one to nine activation rows, fewer weight rows than SMs,
rows that end inside a group of 16, inputs that end inside a piece and inside a unit of 32, activations in several windows of shared
memory, several blocks of rows per CTA; and rows that do not depend on how many rows a call has."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _run(M, n_in, n_rows, epi, norm, x, W, gain, res):
    import torch
    import paper_2410_01028_b200 as asd
    dev = torch.device("cuda:0")
    bf = lambda a: torch.from_numpy(a.view(np.int16)).to(dev).view(torch.bfloat16)
    x_d = torch.from_numpy(x[:M].copy()).to(dev)
    x_d = x_d if norm else x_d.to(torch.bfloat16)  # the inputs are bf16-representable
    if epi == asd.EPI_SWIGLU:
        out = torch.full((M, n_rows // 2), float("nan"), dtype=torch.bfloat16, device=dev)
    elif epi == asd.EPI_RESIDUAL:
        out = torch.from_numpy(res[:M].copy()).to(dev)
    else:
        out = torch.full((M, n_rows), float("nan"), dtype=torch.float32, device=dev)
    cos = torch.full((M,), float("nan"), dtype=torch.float32, device=dev)
    scratch = torch.zeros(asd.fused_gemv_scratch_bytes(), dtype=torch.uint8, device=dev)
    asd.fused_gemv(x_d, bf(W), epi, out, gain=bf(gain) if norm else None, cos=cos if epi == asd.EPI_RESIDUAL else None, scratch=scratch)
    torch.cuda.synchronize()
    return out.float().cpu().numpy(), cos.cpu().numpy()


@pytest.mark.parametrize("n_in,n_rows", [(8, 1), (120, 3), (136, 295), (2056, 4737), (72, 40001), (13760, 40), (22016, 296)])
@pytest.mark.parametrize("epi,norm", [(0, True), (0, False), (1, True), (2, True), (2, False)])
def test_plans_match_oracle_and_rows_do_not_depend_on_M(n_in, n_rows, epi, norm):
    if epi == 1 and n_rows % 2:  # gate and up rows come in pairs
        n_rows += 1
    if norm and n_in * 9 * 2 > 200000:
        n_in = 8200  # RMSNorm takes rows that fit shared memory
    x = synth.make_array_f32((9, n_in), seed=n_in, stream=1)
    W = synth.make_matrix_bf16((n_rows, n_in), seed=n_rows, stream=2, std=0.05)
    gain = synth.make_matrix_bf16((n_in,), seed=3, stream=3, mean=1.0)
    res = synth.make_array_f32((9, n_rows), seed=4, stream=4)
    pairs = dict(W2=np.ascontiguousarray(W[1::2])) if epi == 1 else {}  # the oracle takes gate and up rows apart
    ref, ref_cos = oracle.fused_matvec(x, np.ascontiguousarray(W[0::2]) if epi == 1 else W, epilogue=epi, gain=gain if norm else None,
                                       res=res if epi == 2 else None, **pairs)
    full, full_cos = _run(9, n_in, n_rows, epi, norm, x, W, gain, res)
    scale = np.abs(ref).max()
    if epi == 1:  # bf16 outputs: one-ulp flips
        assert np.all(np.abs(full - ref) <= 2 ** -7 * np.abs(ref) + 1e-3 * scale)
    else:  # a flipped bf16 rounding of a normalised input moves one product by 2^-8; otherwise fp32 sums only
        assert np.all(np.abs(full - ref) <= (2e-3 if norm else 1e-5) * scale)
    if epi == 2:
        assert np.abs(full_cos - ref_cos).max() <= 1e-5 + (1e-3 if norm else 0)
    for M in (1, 2, 5, 8):
        part, part_cos = _run(M, n_in, n_rows, epi, norm, x, W, gain, res)
        assert np.array_equal(part, full[:M]), M
        if epi == 2:
            assert np.array_equal(part_cos, full_cos[:M]), M


# the RMSNorm takes rows of up to 4096 inputs five at a time and longer ones in groups of two to five: whole and partial groups,
# activations in one window and in several
@pytest.mark.parametrize("M", [3, 4, 6, 7])
@pytest.mark.parametrize("n_in,n_rows", [(136, 295), (2056, 4737), (8200, 296)])
def test_rows_of_partial_groups_equal_those_of_nine_rows(M, n_in, n_rows):
    x = synth.make_array_f32((9, n_in), seed=n_in, stream=1)
    W = synth.make_matrix_bf16((n_rows, n_in), seed=n_rows, stream=2, std=0.05)
    gain = synth.make_matrix_bf16((n_in,), seed=3, stream=3, mean=1.0)
    full, _ = _run(9, n_in, n_rows, 0, True, x, W, gain, None)  # compared with the oracle above
    part, _ = _run(M, n_in, n_rows, 0, True, x, W, gain, None)
    assert np.array_equal(part, full[:M])


# the stream's own edges: pieces of 1024 and (from 4096 inputs, where three fit the ring) 2048 inputs, sums kept in registers over
# 4096, one to four units of 32 inputs per warp, rows of one to three groups of 16, and activations in windows of multiples of 4096
# inputs (nine rows of 13768). Bounds: sums of at most 13768 products in fp32 (1e-5 of the output scale, as above); rows equal
# whatever the pieces and windows.
@pytest.mark.parametrize("n_in", [512, 520, 1024, 1032, 4096, 4104, 8192, 13768])
@pytest.mark.parametrize("n_rows", [148, 2 * 148 * 16 + 6])
def test_pieces_epochs_and_windows(n_in, n_rows):
    x = synth.make_array_f32((9, n_in), seed=n_in, stream=1)
    W = synth.make_matrix_bf16((n_rows, n_in), seed=n_rows, stream=2, std=0.05)
    full, _ = _run(9, n_in, n_rows, 0, False, x, W, None, None)
    ref, _ = oracle.fused_matvec(x, W, epilogue=0, gain=None, res=None)
    assert np.all(np.abs(full - ref) <= 1e-5 * np.abs(ref).max())
    for M in (1, 4, 5):
        part, _ = _run(M, n_in, n_rows, 0, False, x, W, None, None)
        assert np.array_equal(part, full[:M]), M
