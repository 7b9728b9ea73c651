"""GPU parity of the stand-alone fused product where its variants meet: RMSNorm of rows that are held in registers or read twice, in
groups of one to five; groups of short weight rows by a warp each; the last piece of a row; blocks of weight rows together with windows
of activations; and activations that are not finite. Every row of a call equals the same row of a call with nine rows."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_fused_gemv_plans import _run

pytestmark = pytest.mark.gpu


def _check(n_in, n_rows, epi, norm, rows, tol):
    x = synth.make_array_f32((9, n_in), seed=n_in, stream=1)
    W = synth.make_matrix_bf16((n_rows, n_in), seed=n_rows, stream=2, std=0.05)
    gain = synth.make_matrix_bf16((n_in,), seed=3, stream=3, mean=1.0)
    res = synth.make_array_f32((9, n_rows), seed=4, stream=4)
    most = max(rows)
    pairs = dict(W2=np.ascontiguousarray(W[1::2])) if epi == 1 else {}
    ref, ref_cos = oracle.fused_matvec(x[:most], np.ascontiguousarray(W[0::2]) if epi == 1 else W, epilogue=epi,
                                       gain=gain if norm else None, res=res[:most] if epi == 2 else None, **pairs)
    full, full_cos = _run(most, n_in, n_rows, epi, norm, x, W, gain, res)
    scale = np.abs(ref).max()
    assert np.all(np.abs(full - ref) <= (2 ** -7 * np.abs(ref) if epi == 1 else 0) + tol * scale)
    if epi == 2:
        assert np.abs(full_cos - ref_cos).max() <= 1e-5 + (1e-3 if norm else 0)
    for M in rows:
        part, part_cos = _run(M, n_in, n_rows, epi, norm, x, W, gain, res)
        assert np.array_equal(part, full[:M]), M
        if epi == 2:
            assert np.array_equal(part_cos, full_cos[:M]), M


# Bound behind an RMSNorm: a flipped bf16 rounding of a normalised input moves one product by 2^-8 of itself, a few of thousands
# flip (2e-3 of the output scale, as in the tests of the launch plans). Up to 5120 inputs rows are held in registers; beyond, they are read
# in batches of 1024 x (12 / rows of a group) inputs; 12296 and 34000 inputs have activations in several windows.
@pytest.mark.parametrize("n_in,rows", [(3080, (1, 2, 3, 5, 9)), (4096, (1, 2, 3, 5, 9)), (4104, (1, 2, 3, 5, 9)), (5120, (1, 2, 3, 5, 9)),
                                       (5128, tuple(range(1, 10))), (6144, tuple(range(1, 10))), (9224, tuple(range(1, 10))),
                                       (12296, tuple(range(1, 9))), (22016, (1, 2, 3, 4)), (34000, (1, 2, 3))])
def test_norm_of_long_rows(n_in, rows):
    _check(n_in, 297, 0, True, rows, 2e-3)


# Groups of 16 rows by a warp each: up to 768 inputs and from 50 weight rows per SM on (7104 weight rows: 48 per SM), one to three
# units of 256 inputs, a ring of 8 and of 16 stages, one lap of it and several
@pytest.mark.parametrize("n_in", [8, 248, 256, 264, 512, 520, 688, 768, 776])
@pytest.mark.parametrize("n_rows", [7104, 7106, 148 * 130 + 7, 148 * 300])
@pytest.mark.parametrize("epi,norm", [(0, False), (1, True), (2, False), (2, True)])
def test_short_rows(n_in, n_rows, epi, norm):
    _check(n_in, n_rows + (n_rows % 2 if epi == 1 else 0), epi, norm, (1, 2, 5, 8, 9), 2e-3 if norm else 1e-5)


# The last piece of a row takes what is left up to half a piece more (1024 and, from 4096 inputs on, 2048 inputs)
@pytest.mark.parametrize("n_in", [1032, 1536, 1544, 2056, 2560, 2568, 3080, 4104, 5632, 6152, 7168, 7176, 11008])
def test_last_piece_of_a_row(n_in):
    _check(n_in, 2371, 0, False, (1, 3, 5, 7, 9), 1e-5)


# More than 256 weight rows per SM, so several blocks, each going through two windows of the activations anew
@pytest.mark.parametrize("norm", [False, True])
def test_blocks_of_rows_and_windows(norm):
    import torch
    import paper_2410_01028_b200 as asd
    M, n_in, n_rows = 9, 11000, 38500
    gen = torch.Generator(device="cuda").manual_seed(11)
    x = torch.randn((M, n_in), generator=gen, device="cuda")
    x = x if norm else x.to(torch.bfloat16)
    W = torch.randn((n_rows, n_in), generator=gen, device="cuda").mul_(0.05).to(torch.bfloat16)
    gain = torch.randn(n_in, generator=gen, device="cuda").mul_(0.1).add_(1).to(torch.bfloat16)
    scratch = torch.zeros(asd.fused_gemv_scratch_bytes(), dtype=torch.uint8, device="cuda")
    out = torch.empty((M, n_rows), device="cuda")
    asd.fused_gemv(x, W, asd.EPI_PLAIN, out, gain=gain if norm else None, scratch=scratch)
    xin = x.double()
    if norm:
        xin = (xin * torch.rsqrt((xin * xin).mean(-1, keepdim=True) + 1e-5) * gain.double()).to(torch.bfloat16).double()
    ref = torch.cat([xin @ w.double().T for w in W.split(4096)], 1)
    assert (out.double() - ref).abs().max() <= (2e-3 if norm else 1e-5) * ref.abs().max()
    few = torch.empty((2, n_rows), device="cuda")
    asd.fused_gemv(x[:2].contiguous(), W, asd.EPI_PLAIN, few, gain=gain if norm else None, scratch=scratch)
    assert torch.equal(few, out[:2])


# What is not finite stays in its row of the results
@pytest.mark.parametrize("n_in,n_rows", [(520, 8000), (2056, 300), (13768, 300)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("norm", [False, True])
def test_rows_that_are_not_finite(n_in, n_rows, bad, norm):
    M = 9 if n_in < 13000 else 8
    x = synth.make_array_f32((9, n_in), seed=n_in, stream=1)
    W = synth.make_matrix_bf16((n_rows, n_in), seed=n_rows, stream=2, std=0.05)
    gain = synth.make_matrix_bf16((n_in,), seed=3, stream=3, mean=1.0)
    good, _ = _run(M, n_in, n_rows, 0, norm, x, W, gain, None)
    x[2, n_in - 3] = bad
    got, _ = _run(M, n_in, n_rows, 0, norm, x, W, gain, None)
    others = [m for m in range(M) if m != 2]
    assert np.array_equal(got[others], good[others])
    # (a row with an infinity has a root mean square of infinity: zeros, but for infinity over infinity)
    assert np.all(np.isnan(got[2])) if norm or np.isnan(bad) else not np.any(np.isfinite(got[2]))
