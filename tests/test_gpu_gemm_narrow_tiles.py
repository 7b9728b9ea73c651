"""Dense products whose last rounds run on narrower tiles than the first: the tiles cover every column once and need no more rounds (no GPU
needed), and the products agree with 64 bits at ragged edges of wide and narrow tiles."""
import ctypes
import functools
import os
import random
import subprocess
import tempfile

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_01028_b200", "csrc")


@functools.lru_cache(None)
def _lib():
    with tempfile.TemporaryDirectory() as tmp:
        src, lib = os.path.join(tmp, "plan.cpp"), os.path.join(tmp, "plan.so")
        with open(src, "w") as f:
            f.write('#include "gemm_plan.h"\nextern "C" void plan(int m, int n, int k, int parts, int sms, int* o) {\n'
                    "    const asd::GemmPlan p = asd::plan_gemm(m, n, k, parts, sms);\n"
                    "    o[0] = p.bn, o[1] = p.cg, o[2] = p.m_tiles, o[3] = p.tiles, o[4] = p.parts, o[5] = p.wide, o[6] = p.narrow, o[7] = p.items;\n}\n")
        subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", lib, src], check=True)
        return ctypes.CDLL(lib)


def _plan(M, N, K, parts=1, sms=148):
    out = (ctypes.c_int * 8)()
    _lib().plan(M, N, K, parts, sms, out)
    return list(out)


def test_tiles_cover_the_columns_in_as_many_rounds():
    rng, mixed = random.Random(3), 0
    for _ in range(4000):
        M, N, K, sms = rng.randint(1, 2048), rng.randint(1, 44032), 8 * rng.randint(1, 1376), rng.choice([2, 132, 148, 160])
        bn, cg, m_tiles, tiles, parts, wide, narrow, items = _plan(M, N, K, rng.randint(1, 8), sms)
        assert 0 < narrow <= bn and narrow % 32 == 0 and items % m_tiles == 0 and 0 <= wide <= items // m_tiles
        cols, units = items // m_tiles, sms // cg
        assert wide * bn + (cols - wide) * narrow >= N and wide * bn + (cols - wide - 1) * narrow < N  # the last tile has columns
        if narrow < bn:
            mixed += 1
            assert cg == 2 and parts == 1 and cols > wide and -(-items // units) == -(-tiles // units)
        else:
            assert items == tiles
    assert mixed > 200


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,widths", [(511, 12288, 200, (192, 160)), (512, 22010, 136, (224, 160)), (1023, 11001, 1032, (224, 160)), (2048, 4095, 72, (256, 224)),
                                          (2048, 27640, 72, (256, 192))])
def test_products_with_two_widths(M, N, K, widths):
    import torch
    import paper_2410_01028_b200 as asd
    plan = _plan(M, N, K, sms=torch.cuda.get_device_properties(0).multi_processor_count)
    assert (plan[0], plan[6]) == widths
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
    # fp32 sums of K products: an error of at most K 2^-24 of the sum of magnitudes, below 1e-5 of the largest output
    assert bool(((C.double() - ref).abs() <= 1e-5 * ref.abs().max()).all())
    assert bool(torch.isnan(guard[M * N:]).all())
