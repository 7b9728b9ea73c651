"""Dense products whose last rounds run on narrower tiles than the first: the tiles cover every column once and need no more rounds (no GPU
needed), and the products agree with 64 bits at ragged edges of wide and narrow tiles, and of tiles of one width where the rule asks for that."""
import random

import pytest

from helpers import gemm_plan


def test_tiles_cover_the_columns_in_as_many_rounds():
    rng, mixed = random.Random(3), 0
    for _ in range(4000):
        M, N, K, sms = rng.randint(1, 2048), rng.randint(1, 44032), 8 * rng.randint(1, 1376), rng.choice([2, 132, 148, 160])
        if rng.random() < 0.5:
            N, K = 8 * (N // 8 + 1), 32 * (K // 32 + 1)
        bn, cg, m_tiles, tiles, parts, wide, narrow, items = gemm_plan(M, N, K, rng.randint(1, 8), sms)
        assert 0 < narrow <= bn and narrow % 32 == 0 and items % m_tiles == 0 and 0 <= wide <= items // m_tiles
        cols, units = items // m_tiles, sms // cg
        assert wide * bn + (cols - wide) * narrow >= N and wide * bn + (cols - wide - 1) * narrow < N  # the last tile has columns
        if narrow < bn:
            mixed += 1
            assert cg == 2 and parts == 1 and K % 32 == 0 and N % 8 == 0 and cols > wide and -(-items // units) == -(-tiles // units)
        else:
            assert items == tiles
    assert mixed > 200


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K,widths", [(511, 12288, 224, (192, 160)), (512, 22008, 160, (224, 160)), (1023, 11000, 1056, (224, 160)), (2048, 4088, 96, (256, 224)),
                                          (2048, 27640, 96, (256, 192)),
                                          # rows of A and W that are no multiple of 64 bytes, rows of C that are none of 32: one width
                                          (511, 12288, 200, (192, 192)), (1023, 11000, 1032, (224, 224)), (2048, 4095, 96, (256, 256)), (512, 22012, 160, (224, 224))])
def test_products_with_two_widths(M, N, K, widths):
    import torch
    import paper_2410_01028_b200 as asd
    plan = gemm_plan(M, N, K, sms=torch.cuda.get_device_properties(0).multi_processor_count)
    assert (plan.bn, plan.narrow) == widths
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
    error = float((C.double() - ref).abs().max() / ref.abs().max())
    print("largest error %.2e of the largest output" % error)
    # a measured limit: sums in fp32 come within 2e-6 of the largest output here (1.5e-6 at K = 1056, 4e-7 at 224), 16 products that are missing or another row's are 1e-2 of it
    assert error <= 1e-5
    assert bool(torch.isnan(guard[M * N:]).all())
