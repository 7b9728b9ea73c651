"""A product that is abandoned in mid-run (another CTA's wait has run out: its error word is set, here by a copy from the
host) returns, leaves nothing in flight behind, and the next product on the same SMs is right."""
import time

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(2048, 12288, 8192),   # pairs of SMs
                                   (64, 9472, 32768)])    # single SMs
def test_abandoned_product_leaves_nothing_behind(M, N, K):
    import torch
    import paper_2410_01028_b200 as asd
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(5)
    A = torch.randn((M, K), generator=gen, device=dev).to(torch.bfloat16)
    W = torch.randn((N, K), generator=gen, device=dev).to(torch.bfloat16)
    C = torch.empty((M, N), dtype=torch.float32, device=dev)
    status = torch.zeros(8, dtype=torch.int32, device=dev)
    asd.gemm_bf16(A, W, C, status)
    want = C.clone()
    sel = torch.arange(0, M * N, 9973, device=dev)
    ref = (A[sel // N].double() * W[sel % N].double()).sum(1)
    # fp32 sums of K products of mean magnitude 2 / pi: an error of at most K 2^-24 of the sum of magnitudes
    assert (want.flatten()[sel].double() - ref).abs().max() <= 2.0 ** -24 * K * K
    word = torch.full((1,), 77, dtype=torch.int32).pin_memory()
    side = torch.cuda.Stream()
    seen = 0
    for attempt in range(60):
        C.fill_(float("nan"))
        torch.cuda.synchronize()
        asd.gemm_bf16(A, W, C, status)
        until = time.perf_counter() + 1e-6 * (5 + 10 * (attempt % 12))
        while time.perf_counter() < until:
            pass
        with torch.cuda.stream(side):
            status[:1].copy_(word, non_blocking=True)
        asd_status = torch.zeros(8, dtype=torch.int32, device=dev)
        after = torch.empty_like(C)
        asd.gemm_bf16(A, W, after, asd_status)  # right behind it, on the same SMs
        torch.cuda.synchronize()
        assert asd_status.tolist() == [0] * 8
        assert torch.equal(after, want)
        left = torch.isnan(C)
        assert torch.equal(C[~left], want[~left])  # what was written is right
        seen += bool(left.any())
    assert seen > 0  # at least one was in fact cut short
