"""The tcgen05 GEMM around the number of tiles where 128x128 tiles change from one CTA an SM
with a 4-slot operand ring to two CTAs with 2 slots (two tiles for each of 152 SMs), and with
persistent CTAs whose walk over (M tile, N tile, K split) carries in every digit.

Reference: C = A B^T in float64 on the same bf16 values; the kernel accumulates in fp32, so
|error| <= 4e-5 sqrt(K) for normal operands.
"""
import numpy as np
import pytest
import torch

from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [
    (303 * 128, 128, 64), (304 * 128 - 1, 100, 200), (304 * 128, 128, 16), (305 * 128 + 5, 72, 136),
    (153 * 128, 200, 264), (400, 128 * 97 + 8, 80), (130, 128 * 200, 328), (3000, 2000, 1032)])
def test_around_the_ring_rule(M, N, K):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda", generator=g).bfloat16()
    Bm = torch.randn(N, K, device="cuda", generator=g).bfloat16()
    C = torch.full((M, N), 7.0, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert B.ddppo_gemm_backend(A, Bm)
    B.ddppo_gemm(A, Bm, C, status=st)
    torch.cuda.synchronize()
    assert st.item() == 0
    assert (C.double() - A.double() @ Bm.double().t()).abs().max().item() <= 4e-5 * np.sqrt(K)
