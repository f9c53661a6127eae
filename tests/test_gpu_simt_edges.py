"""The FP32 GEMM at the edges of its tiles and loads, and the bias-gradient column sums at
the sizes where their cluster grows.

GEMM: C = A B^T in float64 on the operands' values; the kernel's only difference is its fp32
accumulation, so |error| <= 4e-5 sqrt(K) for normal operands. Tiles: 128x32 for N <= 32,
32x128 for M <= 32, 128x64 for many tiles, else 64x64; an operand's 4-element loads need
rows of a multiple of 4 elements on a 16-byte base, ragged ones are read one by one.

Column sums: the cluster has one CTA per 256 rows, 1 to 8. The rows here are T x E, the
columns 4 x hidden, and both LSTM biases take the same sums; limits as where the same
gradients are checked at other sizes.
"""
import numpy as np
import pytest
import torch

from paper_1911_00357_gb300 import binding as B
from tests.test_gpu_lstm_cluster import test_gradients_match_float64 as lstm_gradients

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (33, 31, 17), (127, 32, 16), (129, 33, 33), (31, 129, 19),
                                   (32, 128, 500), (65, 63, 515), (9730, 257, 35), (4864, 512, 32)])
@pytest.mark.parametrize("a_t,b_t", [(0, 0), (1, 0), (0, 1), (1, 1)])
@pytest.mark.parametrize("pad", [0, 1, 4])
def test_tiles_and_loads(M, N, K, a_t, b_t, pad):
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, device="cuda", generator=g)
    Bm = torch.randn(N, K, device="cuda", generator=g)

    def stored(x, t):  # rows padded by `pad`, the base `pad` elements into its buffer
        x = x.t() if t else x
        buf = torch.full((x.shape[0] * (x.shape[1] + pad) + pad,), 1e9, device="cuda")
        v = torch.as_strided(buf, x.shape, (x.shape[1] + pad, 1), pad)
        v.copy_(x)
        return v

    C0 = torch.randn(M, N + pad, device="cuda", generator=g)
    C = C0.clone()
    bias = torch.randn(N, device="cuda", generator=g)
    B.ddppo_gemm(stored(A, a_t), stored(Bm, b_t), C, beta=0.5, bias=bias, relu=True, M=M, N=N, K=K,
                 lda=(M if a_t else K) + pad, ldb=(N if b_t else K) + pad, ldc=N + pad, a_t=bool(a_t), b_t=bool(b_t))
    torch.cuda.synchronize()
    ref = (A.double() @ Bm.double().t() + 0.5 * C0[:, :N].double() + bias.double()).clamp_min(0)
    assert (C[:, :N].double() - ref).abs().max().item() <= 4e-5 * np.sqrt(K)
    assert torch.equal(C[:, N:], C0[:, N:])


@pytest.mark.parametrize("hidden,layers,T,E", [(64, 1, 16, 16), (64, 1, 257, 1), (128, 2, 20, 26), (64, 2, 64, 33)])
def test_bias_gradient_rows(hidden, layers, T, E):
    lstm_gradients(hidden, layers, T, E, 0)
