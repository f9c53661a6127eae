"""The weight gradient from staged boxes where the input holds infinities or NaN: a pixel spoils
the taps it belongs to and no other, as in the float64 sum (the pad anchors beside it carry zero
gradients, and 0 x infinity is NaN). One such pixel in each corner and side, on channels of
their own; maps whose rows do not fill a unit; both kinds of job. Finite entries keep the bound
of the finite test, 4e-5 sqrt(pixels)."""
import pytest
import torch
import torch.nn.functional as F

from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W,C,Co,beta", [
    (7, 16, 16, 64, 64, 1.0), (2, 32, 32, 64, 64, 0.0), (1, 16, 4, 64, 64, 0.0),
    (5, 8, 8, 128, 128, 0.0), (2, 4, 4, 128, 256, 1.0), (64, 1, 1, 128, 128, 0.0)])
def test_only_a_pixels_own_taps_are_spoilt(N, H, W, C, Co, beta):
    g = torch.Generator(device="cuda").manual_seed(N + H + C)
    x = torch.randn(N, H, W, C, device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn(N, H, W, Co, device="cuda", generator=g).to(torch.bfloat16)
    dy[dy == 0] = 1.0
    spots = [(0, 0), (0, W - 1), (H - 1, 0), (H - 1, W - 1), (H // 2, W - 1), (H // 2, 0), (0, W // 2),
             (H - 1, W // 2)]
    for i, (r, c) in enumerate(spots):
        for k, v in enumerate((float("nan"), float("inf"), -float("inf"))):
            x[(i + k) % N, r, c, 3 * i + k] = v
    ref = torch.zeros(Co, 9 * C, dtype=torch.float64, device="cuda")
    xp = F.pad(x.double(), (0, 0, 1, 1, 1, 1))
    for ky in range(3):
        for kx in range(3):
            tap = xp[:, ky:ky + H, kx:kx + W]
            ref[:, (ky * 3 + kx) * C:(ky * 3 + kx + 1) * C] = dy.double().flatten(0, 2).t() @ tap.flatten(0, 2)
    dw = torch.randn(Co, 9 * C, device="cuda", generator=g)
    ref += beta * dw.double()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.ddppo_conv2d_wgrad(x, dy, dw, 3, 1, 1, beta=beta, status=status)
    assert status.item() == 0
    got = dw.double()
    assert torch.equal(got.isnan(), ref.isnan())
    assert torch.equal(got.isposinf(), ref.isposinf()) and torch.equal(got.isneginf(), ref.isneginf())
    ok = ref.isfinite()
    assert (got - ref)[ok].abs().max().item() <= 4e-5 * (N * H * W) ** 0.5 if ok.any() else True
