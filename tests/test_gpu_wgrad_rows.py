"""Weight gradient of the 3x3 stride-1 convolutions with 64 or more channels (shifted views
of one staged box per unit), against the float64 sum over exactly the bf16 values it reads;
only the fp32 accumulation differs: within 4e-5 sqrt(pixels), the bound of the other
contraction tests. Sizes: one image, images per unit that do not divide the batch, row
blocks, maps from 1x1 to 32x32, several jobs per kind, one unit and many, accumulation."""
import pytest
import torch
import torch.nn.functional as F

from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W,C,Co,beta", [
    (1, 16, 16, 64, 64, 0.0), (7, 16, 16, 64, 64, 1.0), (3, 32, 32, 64, 64, 0.0),
    (9, 16, 4, 64, 64, 0.0), (700, 16, 16, 64, 64, 0.0), (2, 4, 4, 64, 64, 0.0),
    (5, 8, 8, 128, 128, 0.0), (1, 8, 8, 256, 128, 1.0), (2, 4, 4, 128, 256, 0.0),
    (33, 4, 4, 256, 256, 0.0), (3, 2, 2, 128, 128, 0.0), (64, 1, 1, 128, 128, 0.0),
    (3, 32, 32, 128, 128, 0.5), (900, 8, 8, 128, 128, 0.0), (5, 4, 4, 512, 512, 0.0)])
def test_weight_gradient_rows(N, H, W, C, Co, beta):
    g = torch.Generator(device="cuda").manual_seed(N + 17 * H + C + Co)
    x = torch.randn(N, H, W, C, device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn(N, H, W, Co, device="cuda", generator=g).to(torch.bfloat16)
    dw = torch.randn(Co, 9 * C, device="cuda", generator=g)
    ref = torch.zeros(Co, C * 9, dtype=torch.float64, device="cuda")
    for xi, yi in zip(x.split(64), dy.split(64)):
        cols = F.unfold(xi.double().permute(0, 3, 1, 2), 3, padding=1)
        ref += torch.einsum("npo,nkp->ok", yi.double().flatten(1, 2), cols)
    ref = ref.view(Co, C, 9).transpose(1, 2).reshape(Co, 9 * C) + beta * dw.double()
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.ddppo_conv2d_wgrad(x, dy, dw, 3, 1, 1, beta=beta, status=status)
    assert status.item() == 0
    assert (dw.double() - ref).abs().max().item() <= 4e-5 * (N * H * W) ** 0.5
