"""The stem kernels (7x7 / stride 2 / pad 3, one channel): rows of 16 to 128 output pixels, one
and many tiles a CTA, 32 and 64 output channels, accumulation.

Forward: float64 convolution of the same bf16 values; fp32 accumulation of 49 products, so
|error| <= 4e-5 * 7 for normal operands. Gradient, through the whole-agent backward: the
stem's weight gradient of the BF16 form has noise of its own, so the kernel is compared with
the general path instead, by taking the observations once on a 16-byte boundary and once off
it: the forward gives the same bits either way, hence the same output gradient, and the sums
over pixels differ by their fp32 order only: 1e-4 relative L2 (sums of 2e4 terms or fewer).
"""
import pytest
import torch
import torch.nn.functional as F

from paper_1911_00357_gb300 import binding as B
from tests import inputs as I
from tests import test_gpu_policy as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,side,Co", [(1, 32, 32), (3, 64, 32), (1500, 32, 64), (40, 128, 32), (5, 256, 64)])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_forward(N, side, Co, beta):
    g = torch.Generator(device="cuda").manual_seed(N + side + Co)
    x = torch.randn(N, side, side, 1, device="cuda", generator=g).bfloat16()
    w = torch.randn(Co, 49, device="cuda", generator=g).bfloat16()
    y0 = torch.randn(N, side // 2, side // 2, Co, device="cuda", generator=g)
    y, st = y0.clone(), torch.zeros(1, dtype=torch.int32, device="cuda")
    B.ddppo_conv2d(x, w, y, 7, 2, 3, beta=beta, status=st)
    torch.cuda.synchronize()
    assert st.item() == 0
    ref = F.conv2d(x.double().permute(0, 3, 1, 2), w.double().view(Co, 1, 7, 7), stride=2, padding=3)
    ref = ref.permute(0, 2, 3, 1) + beta * y0.double()
    assert (y.double() - ref).abs().max().item() <= 4e-5 * 7


@pytest.mark.parametrize("E,base", [(1, 32), (6, 32), (4, 64)])
def test_gradient_matches_the_general_path(E, base):
    net = P.Net(P._cfg("resnet_small", E, 1, 1, base_ch=base), seed=1)
    try:
        dev, _ = P._dev_inputs(net.cfg, I.minibatch(net.ncfg, T=1, E=E, seed=2))
        obs = dev["obs"][:1].contiguous()
        off = torch.empty(obs.numel() + 1, dtype=obs.dtype, device="cuda")[1:].view(obs.shape)
        off.copy_(obs)
        assert obs.data_ptr() % 16 == 0 and off.data_ptr() % 16 == 2
        g = torch.Generator().manual_seed(3)
        dl, dv = torch.randn(1, E, 4, generator=g).cuda(), torch.randn(1, E, generator=g).cuda()
        out = []
        for o in (obs, off):
            logits, values = torch.zeros(1, E, 4, device="cuda"), torch.zeros(1, E, device="cuda")
            B.ddppo_policy_evaluate(net.h, 1, E, o, dev["goal"][:1], dev["prev_a"][:1], dev["masks"][:1],
                                    dev["h0"], dev["c0"], logits, values)
            grad = torch.zeros(net.P, device="cuda")
            B.ddppo_policy_backward(net.h, dl, dv, grad)
            torch.cuda.synchronize()
            out.append((logits.cpu(), grad.cpu().double()))
        assert torch.equal(out[0][0], out[1][0])
        n = base * 49  # the stem's weights come first
        a, b = out[0][1][:n], out[1][1][:n]
        assert torch.linalg.vector_norm(b) > 0
        assert torch.linalg.vector_norm(a - b) <= 1e-4 * torch.linalg.vector_norm(b)
        assert torch.equal(out[0][1][n:], out[1][1][n:])
    finally:
        net.close()
