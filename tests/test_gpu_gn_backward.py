"""The GroupNorm backward's forms (the shared-memory ring, one block per image, channel slices,
two launches) inside the FP32 encoder, against float64 autograd of the oracle's encoder: base
widths whose channel counts divide 256 and ones that do not, batches on both sides of four
images an SM (the ring's limit), 64x64 frames (256, 64, 16 and 4 pixels a stage, so that units
are uneven: 96 channels take 20, 20, 20 and 4 pixels). Every masked GroupNorm of the block
outputs reads the stored bits, the others recompute the mask; the identity blocks return the
masked gradient in place.

Bound, per tensor: 3e-2 of its norm, the FP32 ResNet encoder's bound in the other gradient
tests (ReLU kinks: an activation within fp32 rounding of zero flips its mask). A unit, row or
mask read from the wrong place changes at least one of its 4 or more units an image, a tenth of
a tensor's norm or more."""
import pytest
import torch

from oracle import policy as OP
from paper_1911_00357_gb300 import binding as B
from paper_1911_00357_gb300.presets import make_config
from tests import inputs as I
from tests.gpu_util import net_config_from

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,over", [(24, 1), (32, 1), (48, 1), (56, 1), (32, -1), (48, -1)])
def test_encoder_gradient_at_every_form(base, over):
    N = 4 * torch.cuda.get_device_properties(0).multi_processor_count + over
    cfg = make_config("nature_fp32", net_kind=1, base_ch=base, hidden=64, num_envs=1, rollout_T=N,
                      minibatches=1, encoder_chunk=N)
    nc = net_config_from(cfg)
    h = B.ddppo_create(cfg)
    try:
        flat = I.params(nc, 20 + base).float()
        B.ddppo_set_params(h, flat.cuda())
        g = torch.Generator().manual_seed(base)
        obs = torch.rand(N, 1, 8, 8, generator=g).repeat_interleave(8, 2).repeat_interleave(8, 3)
        obs = (0.8 * obs + 0.2 * torch.rand(N, 1, 64, 64, generator=g)).cuda()
        F = OP.feature_dim(nc)
        dfeat = torch.randn(N, F, generator=g).cuda()
        feat, grad = torch.zeros(N, F, device="cuda"), torch.zeros(flat.numel(), device="cuda")
        B.ddppo_encoder_forward(h, N, obs, feat)
        B.ddppo_encoder_backward(h, dfeat, grad)
        assert B.ddppo_device_status(h) == 0
        p = flat.double().cuda().requires_grad_(True)
        ref, feat_r = torch.zeros_like(p), []
        for o, d in zip(obs.split(64), dfeat.split(64)):
            f = OP.encoder(OP.unflatten(p, nc), o.double(), nc)
            ref += torch.autograd.grad(f, p, d.double())[0]
            feat_r.append(f.detach())
        feat_r = torch.cat(feat_r)
        assert (feat.double() - feat_r).abs().max() <= 1e-4 * feat_r.abs().max()
        got, want = OP.unflatten(grad.double(), nc), OP.unflatten(ref, nc)
        for name in got:
            if name.startswith(("stem.", "b", "cmp.")):
                err = (got[name] - want[name]).norm() / want[name].norm()
                assert err <= 3e-2, (name, err.item())
    finally:
        B.ddppo_destroy(h)
