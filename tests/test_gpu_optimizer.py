"""The optimizer step (norm, bias corrections, Adam) and the weights' operand copies.

Adam against float64 on the same fp32 inputs, two steps, at parameter counts that are not a
multiple of 4, with gradients at 16-byte aligned and unaligned addresses and a scale. Each
step rounds a dozen times (2^-24 each, relative to the larger of the two gradients where
the moments cancel), so a coordinate moves by lr within 1e-5 relative and keeps one
rounding of itself per step: |p - p64| <= 2e-5 lr + 2^-22 |p|.

The copies through what reads them: the FP32 forward of the 3-layer agent against the
float64 oracle (1e-4 of scale, the bound of the policy tests) where tiles are ragged: fewer
rows than a tile, feature maps with more pixels than a tile has columns."""
import pytest
import torch

from oracle import policy as OP
from paper_1911_00357_gb300 import binding as B
from paper_1911_00357_gb300.presets import make_config
from tests import inputs as I
from tests.gpu_util import net_config_from

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,offset,scale", [(8, 0, 1.0), (8, 1, 0.5), (24, 3, 1.0), (128, 0, 0.25),
                                                 (128, 2, 1.0)])
def test_adam_matches_float64(hidden, offset, scale):
    cfg = make_config("nature_fp32", num_envs=2, rollout_T=2, hidden=hidden)
    h = B.ddppo_create(cfg)
    try:
        flat = I.params(net_config_from(cfg), 1).float()
        P = flat.numel()
        B.ddppo_set_params(h, flat.cuda())
        g = torch.Generator().manual_seed(2)
        p, m, v = flat.double(), torch.zeros(P, dtype=torch.float64), torch.zeros(P, dtype=torch.float64)
        stats, out = torch.zeros(8, device="cuda"), torch.empty(P, device="cuda")
        hp = B.default_hparams()
        for t in (1, 2):
            gr = 1e-2 * torch.randn(P, generator=g)
            buf = torch.zeros(P + 4, device="cuda")
            buf[offset:offset + P] = gr.cuda()
            B.ddppo_apply_grad(h, buf[offset:offset + P], scale, hp, stats)
            gd = scale * gr.double()
            norm = gd.norm()
            assert abs(stats[6].item() - norm.item()) <= 1e-5 * norm.item()
            gd = gd * min(1.0, 0.5 / (norm.item() + 1e-6))
            m, v = 0.9 * m + 0.1 * gd, 0.999 * v + 0.001 * gd * gd
            p = p - 2.5e-4 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-5)
        B.ddppo_get_params(h, out)
        err = (out.cpu().double() - p).abs()
        assert (err <= 2e-5 * 2.5e-4 + 2.0 ** -22 * p.abs()).all(), err.max()
    finally:
        B.ddppo_destroy(h)


@pytest.mark.parametrize("hidden,depth", [(8, 64), (40, 128), (16, 256)])
def test_operand_copies(hidden, depth):
    E, T = 3, 2
    cfg = make_config("nature_fp32", num_envs=E, rollout_T=T, minibatches=1, hidden=hidden,
                      depth_h=depth, depth_w=depth)
    h = B.ddppo_create(cfg)
    try:
        ncfg = net_config_from(cfg)
        flat = I.params(ncfg, 5).float()
        B.ddppo_set_params(h, flat.cuda())
        mb = I.minibatch(ncfg, T=T, E=E, seed=6)
        d = {k: mb[k].float().cuda().contiguous() for k in ("obs", "goal", "h0", "c0")}
        prev_a, masks = mb["prev_a"].int().cuda(), mb["masks"].cuda()
        logits, values = torch.zeros(T, E, 4, device="cuda"), torch.zeros(T, E, device="cuda")
        B.ddppo_policy_evaluate(h, T, E, d["obs"], d["goal"], prev_a, masks, d["h0"], d["c0"], logits,
                                values)
        p = OP.unflatten(flat.double(), ncfg)
        lg, val = OP.sequence_forward(p, d["obs"].cpu().double(), d["goal"].cpu().double(), mb["prev_a"],
                                      mb["masks"], d["h0"].cpu().double(), d["c0"].cpu().double(), ncfg)[:2]
        for a, b in ((logits, lg), (values, val)):
            b = b.detach().reshape(a.shape)
            assert (a.cpu().double() - b).abs().max() <= 1e-4 * max(b.abs().max().item(), 1e-6)
    finally:
        B.ddppo_destroy(h)
