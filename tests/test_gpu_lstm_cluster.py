"""The whole-segment cluster forms of the LSTM recurrence (the default where covered).

BF16 forward: bit-identical with the step-by-step path, which single-step act passes take: the
values of a [T, E] evaluate equal those of T chained act passes where both form the input
projection by the same contraction (at most 64 rows, T E <= 64). Forward and backward: output and
gradients of the parameters and of the input against float64 autograd on the same inputs. Operands,
states and gate gradients are rounded to bf16 (relative 2^-9 each), so an element carries
a few such units and a tensor's relative L2 error stays below 2e-2; a wrong exchange,
slice or env would be an error of order one. FP32 operands: sums of at most 4 x 256 terms
over a few steps, each within some 1e-6 of its terms' size, so 2e-5. Sizes: one env, ragged
env counts per cluster, one wave of clusters and two, every covered hidden size, one step
(FP32), two and more."""
import pytest
import torch

from oracle import policy as OP
from paper_1911_00357_gb300 import binding as B
from paper_1911_00357_gb300.presets import make_config
from tests import inputs as I
from tests.gpu_util import net_config_from

pytestmark = pytest.mark.gpu

SHAPES = [(64, 1, 2, 1), (64, 2, 5, 64), (128, 1, 3, 7), (256, 2, 4, 17), (512, 1, 2, 57),
          (512, 2, 5, 32), (512, 1, 4, 64), (512, 2, 3, 9)]

SHAPES32 = [(64, 1, 1, 1), (64, 2, 5, 70), (128, 1, 3, 7), (128, 2, 4, 33), (256, 1, 4, 9),
            (256, 2, 2, 110)]


def _make(hidden, layers, T, E, precision=1):
    cfg = make_config("blind", num_envs=E, hidden=hidden, lstm_layers=layers, rollout_T=T,
                      minibatches=1, precision=precision)
    h = B.ddppo_create(cfg)
    ncfg = net_config_from(cfg)
    flat = I.params(ncfg, 3).float()
    B.ddppo_set_params(h, flat.cuda())
    return cfg, h, ncfg, flat


@pytest.mark.parametrize("hidden,layers,T,E", [s for s in SHAPES if s[2] * s[3] <= 64])
def test_forward_gives_the_bits_of_single_steps(hidden, layers, T, E):
    cfg, h, ncfg, _ = _make(hidden, layers, T, E)
    try:
        mb = I.minibatch(ncfg, T=T, E=E, seed=4)
        d = {k: mb[k].float().cuda().contiguous() for k in ("goal", "h0", "c0")}
        prev_a, masks = mb["prev_a"].int().cuda(), mb["masks"].cuda()
        obs = torch.zeros(T, E, 1, 128, 128, dtype=torch.bfloat16, device="cuda")
        logits, values = torch.zeros(T, E, 4, device="cuda"), torch.zeros(T, E, device="cuda")
        B.ddppo_policy_evaluate(h, T, E, obs, d["goal"], prev_a, masks, d["h0"], d["c0"], logits,
                                values)
        hs, cs = d["h0"].clone(), d["c0"].clone()
        u = torch.full((E,), 0.5, device="cuda")
        act = torch.zeros(E, dtype=torch.int32, device="cuda")
        logp, val = torch.zeros(E, device="cuda"), torch.zeros(E, device="cuda")
        for t in range(T):
            B.ddppo_policy_act(h, obs[t], d["goal"][t], prev_a[t], masks[t], hs, cs, u, act, logp, val)
            assert torch.equal(val, values[t]), t
        assert B.ddppo_device_status(h) == 0
    finally:
        B.ddppo_destroy(h)


@pytest.mark.parametrize("hidden,layers,T,E,precision",
                         [s + (1,) for s in SHAPES] + [s + (0,) for s in SHAPES32])
def test_gradients_match_float64(hidden, layers, T, E, precision):
    cfg, h, ncfg, flat = _make(hidden, layers, T, E, precision)
    lim = 2e-2 if precision else 2e-5
    try:
        g = torch.Generator().manual_seed(5)
        x = torch.randn(T, E, 64, generator=g)
        masks = (torch.rand(T, E, generator=g) > 0.2).to(torch.uint8)
        h0, c0 = (0.5 * torch.randn(layers, E, hidden, generator=g) for _ in range(2))
        dy = torch.randn(T, E, hidden, generator=g)
        y, dx = torch.zeros(T, E, hidden, device="cuda"), torch.zeros(T, E, 64, device="cuda")
        grad = torch.zeros(flat.numel(), device="cuda")
        # held until the backward has run: it reads the masks and the entering state again
        dev = [t.cuda() for t in (x, masks, h0, c0, dy)]
        B.ddppo_lstm_forward(h, T, E, *dev[:4], y)
        B.ddppo_lstm_backward(h, dev[4], dx, grad)
        assert B.ddppo_device_status(h) == 0
        p = OP.unflatten(flat.double(), ncfg)
        p = {k: v.clone().requires_grad_(k.startswith("lstm")) for k, v in p.items()}
        names = [k for k in p if k.startswith("lstm")]
        xr = x.double().requires_grad_(True)
        yr, hs = xr, []
        for l in range(layers):
            q = [p[n] for n in names[4 * l:4 * l + 4]]  # w_ih, w_hh, b_ih, b_hh
            hh, cc, out = h0[l].double(), c0[l].double(), []
            for t in range(T):
                m = masks[t].double()[:, None]
                i, f, gg, o = (yr[t] @ q[0].t() + (hh * m) @ q[1].t() + q[2] + q[3]).chunk(4, -1)
                cc = torch.sigmoid(f) * (cc * m) + torch.sigmoid(i) * torch.tanh(gg)
                hh = torch.sigmoid(o) * torch.tanh(cc)
                out.append(hh)
            yr = torch.stack(out)
        gr = torch.autograd.grad(yr, [xr] + [p[n] for n in names], dy.double())
        # (a gradient that is exactly zero -- one masked step -- has to be zero)
        rel = lambda a, b: (torch.linalg.vector_norm(a.cpu().double() - b) /
                            (torch.linalg.vector_norm(b) if b.any() else 1.0)).item()
        assert rel(y, yr.detach()) <= lim
        assert rel(dx, gr[0]) <= lim
        gp = OP.unflatten(grad.cpu().double(), ncfg)
        for n, r in zip(names, gr[1:]):
            assert rel(gp[n], r) <= lim, n
    finally:
        B.ddppo_destroy(h)
