"""GAE and the PPO loss at the edges of their splits against the float64 oracle.

GAE splits T over 16 warps and the envs in tiles of 32: T below, at and above 16, an uneven
last warp, and the longest tile that fits in shared memory (908 steps). The loss splits the
samples over a cluster of 1 to 16 CTAs of 256 threads, then 1024 threads, then several
samples a thread.

Tolerances: 1e-5 relative for GAE's values, the loss' statistics and its gradients, as in
the tests at other sizes (fp32 sums of at most 908 discounted terms: error of a few 1e-6).
The entries of the means are of order one and the fp32 sums are trees over threads, so their
error stays near 1e-6 of the mean magnitude also at 40,000 samples.
"""
import numpy as np
import pytest
import torch

from oracle import rl as OR
from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu
DT = torch.float64


@pytest.mark.parametrize("T,E", [(1, 1), (15, 31), (16, 32), (17, 33), (31, 64), (908, 3)])
def test_gae_splits(T, E):
    rng = np.random.default_rng(T * 100 + E)
    r = rng.normal(size=(T, E)).astype(np.float32)
    d = (rng.random((T, E)) < 0.05).astype(np.uint8)
    v = (3 * rng.normal(size=(T + 1, E))).astype(np.float32)
    A_ref, R_ref = OR.gae(r, d, v, np.float32(0.99), np.float32(0.95))
    adv = torch.zeros(T, E, device="cuda")
    ret = torch.zeros(T, E, device="cuda")
    rt, dt, vt = (torch.from_numpy(x).cuda() for x in (r, d, v))
    B.ddppo_gae(rt, dt, vt, T, E, 0.99, 0.95, adv, ret)
    for got, ref in ((adv, A_ref), (ret, R_ref)):
        g = got.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(g - ref) <= 1e-5 * np.maximum(1.0, np.abs(ref)))


@pytest.mark.parametrize("n", [255, 257, 2049, 4096, 16385, 40000])
def test_loss_cluster_sizes(n):
    g = torch.Generator().manual_seed(n)
    logits = torch.randn(n, 4, generator=g)
    values, adv, ret = (torch.randn(n, generator=g) for _ in range(3))
    actions = torch.randint(0, 4, (n,), generator=g, dtype=torch.int32)
    lp = torch.log_softmax(logits.double(), -1).gather(1, actions.long().unsqueeze(1))[:, 0]
    old = (lp + 0.3 * torch.randn(n, generator=g, dtype=DT)).float()
    hp = OR.PPOHParams()
    stats, dl, dv = (torch.zeros(*k, device="cuda") for k in ((8,), (n, 4), (n,)))
    dev = [x.cuda() for x in (logits, values, actions, old, adv, ret)]
    B.ddppo_ppo_loss(n, *dev, hp.clip, hp.value_coef, hp.entropy_coef, stats, dl, dv)
    torch.cuda.synchronize()
    L, V = logits.double().requires_grad_(True), values.double().requires_grad_(True)
    loss, st = OR.ppo_loss(L, V, actions, old.double(), adv.double(), ret.double(), hp)
    gl, gv = torch.autograd.grad(loss, (L, V))
    s = stats.cpu().double()
    for i, key in enumerate(["loss", "policy_loss", "value_loss", "entropy", "clip_frac", "approx_kl"]):
        ref = st[key].item()
        assert abs(s[i].item() - ref) <= 1e-5 * max(1.0, abs(ref)), (key, s[i].item(), ref)
    for got, ref in ((dl, gl), (dv, gv)):
        assert (got.cpu().double() - ref).abs().max() <= 1e-5 * ref.abs().max()
