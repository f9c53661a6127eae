"""The frame fill of the ray caster: pooled and plain frames, fp32 and bf16, written in pairs
and, into a buffer one element off its pair's boundary, singly: the same bits, nothing
written outside, and equal to the raw depth image pooled and normalised in the same order of
float32 operations."""
import pytest
import torch

from paper_1911_00357_gb300 import binding as B
from paper_1911_00357_gb300.presets import make_config
from tests.gpu_util import Env, obs_dtype

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [32, 96, 256])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("pool", [0, 1])
def test_pairs_and_singles(side, precision, pool):
    E = 5
    cfg = make_config("blind", num_envs=E, depth_h=side, depth_w=side, pool2x2=pool, precision=precision,
                      rollout_T=1, minibatches=1)
    env = Env(cfg)
    try:
        out = side >> pool
        n, dt = E * out * out, obs_dtype(cfg)
        goal, reward = torch.zeros(E, 3, device="cuda"), torch.zeros(E, device="cuda")
        done = torch.zeros(E, dtype=torch.uint8, device="cuda")
        actions = torch.ones(E, dtype=torch.int32, device="cuda")
        first = torch.zeros(E, 1, out, out, dtype=dt, device="cuda")
        got = []
        for off in (0, 1):
            buf = torch.full((n + 8,), -7.0, dtype=dt, device="cuda")
            view = buf[off:off + n].view(E, 1, out, out)
            assert view.data_ptr() % 8 == off * view.element_size()
            B.ddppo_env_reset(env.h, first, goal)
            B.ddppo_env_step(env.h, actions, view, goal, reward, done)
            torch.cuda.synchronize()
            assert (buf[:off] == -7).all() and (buf[off + n:] == -7).all()
            got.append(view[:, 0].clone())
        assert torch.equal(got[0], got[1])
        d = torch.as_tensor(env.get_depth()).cuda().float().view(E, side, side)
        inv = torch.tensor(1.0, device="cuda") / torch.tensor(cfg.max_depth_m, dtype=torch.float32, device="cuda")
        if pool:
            c = d[:, 0::2] + d[:, 1::2]
            d = (c[..., 0::2] + c[..., 1::2]) * 0.25
        assert torch.equal(got[0], (d * inv).to(dt))
    finally:
        env.close()
