"""Performance cases of the DD-PPO hot path: the calls a training program makes, through the
binding of the C ABI, at the sizes of the named workloads (``presets.py``) and around them.

Every case is one layer, one block or one whole call of the synchronous
collect-then-update loop. ``listed`` holds the fixed ones, ``draw`` gives more over the
ranges they stand for, ``prepare`` makes a case's inputs and the worker it runs on,
``run`` is one pass, ``work`` its algorithmic bytes and operations, ``exact`` the same
outputs from plain float64 PyTorch.

The workers of the BF16 cases run with the GEMM autotuner frozen (its fixed heuristic), the
setting of a bit-reproducible run: tuned tile shapes may differ between two runs, and with
them the split of a K sum and every BF16 rounding downstream.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

from paper_1911_00357_gb300 import binding as B
from paper_1911_00357_gb300.presets import make_config

DEV = "cuda"
GAMMA, LAM = 0.99, 0.95
CLIP, VALUE_COEF, ENTROPY_COEF = 0.2, 0.5, 0.01


# ---------------------------------------------------------------- cases
def listed():
    return [
        # GAE over one rollout of the paper-shaped run (64 envs x 128 steps): the smallest
        # call of an iteration, once per update
        dict(name="gae_rollout", kind="gae", T=128, E=64),
        # the PPO loss with its exact gradient on one minibatch (128 steps x 32 envs), the
        # call behind the autograd wrapper
        dict(name="ppo_loss_minibatch", kind="ppo_loss", n=4096),
        # one optimizer step of the ResNet agent (8.5 M parameters): clip, Adam, and the
        # GEMM-layout weights every following forward reads; four times per iteration, and
        # once per exchanged gradient with several workers
        dict(name="optimizer_resnet", kind="optimizer", base_ch=32, hidden=512, layers=2),
        # one environment step of the paper-shaped run: 64 rooms-and-doors worlds, depth
        # 256x256 pooled to 128x128, next episodes prepared as the collect loop does
        dict(name="env_step_rooms", kind="env_step", E=64, gen=1, grid_min=128, grid_max=128,
             depth=256, pool=1, task=0),
        # one whole-agent inference step on 64 frames (128 times per rollout): the
        # latency-bound half of an iteration
        dict(name="act_resnet", kind="act", E=64, base_ch=32),
        # the 2 x 512 LSTM over one minibatch (128 steps x 32 envs), forward and
        # back-propagation through time, BF16 operands
        dict(name="lstm_train", kind="lstm", T=128, E=32, hidden=512, layers=2),
        # GroupNorm + residual + ReLU after a first-stage convolution, one minibatch
        dict(name="group_norm_stage1", kind="group_norm", N=4096, HW=1024, C=32, resid=True,
             relu=True),
        # first-stage 3x3 convolution of one minibatch (4096 frames, 32x32x32), BF16
        dict(name="conv_stage1", kind="conv", N=4096, H=32, W=32, C=32, Cout=32, k=3, s=1, p=1),
        # second-stage 3x3 convolution of the 64-base encoder at FP8 inference, 256 frames
        dict(name="conv_fp8_infer", kind="conv_fp8", N=256, H=16, W=16, C=128, Cout=128, k=3, s=1,
             p=1),
        # weight gradient of a second-stage 3x3 convolution of one minibatch, BF16
        dict(name="wgrad_stage2", kind="wgrad", N=4096, H=16, W=16, C=64, Cout=64, k=3, s=1, p=1),
        # the ResNet-18/32 encoder's training pass over one minibatch (4096 depth frames of
        # 128x128), forward and backward: the largest part of the update
        dict(name="encoder_train", kind="encoder", N=4096, base_ch=32),
        # the whole PPO update of the small FP32 workload: 16 envs x 32 steps, 3-layer
        # convolution, LSTM 128, 2 epochs x 2 minibatches
        dict(name="update_nature_fp32", kind="update", E=16, T=32),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _stage(rng, fp8=False):
    """(size, channels in, channels out, stride) of a 3x3 convolution of the ResNet encoders."""
    base = 64 if fp8 else rng.choice([32, 64])
    i = rng.randrange(4)
    size, c = 32 >> i, base << i
    if i < 3 and rng.random() < 0.25:
        return size, c, 2 * c, 2  # first convolution of the next stage
    return size, c, c, 1


def draw(rng):
    kind = rng.choice(["gae", "ppo_loss", "optimizer", "env_step", "act", "lstm", "group_norm",
                       "conv", "conv_fp8", "wgrad", "encoder", "update"])
    if kind == "gae":
        return dict(kind=kind, T=_log_int(rng, 8, 256), E=_log_int(rng, 1, 16384))
    if kind == "ppo_loss":
        return dict(kind=kind, n=_log_int(rng, 1, 131072))
    if kind == "optimizer":
        return dict(kind=kind, base_ch=rng.choice([32, 64]), hidden=64 * rng.randrange(2, 17),
                    layers=rng.randrange(1, 3))
    if kind == "env_step":
        gen, pool = rng.randrange(2), rng.randrange(2)
        # rooms and doors at 0.1 m, as in the mixed-grid workload; Bernoulli walls at 0.25 m
        g0 = rng.choice([64, 128, 256, 512] if gen else [32, 64, 128])
        return dict(kind=kind, E=_log_int(rng, 1, 1024), gen=gen, grid_min=g0,
                    grid_max=min(512 if gen else 128, g0 << rng.randrange(3)),
                    depth=rng.choice([64, 128] if not pool else [128, 256]), pool=pool,
                    task=rng.randrange(3))
    if kind == "act":
        return dict(kind=kind, E=_log_int(rng, 1, 256), base_ch=rng.choice([32, 32, 64]))
    if kind == "lstm":
        return dict(kind=kind, T=_log_int(rng, 8, 128), E=_log_int(rng, 2, 64),
                    hidden=rng.choice([128, 512, 512]), layers=rng.choice([1, 2, 2]))
    if kind == "group_norm":
        C = rng.choice([32, 64, 128, 256, 512, 2 * rng.randrange(4, 120)])
        HW = rng.choice([64 * 64, 32 * 32, 16 * 16, 8 * 8, 4 * 4, rng.randrange(1, 2000)])
        top = min(8192, max(1, 4096 * 1024 * 32 // (C * HW)))
        return dict(kind=kind, N=_log_int(rng, 1, top), HW=HW, C=C, resid=rng.random() < 0.5,
                    relu=rng.random() < 0.8)
    if kind in ("conv", "conv_fp8", "wgrad"):
        size, ci, co, s = _stage(rng, kind == "conv_fp8")
        H = W = size
        if kind == "conv" and rng.random() < 0.3:  # first stage of another camera shape
            ci = co = 32
            s, H, W = 1, rng.randrange(5, 48), rng.randrange(5, 48)
        # within the listed convolutions' operations and bytes
        top = max(1, min(4096, int(77e9 / (2 * 9 * ci * co * H * W / (s * s))),
                         int(134e6 / (H * W * ci))))
        return dict(kind=kind, N=_log_int(rng, 1, top), H=H, W=W, C=ci, Cout=co, k=3, s=s, p=1)
    if kind == "encoder":
        return dict(kind=kind, N=_log_int(rng, 16, 4000), base_ch=32)
    return dict(kind=kind, E=2 * _log_int(rng, 1, 16), T=_log_int(rng, 4, 48))


# ---------------------------------------------------------------- parameters
def _encoder_spec(kind, base, feat_hw):
    if kind == 0:
        return [("c1.w", (32, 1, 8, 8)), ("c1.b", (32,)), ("c2.w", (64, 32, 4, 4)), ("c2.b", (64,)),
                ("c3.w", (32, 64, 3, 3)), ("c3.b", (32,))], 32 * feat_hw
    spec = [("stem.w", (base, 1, 7, 7)), ("stem.g", (base,)), ("stem.b", (base,))]
    cin = base
    for i in range(4):
        w = base << i
        for r in range(2):
            n = "l%d.%d." % (i, r)
            spec += [(n + "c1.w", (w, cin, 3, 3)), (n + "n1.g", (w,)), (n + "n1.b", (w,)),
                     (n + "c2.w", (w, w, 3, 3)), (n + "n2.g", (w,)), (n + "n2.b", (w,))]
            if cin != w:
                spec += [(n + "d.w", (w, cin, 1, 1)), (n + "nd.g", (w,)), (n + "nd.b", (w,))]
            cin = w
    spec += [("cmp.w", (128, 8 * base, 3, 3)), ("cmp.g", (128,)), ("cmp.b", (128,))]
    return spec, 128 * feat_hw


def _spec(cfg):
    """The flat parameter order of the agent (net_kind 0 and 1)."""
    side = cfg.depth_h >> cfg.pool2x2
    hw = ((((side - 8) // 4 + 1) - 4) // 2 + 1 - 2) ** 2 if cfg.net_kind == 0 else (side // 32) ** 2
    spec, feat = _encoder_spec(cfg.net_kind, cfg.base_ch, hw)
    H = cfg.hidden
    spec += [("vis.w", (H, feat)), ("vis.b", (H,)), ("goal.w", (32, 3)), ("goal.b", (32,)),
             ("act.emb", (5, 32))]
    for l in range(cfg.lstm_layers):
        n = "lstm%d." % l
        spec += [(n + "w_ih", (4 * H, H + 64 if l == 0 else H)), (n + "w_hh", (4 * H, H)),
                 (n + "b_ih", (4 * H,)), (n + "b_hh", (4 * H,))]
    return spec + [("actor.w", (4, H)), ("actor.b", (4,)), ("critic.w", (1, H)), ("critic.b", (1,))]


def _params(cfg, gen):
    """Weights N(0, 1/fan_in), normalisation gains near 1, small biases."""
    parts = []
    for name, shape in _spec(cfg):
        r = torch.randn(shape, generator=gen, device=DEV)
        if name.endswith(".g"):
            r = 1.0 + 0.1 * r
        elif len(shape) == 1:
            r = 0.1 * r
        else:
            r = r / math.sqrt(math.prod(shape[1:]))
        parts.append(r.reshape(-1))
    return torch.cat(parts)


def _unflatten(flat, cfg):
    out, o = {}, 0
    for name, shape in _spec(cfg):
        k = math.prod(shape)
        out[name] = flat[o:o + k].view(shape)
        o += k
    return out


# ---------------------------------------------------------------- inputs
class _Worker:
    """A library context that is freed with the state that holds it."""

    def __init__(self, cfg):
        self.h = B.ddppo_create(cfg)

    def __del__(self):
        B.ddppo_destroy(self.h)


def _config(c):
    """The worker configuration of a case: its named workload, cut to the calls made."""
    k = c["kind"]
    if k == "optimizer":
        return make_config("resnet", base_ch=c["base_ch"], hidden=c["hidden"],
                           lstm_layers=c["layers"], num_envs=2, rollout_T=2)
    if k == "env_step":
        # the worlds and the camera alone: no encoder workspace
        return make_config("blind", num_envs=c["E"], gen_kind=c["gen"], grid_min=c["grid_min"],
                           grid_max=c["grid_max"], cell_m=0.1 if c["gen"] else 0.25,
                           depth_h=c["depth"], depth_w=c["depth"], pool2x2=c["pool"], task=c["task"], rollout_T=1,
                           minibatches=1)
    if k == "act":
        return make_config("resnet", base_ch=c["base_ch"], num_envs=c["E"], rollout_T=1,
                           minibatches=1)
    if k == "lstm":
        return make_config("resnet", num_envs=c["E"], hidden=c["hidden"], lstm_layers=c["layers"],
                           rollout_T=c["T"], minibatches=1, encoder_chunk=1)
    if k == "encoder":
        return make_config("resnet", base_ch=c["base_ch"], num_envs=1, rollout_T=c["N"],
                           minibatches=1)
    return make_config("nature_fp32", num_envs=c["E"], rollout_T=c["T"])  # update


def _observations(cfg, gen, n):
    """Depth frames as the camera makes them: a few flat regions, pixel noise, in [0, 1]."""
    side = cfg.depth_h >> cfg.pool2x2
    coarse = torch.rand(n, 1, 8, 8, generator=gen, device=DEV)
    x = coarse.repeat_interleave(side // 8, 2).repeat_interleave(side // 8, 3)
    x = (x + 0.05 * torch.rand(n, 1, side, side, generator=gen, device=DEV)).clamp_(0, 1)
    return x.to(torch.bfloat16) if cfg.precision else x


def _segment(cfg, gen, T, E):
    """Goals, previous actions, masks (rare episode starts) and the entering LSTM state."""
    rand = lambda *s: torch.rand(*s, generator=gen, device=DEV)
    ang = rand(T, E) * 2 * math.pi
    return dict(goal=torch.stack([10 * rand(T, E), torch.cos(ang), torch.sin(ang)], -1).contiguous(),
                prev_a=(rand(T, E) * 5).to(torch.int32).clamp_(0, 4),
                masks=(rand(T, E) > 0.02).to(torch.uint8),
                h0=0.3 * torch.randn(cfg.lstm_layers, E, cfg.hidden, generator=gen, device=DEV),
                c0=0.3 * torch.randn(cfg.lstm_layers, E, cfg.hidden, generator=gen, device=DEV))


def _e4m3(x):
    s = x.abs().max() / 448.0
    return (x / s).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8), s.reshape(1).float()


def _inputs(c, seed):
    """The tensors of a case, a function of the seed alone."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    randn = lambda *s: torch.randn(*s, generator=gen, device=DEV)
    rand = lambda *s: torch.rand(*s, generator=gen, device=DEV)
    k, d = c["kind"], {}
    if k == "gae":
        T, E = c["T"], c["E"]
        d.update(reward=0.25 * randn(T, E), done=(rand(T, E) < 0.01).to(torch.uint8),
                 value=randn(T + 1, E))
    elif k == "ppo_loss":
        n = c["n"]
        d.update(logits=randn(n, 4), values=randn(n), adv=randn(n), ret=randn(n),
                 actions=(rand(n) * 4).to(torch.int32).clamp_(0, 3))
        old = torch.log_softmax(d["logits"] + 0.2 * randn(n, 4), -1)
        d["logp_old"] = old.gather(1, d["actions"].long()[:, None])[:, 0].contiguous()
    elif k == "optimizer":
        cfg = _config(c)
        d["flat"] = _params(cfg, gen)
        d["grad"] = 1e-3 * randn(d["flat"].numel())
    elif k == "env_step":
        d["actions"] = (rand(64, c["E"]) * 3).to(torch.int32).clamp_(0, 2) + 1
        d["actions"][rand(64, c["E"]) < 0.005] = 0
    elif k == "act":
        cfg = _config(c)
        d.update(flat=_params(cfg, gen), obs=_observations(cfg, gen, c["E"]))
        d.update(_segment(cfg, gen, 1, c["E"]))
    elif k == "lstm":
        cfg = _config(c)
        T, E = c["T"], c["E"]
        d.update(flat=_params(cfg, gen), x=randn(T, E, c["hidden"] + 64).clamp_(min=0),
                 dy=0.01 * randn(T, E, c["hidden"]))
        d.update(_segment(cfg, gen, T, E))
    elif k == "group_norm":
        N, HW, C = c["N"], c["HW"], c["C"]
        d.update(z=randn(N, HW, C) + 0.3 * randn(1, 1, C), gamma=1 + 0.1 * randn(C),
                 beta=0.1 * randn(C), resid=randn(N, HW, C).clamp_(min=0) if c["resid"] else None)
    elif k in ("conv", "conv_fp8", "wgrad"):
        x = randn(c["N"], c["H"], c["W"], c["C"]).clamp_(min=0)  # after a ReLU
        fan = c["k"] ** 2 * c["C"]
        if k == "wgrad":
            Ho, Wo = _out(c)
            d.update(x=x.to(torch.bfloat16),
                     dy=(0.01 * randn(c["N"], Ho, Wo, c["Cout"])).to(torch.bfloat16))
        else:
            w = randn(c["Cout"], fan) / math.sqrt(fan)
            if k == "conv":
                d.update(x=x.to(torch.bfloat16), w=w.to(torch.bfloat16))
            else:
                (d["x"], d["sx"]), (d["w"], d["sw"]) = _e4m3(x), _e4m3(w)
    elif k == "encoder":
        cfg = _config(c)
        d.update(flat=_params(cfg, gen), obs=_observations(cfg, gen, c["N"]))
        d["dfeat"] = 1e-3 * randn(c["N"], 2048)
    else:  # update
        cfg = _config(c)
        T, E = c["T"], c["E"]
        d["flat"] = _params(cfg, gen)
        d["obs"] = _observations(cfg, gen, (T + 1) * E).view(T + 1, E, 1, cfg.depth_h, cfg.depth_w)
        d.update(_segment(cfg, gen, T, E))
        d.update(actions=(rand(T, E) * 4).to(torch.int32).clamp_(0, 3),
                 logp=math.log(0.25) + 0.3 * randn(T, E), adv=randn(T, E), ret=randn(T, E))
    return d


def _out(c):
    return tuple((v + 2 * c["p"] - c["k"]) // c["s"] + 1 for v in (c["H"], c["W"]))


def prepare(case, seed):
    c, k = dict(case), case["kind"]
    d = _inputs(c, seed)
    st = dict(case=c, **d)
    new = lambda *s: torch.empty(*s, device=DEV)
    if k in ("optimizer", "env_step", "act", "lstm", "encoder", "update"):
        cfg = _config(c)
        if k == "env_step":
            cfg.seed = seed
        st["worker"] = _Worker(cfg)
        h = st["h"] = st["worker"].h
        if cfg.precision:
            B.ddppo_autotune(h, False)
        if "flat" in d:
            B.ddppo_set_params(h, d["flat"])
    if k == "gae":
        st.update(out_adv=new(c["T"], c["E"]), out_ret=new(c["T"], c["E"]))
    elif k == "ppo_loss":
        st.update(stats=new(8), dl=new(c["n"], 4), dv=new(c["n"]))
    elif k == "optimizer":
        st.update(hp=B.default_hparams(), params=new(d["flat"].numel()), stats=torch.zeros(8, device=DEV))
    elif k == "env_step":
        side = c["depth"] >> c["pool"]
        E = c["E"]
        st.update(obs=torch.empty(E, 1, side, side, dtype=torch.bfloat16, device=DEV), goal=new(E, 3),
                  reward=new(E), done=torch.empty(E, dtype=torch.uint8, device=DEV), info=new(E, 4), t=0)
        B.ddppo_env_reset(h, st["obs"], st["goal"])
    elif k == "act":
        st.update(logits=new(1, c["E"], 4), values=new(1, c["E"]))
    elif k == "lstm":
        st.update(y=new(c["T"], c["E"], c["hidden"]), dx=torch.empty_like(d["x"]),
                  grad=new(d["flat"].numel()))
    elif k == "group_norm":
        st.update(out=torch.empty_like(d["z"]), mean=new(c["N"], c["C"] // 2),
                  rstd=new(c["N"], c["C"] // 2))
    elif k in ("conv", "conv_fp8"):
        st["y"] = new(c["N"], *_out(c), c["Cout"])
    elif k == "wgrad":
        st["dw"] = new(c["Cout"], c["k"] ** 2 * c["C"])
    elif k == "encoder":
        st.update(feat=new(c["N"], 2048), grad=new(d["flat"].numel()))
    elif k == "update":
        st.update(hp=B.default_hparams(), stats=torch.zeros(4, 8, device=DEV), k=0,
                  params=new(d["flat"].numel()))
        ro = st["ro"] = B.Rollout()
        for name in ("obs", "goal", "prev_a", "masks", "actions", "logp", "adv", "ret", "h0", "c0"):
            setattr(ro, name, d[name].data_ptr())
    return st


def run(st):
    c, k = st["case"], st["case"]["kind"]
    if k == "gae":
        B.ddppo_gae(st["reward"], st["done"], st["value"], c["T"], c["E"], GAMMA, LAM,
                    st["out_adv"], st["out_ret"])
        return st["out_adv"], st["out_ret"]
    if k == "ppo_loss":
        B.ddppo_ppo_loss(c["n"], st["logits"], st["values"], st["actions"], st["logp_old"],
                         st["adv"], st["ret"], CLIP, VALUE_COEF, ENTROPY_COEF, st["stats"],
                         st["dl"], st["dv"])
        return st["stats"], st["dl"], st["dv"]
    if k == "optimizer":
        B.ddppo_apply_grad(st["h"], st["grad"], 1.0, st["hp"], st["stats"])
        B.ddppo_get_params(st["h"], st["params"])
        return st["params"], st["stats"]
    if k == "env_step":
        B.ddppo_env_prefetch(st["h"])
        B.ddppo_env_step(st["h"], st["actions"][st["t"] % 64], st["obs"], st["goal"], st["reward"],
                         st["done"], st["info"])
        st["t"] += 1
        return st["obs"], st["goal"], st["reward"], st["done"], st["info"]
    if k == "act":
        B.ddppo_policy_evaluate(st["h"], 1, c["E"], st["obs"], st["goal"], st["prev_a"],
                                st["masks"], st["h0"], st["c0"], st["logits"], st["values"])
        return st["logits"], st["values"]
    if k == "lstm":
        B.ddppo_lstm_forward(st["h"], c["T"], c["E"], st["x"], st["masks"], st["h0"], st["c0"],
                             st["y"])
        B.ddppo_lstm_backward(st["h"], st["dy"], st["dx"], st["grad"])
        return st["y"], st["dx"], st["grad"]
    if k == "group_norm":
        B.ddppo_group_norm(st["z"], st["gamma"], st["beta"], st["out"], st["mean"], st["rstd"],
                           resid=st["resid"], relu=c["relu"])
        return st["out"], st["mean"], st["rstd"]
    if k == "conv":
        B.ddppo_conv2d(st["x"], st["w"], st["y"], c["k"], c["s"], c["p"])
        return st["y"]
    if k == "conv_fp8":
        B.ddppo_conv2d_e4m3(st["x"], st["w"], st["y"], c["k"], c["s"], c["p"], st["sx"], st["sw"])
        return st["y"]
    if k == "wgrad":
        B.ddppo_conv2d_wgrad(st["x"], st["dy"], st["dw"], c["k"], c["s"], c["p"])
        return st["dw"]
    if k == "encoder":
        B.ddppo_encoder_forward(st["h"], c["N"], st["obs"], st["feat"])
        B.ddppo_encoder_backward(st["h"], st["dfeat"], st["grad"])
        return st["feat"], st["grad"]
    st["hp"].update_index = st["k"]
    st["k"] += 1
    B.ddppo_ppo_update(st["h"], st["ro"], st["hp"], st["stats"])
    B.ddppo_get_params(st["h"], st["params"])
    return st["params"], st["stats"]


# ---------------------------------------------------------------- work
def _encoder_macs(kind, base, side):
    """Multiply-adds of one frame's encoder forward."""
    if kind == 0:
        a = (side - 8) // 4 + 1
        b = (a - 4) // 2 + 1
        return a * a * 32 * 64 + b * b * 64 * 512 + (b - 2) ** 2 * 32 * 576
    macs, s, cin = (side // 2) ** 2 * base * 49, side // 4, base
    for i in range(4):
        w, so = base << i, s >> (i > 0)
        macs += so * so * w * 9 * (cin + 3 * w) + (so * so * w * cin if cin != w else 0)
        s, cin = so, w
    return macs + s * s * 128 * 9 * cin


def work(case):
    c, k = case, case["kind"]
    if k == "gae":
        n = c["T"] * c["E"]
        return dict(bytes=17 * n + 4 * c["E"], flops=8 * n)
    if k == "ppo_loss":
        return dict(bytes=56 * c["n"] + 32, flops=80 * c["n"])
    if k == "optimizer":
        P = sum(math.prod(s) for _, s in _spec(_config(c)))
        # gradient, parameters and moments read; parameters and moments written; one BF16
        # copy for the contractions; the parameters returned
        return dict(bytes=(16 + 12 + 2 + 8) * P, flops=15 * P)
    if k == "env_step":
        side = c["depth"] >> c["pool"]
        # the observation written, one 32-cell-square neighbourhood of wall bits read at least,
        # state and scalars; a depth column takes a DDA walk of some 20 cells
        return dict(bytes=c["E"] * (2 * side * side + 128 + 130),
                    flops=c["E"] * (c["depth"] * 20 * 8 + c["depth"] ** 2 * 6))
    if k in ("act", "encoder", "update", "lstm"):
        cfg = _config(c)
        side = cfg.depth_h >> cfg.pool2x2
        P = sum(math.prod(s) for _, s in _spec(cfg))
        H, L = cfg.hidden, cfg.lstm_layers
        lstm = 4 * H * (H + 64 + H) + (L - 1) * 4 * H * 2 * H
        enc = _encoder_macs(cfg.net_kind, cfg.base_ch, side)
        es = 2 if cfg.precision else 4
        if k == "lstm":
            n = c["T"] * c["E"]
            w = sum(math.prod(s) for m, s in _spec(cfg) if m.startswith("lstm"))
            # x, dy read; y, dx and the whole flat gradient written; weights read per direction
            return dict(bytes=4 * n * (2 * (H + 64) + 2 * H) + 2 * es * w + 4 * P, flops=6 * n * lstm)
        if k == "encoder":
            n = c["N"]
            w = sum(math.prod(s) for _, s in _encoder_spec(1, c["base_ch"], 16)[0])
            return dict(bytes=n * (side * side * es * 2 + 2048 * 8) + 2 * es * w + 4 * P,
                        flops=6 * n * enc)
        feat = dict(_spec(cfg))["vis.w"][1]
        frame = enc + H * feat + lstm + 5 * H
        if k == "act":
            return dict(bytes=es * P + c["E"] * (side * side * es + 16 * L * H + 40),
                        flops=2 * c["E"] * frame)
        n = c["T"] * c["E"]
        # two epochs read the rollout; four optimizer steps over the parameters
        return dict(bytes=2 * n * (side * side * es + 40) + 4 * 28 * P, flops=2 * 6 * n * frame)
    if k == "group_norm":
        n = c["N"] * c["HW"] * c["C"]
        return dict(bytes=n * (12 if c["resid"] else 8) + 4 * c["N"] * c["C"], flops=8 * n)
    Ho, Wo = _out(c)
    nin, nout = c["N"] * c["H"] * c["W"] * c["C"], c["N"] * Ho * Wo * c["Cout"]
    nw = c["k"] ** 2 * c["C"] * c["Cout"]
    flops = 2 * c["N"] * Ho * Wo * nw
    if k == "wgrad":
        return dict(bytes=2 * nin + 2 * nout + 4 * nw, flops=flops)
    es = 1 if k == "conv_fp8" else 2
    return dict(bytes=es * (nin + nw) + 4 * nout, flops=flops)


# ---------------------------------------------------------------- float64
def _gn64(x, g, b):
    n, C, h, w = x.shape
    y = x.reshape(n, C // 2, -1)
    m = y.mean(-1, keepdim=True)
    y = (y - m) / torch.sqrt(((y - m) ** 2).mean(-1, keepdim=True) + 1e-5)
    return y.reshape(n, C, h, w) * g.view(1, C, 1, 1) + b.view(1, C, 1, 1)


def _conv64(x, w, s, p):
    """float64 convolution as an unfold and a matrix product."""
    n, _, h, wd = x.shape
    k = w.shape[2]
    cols = F.unfold(x, k, padding=p, stride=s)
    ho, wo = (h + 2 * p - k) // s + 1, (wd + 2 * p - k) // s + 1
    return (w.reshape(w.shape[0], -1) @ cols).view(n, w.shape[0], ho, wo)


def _encode64(p, obs, kind):
    if kind == 0:
        x = obs
        for n, s in (("c1", 4), ("c2", 2), ("c3", 1)):
            x = torch.relu(_conv64(x, p[n + ".w"], s, 0) + p[n + ".b"].view(1, -1, 1, 1))
        return x.flatten(1)
    x = torch.relu(_gn64(_conv64(obs, p["stem.w"], 2, 3), p["stem.g"], p["stem.b"]))
    x = F.max_pool2d(x, 3, 2, 1)
    for i in range(4):
        for r in range(2):
            n = "l%d.%d." % (i, r)
            s = 2 if i > 0 and r == 0 else 1
            y = torch.relu(_gn64(_conv64(x, p[n + "c1.w"], s, 1), p[n + "n1.g"], p[n + "n1.b"]))
            y = _gn64(_conv64(y, p[n + "c2.w"], 1, 1), p[n + "n2.g"], p[n + "n2.b"])
            if n + "d.w" in p:
                x = _gn64(_conv64(x, p[n + "d.w"], s, 0), p[n + "nd.g"], p[n + "nd.b"])
            x = torch.relu(y + x)
    return torch.relu(_gn64(_conv64(x, p["cmp.w"], 1, 1), p["cmp.g"], p["cmp.b"])).flatten(1)


def _lstm64(p, x, masks, h0, c0, L):
    for l in range(L):
        n = "lstm%d." % l
        gx = x @ p[n + "w_ih"].t() + (p[n + "b_ih"] + p[n + "b_hh"])
        h, c, ys = h0[l], c0[l], []
        for t in range(x.shape[0]):
            m = masks[t].double()[:, None]
            i, f, g, o = (gx[t] + (h * m) @ p[n + "w_hh"].t()).chunk(4, -1)
            c = torch.sigmoid(f) * (c * m) + torch.sigmoid(i) * torch.tanh(g)
            h = torch.sigmoid(o) * torch.tanh(c)
            ys.append(h)
        x = torch.stack(ys)
    return x


def _policy64(p, cfg, obs, goal, prev_a, masks, h0, c0):
    T, E = prev_a.shape
    feat = _encode64(p, obs.flatten(0, 1), cfg.net_kind).view(T, E, -1)
    x = torch.cat([torch.relu(feat @ p["vis.w"].t() + p["vis.b"]),
                   goal @ p["goal.w"].t() + p["goal.b"], p["act.emb"][prev_a.long()]], -1)
    y = _lstm64(p, x, masks, h0, c0, cfg.lstm_layers)
    return y @ p["actor.w"].t() + p["actor.b"], (y @ p["critic.w"].t() + p["critic.b"])[..., 0]


def _loss64(logits, values, actions, logp_old, adv, ret):
    lp = torch.log_softmax(logits, -1)
    la = lp.gather(-1, actions.long()[..., None])[..., 0]
    rho = torch.exp(la - logp_old)
    pol = -torch.minimum(rho * adv, rho.clamp(1 - CLIP, 1 + CLIP) * adv).mean()
    val = 0.5 * ((ret - values) ** 2).mean()
    ent = -(lp.exp() * lp).sum(-1).mean()
    frac = ((rho - 1).abs() > CLIP).double().mean()
    loss = pol + VALUE_COEF * val - ENTROPY_COEF * ent
    return loss, [loss, pol, val, ent, frac, (logp_old - la).mean()]


def _adam64(p, g, m, v, t, lr=2.5e-4, eps=1e-5, max_norm=0.5):
    norm = g.norm()
    g = g * min(1.0, max_norm / (norm.item() + 1e-6))
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    step = lr * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + eps)
    return p - step, m, v, norm


def _mix64(z):
    M = (1 << 64) - 1
    z = (z + 0x9E3779B97F4A7C15) & M
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M
    return z ^ (z >> 31)


def _permutation(seed, update, epoch, E):
    """The epoch's env order: Fisher-Yates over the counter hash."""
    perm = list(range(E))
    key = _mix64(_mix64(_mix64(seed)) + update)
    for i in range(E - 1, 0, -1):
        u = _mix64((key + ((7 << 40) | (epoch * E + i))) & ((1 << 64) - 1)) >> 32
        j = (u * (i + 1)) >> 32
        perm[i], perm[j] = perm[j], perm[i]
    return perm


def _exact_update(c, d):
    cfg = _config(c)
    T, E = c["T"], c["E"]
    q = {n: t.double() if t.is_floating_point() else t for n, t in d.items()}
    flat = q["flat"]
    m = v = torch.zeros_like(flat)
    stats, step, Emb = [], 0, E // 2
    for ep in range(2):
        perm = _permutation(int(cfg.seed), 0, ep, E)
        for mb in range(2):
            e = torch.tensor(perm[mb * Emb:(mb + 1) * Emb], device=DEV)
            th = flat.clone().requires_grad_(True)
            lg, val = _policy64(_unflatten(th, cfg), cfg, q["obs"][:T, e], q["goal"][:, e],
                                q["prev_a"][:, e], q["masks"][:, e], q["h0"][:, e], q["c0"][:, e])
            loss, s = _loss64(lg, val, q["actions"][:, e], q["logp"][:, e], q["adv"][:, e],
                              q["ret"][:, e])
            g, = torch.autograd.grad(loss, th)
            step += 1
            flat, m, v, norm = _adam64(flat, g, m, v, step)
            stats.append(torch.stack([x.detach() for x in s] + [norm, torch.zeros_like(norm)]))
    return flat, torch.stack(stats)


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "env_step":
        return None  # integer world; the ray cast is compared with itself
    d = _inputs(c, seed)
    if k == "gae":
        r, v, nd = d["reward"].double(), d["value"].double(), 1.0 - d["done"].double()
        A, adv = torch.zeros_like(v[0]), torch.empty_like(r)
        for t in range(c["T"] - 1, -1, -1):
            A = r[t] + GAMMA * nd[t] * v[t + 1] - v[t] + GAMMA * LAM * nd[t] * A
            adv[t] = A
        return adv, adv + v[:-1]
    if k == "ppo_loss":
        lg, val = d["logits"].double().requires_grad_(True), d["values"].double().requires_grad_(True)
        loss, s = _loss64(lg, val, d["actions"], d["logp_old"].double(), d["adv"].double(),
                          d["ret"].double())
        dl, dv = torch.autograd.grad(loss, (lg, val))
        z = torch.zeros_like(loss.detach())
        return torch.stack([x.detach() for x in s] + [z, z]), dl, dv
    if k == "optimizer":
        p = d["flat"].double()
        p, _, _, norm = _adam64(p, d["grad"].double(), 0 * p, 0 * p, 1)
        return p, torch.stack([0 * norm] * 6 + [norm, 0 * norm])
    if k == "act":
        cfg = _config(c)
        p = _unflatten(d["flat"].double(), cfg)
        return _policy64(p, cfg, d["obs"].double()[None], d["goal"].double(), d["prev_a"],
                         d["masks"], d["h0"].double(), d["c0"].double())
    if k == "lstm":
        cfg = _config(c)
        th, x = d["flat"].double().requires_grad_(True), d["x"].double().requires_grad_(True)
        y = _lstm64(_unflatten(th, cfg), x, d["masks"], d["h0"].double(), d["c0"].double(), c["layers"])
        g, dx = torch.autograd.grad(y, (th, x), d["dy"].double())
        return y.detach(), dx, g
    if k == "group_norm":
        outs = []
        for z, r in zip(d["z"].split(256), d["resid"].split(256) if c["resid"] else [None] * c["N"]):
            y = z.double().view(z.shape[0], c["HW"], c["C"] // 2, 2)
            m = y.mean((1, 3))
            rs = 1 / torch.sqrt(((y - m[:, None, :, None]) ** 2).mean((1, 3)) + 1e-5)
            o = ((y - m[:, None, :, None]) * rs[:, None, :, None]).reshape(z.shape)
            o = o * d["gamma"].double() + d["beta"].double() + (r.double() if r is not None else 0)
            outs.append((torch.relu(o) if c["relu"] else o, m, rs))
        return tuple(torch.cat(t) for t in zip(*outs))
    if k == "encoder":
        cfg = _config(c)
        p = _unflatten(d["flat"].double(), cfg)
        return torch.cat([_encode64(p, o.double(), 1) for o in d["obs"].split(128)]), None
    if k == "update":
        return _exact_update(c, d)
    # convolutions
    if k == "conv_fp8":
        x = d["x"].view(torch.float8_e4m3fn).double() * d["sx"].double()
        w = d["w"].view(torch.float8_e4m3fn).double() * d["sw"].double()
    else:
        x, w = d["x"], d.get("w")
    if k == "wgrad":
        dw = torch.zeros(c["Cout"], c["k"] ** 2 * c["C"], dtype=torch.float64, device=DEV)
        for xi, yi in zip(x.split(128), d["dy"].split(128)):
            cols = F.unfold(xi.double().permute(0, 3, 1, 2), c["k"], padding=c["p"], stride=c["s"])
            dw += torch.einsum("nop,nkp->ok", yi.double().flatten(1, 2).transpose(1, 2), cols)
        return dw.view(c["Cout"], c["C"], -1).transpose(1, 2).reshape(c["Cout"], -1)
    w = w.double().view(c["Cout"], c["k"], c["k"], c["C"]).permute(0, 3, 1, 2)
    return torch.cat([_conv64(xi.double().permute(0, 3, 1, 2), w, c["s"], c["p"]).permute(0, 2, 3, 1)
                      for xi in x.split(128)])
