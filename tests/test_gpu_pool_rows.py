"""The stem's fused max pool and its backward with a thread's column of windows cut into
single rows (20 frames) and into ragged runs of three rows (120 frames, 32 rows): the same 20
frames in both batches give the same logits, and, with no gradient into the other 100, the
same parameter gradients.

FP32 form. Logits within 1e-4 of their scale (each is within 5e-5 of the exact ones). Encoder
gradients pass through ReLU masks and argmax choices that flip under any float32 rounding:
3e-2 relative L2, as for the full-width encoder against float64; a row read or written in the
wrong place changes them by order one."""
import pytest
import torch

from paper_1911_00357_gb300 import binding as B
from tests import inputs as I
from tests import test_gpu_policy as P

pytestmark = pytest.mark.gpu


def _run(E, mb, dl, dv):
    net = P.Net(P._cfg("resnet_small", E, 1, 0), seed=1)
    try:
        dev, _ = P._dev_inputs(net.cfg, mb)
        logits, values = torch.zeros(1, E, 4, device="cuda"), torch.zeros(1, E, device="cuda")
        B.ddppo_policy_evaluate(net.h, 1, E, dev["obs"][:1], dev["goal"][:1], dev["prev_a"][:1], dev["masks"][:1],
                                dev["h0"], dev["c0"], logits, values)
        grad = torch.zeros(net.P, device="cuda")
        B.ddppo_policy_backward(net.h, dl.cuda(), dv.cuda(), grad)
        torch.cuda.synchronize()
        return logits.cpu().double(), grad.cpu().double(), P.OP.param_spec(net.ncfg)
    finally:
        net.close()


def test_runs_of_rows():
    few, many = 20, 120
    ncfg = P.net_config_from(P._cfg("resnet_small", many, 1, 0))
    mb = I.minibatch(ncfg, T=1, E=many, seed=2)
    sub = {}
    for k, v in mb.items():
        env = next((i for i, n in enumerate(v.shape) if n == many), None) if hasattr(v, "shape") else None
        sub[k] = v if env is None else v.narrow(env, 0, few).contiguous()
    g = torch.Generator().manual_seed(3)
    dl, dv = torch.randn(1, few, 4, generator=g), torch.randn(1, few, generator=g)
    pad = lambda t, shape: torch.cat([t, torch.zeros(*shape)], 1)
    la, ga, spec = _run(few, sub, dl, dv)
    lb, gb, _ = _run(many, mb, pad(dl, (1, many - few, 4)), pad(dv, (1, many - few)))
    assert (la - lb[:, :few]).abs().max() <= 1e-4 * la.abs().max()
    off = 0
    for name, shp in spec:
        k = int(torch.tensor(shp).prod())
        a, b = ga[off:off + k], gb[off:off + k]
        off += k
        if torch.linalg.vector_norm(a) > 1e-8:
            assert torch.linalg.vector_norm(a - b) <= 3e-2 * torch.linalg.vector_norm(a), name
