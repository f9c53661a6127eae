"""A host thread's first call into the library: the tensor-core contractions encode tensor maps,
which need a current context in the calling thread, before they launch anything. Each call made
first thing in a new thread gives the bits it gives in this one."""
import threading

import pytest
import torch

from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _bf(*shape):
    return torch.randn(*shape, device="cuda").to(torch.bfloat16)


def _call(kind):
    if kind == "gemm":
        a, b, out = _bf(256, 512), _bf(128, 512), torch.zeros(256, 128, device="cuda")
        return lambda: B.ddppo_gemm(a, b, out), out
    if kind == "conv":
        x, w, out = _bf(8, 32, 32, 32), _bf(32, 288), torch.zeros(8, 32, 32, 32, device="cuda")
        return lambda: B.ddppo_conv2d(x, w, out, 3, 1, 1), out
    c = 64 if kind == "wgrad64" else 32
    x, dy, out = _bf(8, 16, 16, c), _bf(8, 16, 16, c), torch.zeros(c, 9 * c, device="cuda")
    return lambda: B.ddppo_conv2d_wgrad(x, dy, out, 3, 1, 1), out


@pytest.mark.parametrize("kind", ["gemm", "conv", "wgrad32", "wgrad64"])
def test_first_call_of_a_thread(kind):
    torch.manual_seed(1)
    call, out = _call(kind)
    call()
    want = out.clone()
    out.zero_()
    torch.cuda.synchronize()
    stream, errors = B._s(), []

    def work():
        try:
            keep, B._s = B._s, lambda s=None: stream  # (no torch call in the thread before ours)
            call()
        except Exception as e:
            errors.append(e)
        finally:
            B._s = keep

    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert torch.equal(out, want)
