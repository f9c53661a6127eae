"""The calls that take no context, on several streams, threads and captured graphs at once: each
has scratch between two launches of one call (split-K sums, GroupNorm partials and counters, the
grouped weights' layout, the absolute maximum). Every result must be the bits of the same call
made alone: which scratch a call takes changes no arithmetic. 18 streams go past the 16 that
keep a buffer."""
import threading

import pytest
import torch

from paper_1911_00357_gb300 import binding as B

pytestmark = pytest.mark.gpu


def _wgrad(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(96, 16, 16, 64, device="cuda", generator=g).to(torch.bfloat16)
    dy = torch.randn(96, 16, 16, 64, device="cuda", generator=g).to(torch.bfloat16)
    dw = torch.zeros(64, 576, device="cuda")
    return lambda: (B.ddppo_conv2d_wgrad(x, dy, dw, 3, 1, 1), dw)[1]


def _gemm(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    a, b = (torch.randn(n, 8192, device="cuda", generator=g) for n in (40, 72))
    c = torch.zeros(40, 72, device="cuda")
    return lambda: (B.ddppo_gemm(a, b, c), c)[1]


def _norm(seed):  # a statistics launch, with a counter an image, and a normalise launch
    g = torch.Generator(device="cuda").manual_seed(seed)
    z = torch.randn(300, 400, 48, device="cuda", generator=g)
    one, nil = torch.ones(48, device="cuda"), torch.zeros(48, device="cuda")
    out, m, r = torch.zeros_like(z), torch.zeros(300, 24, device="cuda"), torch.zeros(300, 24, device="cuda")
    return lambda: (B.ddppo_group_norm(z, one, nil, out, m, r, relu=True), out)[1]


def _grouped(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(8, 16, 16, 128, device="cuda", generator=g)
    w = torch.randn(128, 4, 3, 3, device="cuda", generator=g)
    z = torch.zeros(8, 16, 16, 128, device="cuda")
    return lambda: (B.ddppo_grouped_conv3x3(x, w, z, 32, 1), z)[1]


def _quant(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = (1.0 + seed) * torch.randn(1 << 18, device="cuda", generator=g)
    q, sc = torch.zeros(1 << 18, dtype=torch.uint8, device="cuda"), torch.zeros(1, device="cuda")
    return lambda: (B.ddppo_quantize_e4m3(x, q, sc), q)[1]


CALLS = {"wgrad": _wgrad, "gemm": _gemm, "norm": _norm, "grouped": _grouped, "quant": _quant}


@pytest.mark.parametrize("call", list(CALLS))
def test_streams_do_not_share_scratch(call):
    runs = [CALLS[call](s) for s in range(18)]
    want = [r().clone() for r in runs]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in runs]
    for rep in range(6):
        got = []
        for r, s in zip(runs, streams):
            with torch.cuda.stream(s):
                got.append(r())
        torch.cuda.synchronize()
        for i, w in enumerate(want):
            assert torch.equal(got[i], w), (rep, i)
            got[i].zero_()
        torch.cuda.synchronize()


@pytest.mark.parametrize("call", list(CALLS))
def test_threads_on_one_stream(call):
    runs = [CALLS[call](s) for s in range(4)]
    want = [r().clone() for r in runs]
    torch.cuda.synchronize()
    stream, outs = torch.cuda.Stream(), [[] for _ in runs]

    def work(i):
        with torch.cuda.stream(stream):
            for _ in range(20):
                outs[i].append(runs[i]().clone())

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(runs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for i, w in enumerate(want):
        assert len(outs[i]) == 20 and all(torch.equal(o, w) for o in outs[i]), i


@pytest.mark.parametrize("call", list(CALLS))
def test_graphs_own_their_scratch(call):
    runs = [CALLS[call](s) for s in range(2)]
    want = [r().clone() for r in runs]
    torch.cuda.synchronize()
    graphs, outs = [], []
    for r in runs:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            outs.append(r())
        graphs.append(g)
    streams = [torch.cuda.Stream() for _ in runs]
    for _ in range(6):
        for o in outs:
            o.zero_()
        torch.cuda.synchronize()
        for g, s in zip(graphs, streams):
            with torch.cuda.stream(s):
                g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(o, w) for o, w in zip(outs, want))
