"""Host model of the LSTM cluster kernels' step exchange and of its drain after an abort, run on
the kernels' own step arithmetic (cluster_steps.cuh, compiled by the host compiler).

The protocol, restated: CTA i at step t waits for the blocks of all CTAs in buffer t & 1, arms
that barrier for step t + 2, and sends its block of step t + 1 to every CTA; blocks land in any
order. A wait that runs out, or the timeout flag seen in one, stops a CTA at its step t. Once
all have stopped, a CTA that gave up counts the blocks of steps t and t + 1 that never come as
delivered and waits for the phase. Random interleavings and aborts check that each of those
waits starts before and ends with the last block in flight, and that nothing is in flight to a
CTA that leaves. An mbarrier phase completes when its one arrival (the arming) and all bytes
armed have come; a wait on parity p returns once the completed-phase count c has c & 1 != p."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_00357_gb300", "csrc")

WRAP = r"""
#include "cluster_steps.cuh"
extern "C" int bar(int s) { return ddppo::step_bar(s); }
extern "C" int parity(int s) { return (int)ddppo::step_parity(s); }
extern "C" int missing(const int* sent, int ctas, int s, int T) {
  return ddppo::step_missing(sent, ctas, s, T);
}
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("steps")
    (d / "w.cpp").write_text(WRAP)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "w.cpp"), "-o",
                    str(d / "w.so")], check=True)
    return ctypes.CDLL(str(d / "w.so"))


class Bar:
    def __init__(self):
        self.done, self.pending, self.tx = 0, 1, 0

    def _settle(self):
        if self.pending == 0 and self.tx == 0:
            self.done += 1
            self.pending = 1

    def arm(self, blocks):
        assert self.pending == 1  # one arrival a phase
        self.pending -= 1
        self.tx += blocks
        self._settle()

    def land(self, blocks=1):
        self.tx -= blocks
        self._settle()

    def ready(self, parity):
        return (self.done & 1) != parity


def _run(L, ctas, T, seed, abort_at):
    rnd = random.Random(seed)
    bars = [[Bar(), Bar()] for _ in range(ctas)]
    for b in bars:
        if T > 1:
            b[L.bar(1)].arm(ctas)
        if T > 2:
            b[L.bar(2)].arm(ctas)
    t = [0] * ctas            # the step a CTA is in
    waited = [True] * ctas    # its wait is over
    out, failed = [False] * ctas, [False] * ctas
    flying = []               # (destination, step)
    ticks, flag = 0, False

    def land(k):
        dst, s = flying.pop(k)
        bars[dst][L.bar(s)].land()

    while not all(out):
        ticks += 1
        if flying and rnd.random() < 0.5:
            land(rnd.randrange(len(flying)))
        i = rnd.randrange(ctas)
        if out[i]:
            continue
        if not waited[i]:
            if bars[i][L.bar(t[i])].ready(L.parity(t[i])):
                assert (i, t[i]) not in flying
                if t[i] + 2 < T:
                    bars[i][L.bar(t[i])].arm(ctas)
                waited[i] = True
            elif ticks >= abort_at:   # a run-out, or a peer's flag seen while waiting
                flag = True
            if flag and rnd.random() < 0.3:  # (some threads of a CTA may have seen the flag
                out[i] = failed[i] = True    # though its first thread's wait went well)
            continue
        if t[i] + 1 < T:
            flying += [(d, t[i] + 1) for d in range(ctas)]
            t[i] += 1
            waited[i] = False
        else:
            out[i] = True
    sent = (ctypes.c_int * ctas)(*[min(v, T - 1) for v in t])
    assert max(sent) - min(sent) <= 1
    for i in range(ctas):
        if not failed[i]:
            assert all(d != i for d, _ in flying)
            continue
        for s in (t[i], t[i] + 1):
            miss = L.missing(sent, ctas, s, T)
            mine = [k for k, f in enumerate(flying) if f == (i, s)]
            if miss < 0:
                assert not mine
                continue
            b = bars[i][L.bar(s)]
            if miss:
                b.land(miss)
            while (i, s) in flying:
                assert not b.ready(L.parity(s))  # not over before the last block is in
                land(flying.index((i, s)))
            assert b.ready(L.parity(s))          # ... and over then
        assert all(d != i for d, _ in flying)    # nothing can land once the CTA has left
    return any(failed), t


@pytest.mark.parametrize("ctas", [2, 4, 8, 16])
def test_drain_waits_for_every_block_in_flight(steps, ctas):
    stops = set()
    for seed in range(400):
        failed, t = _run(steps, ctas, 1 + seed % 14, seed * 37 + ctas, 4 * ctas + seed * 1009 % (30 * ctas * ctas))
        if failed:
            stops |= set(t)
    assert {1, 2, 3, 4, 5, 6, 7} <= stops  # odd and even phases of both barriers


def test_no_abort_leaves_nothing(steps):
    for seed in range(50):
        failed, t = _run(steps, 4, 9, seed, 10 ** 9)
        assert not failed and t == [8] * 4
