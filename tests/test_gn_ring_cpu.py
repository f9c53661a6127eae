"""The rule that sends a GroupNorm backward to the shared-memory ring (gn_ring.cuh), compiled by
the host compiler alone: over every accepted base width (multiples of 4 in [4, 128]), stage and
camera side, each mask-bit copy of an image that the rule accepts -- unit by unit, as the
producer issues them -- has a size and a start that are multiples of 16 bytes, and a unit fits
its slot. Base 32 and 64, the named workloads, must take the ring."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1911_00357_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "gn_ring.cuh"
int main() {
  for (int base = 4; base <= 128; base += 4)
    for (int stage = 0; stage < 4; ++stage)
      for (int side = 32; side <= 1024; side += 16) {
        int s = (side - 1) / 2 + 1;                              // stem
        for (int i = 0; i <= stage; ++i) s = (s - 1) / 2 + 1;    // pool, then stages 2 to 4
        const int C = base << stage, HW = s * s;
        std::printf("%d %d %d %d %d\n", base, C, HW, ddppo::ring_rows(C),
                    ddppo::ring_mask_copies_ok(HW, C) ? 1 : 0);
      }
}
"""


def test_every_accepted_copy_is_aligned(tmp_path):
    src, exe = tmp_path / "walk.cpp", tmp_path / "walk"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    rows = [tuple(map(int, l.split())) for l in
            subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    seen, took = set(), set()
    for base, C, HW, unit, ok in rows:
        if not ok or C > 512 or (C, HW) in seen:
            continue
        seen.add((C, HW))
        took.add(C)
        assert unit * C * 4 <= 2 * 4 * 1024 and unit * C // 4 <= 2 * 256, (C, "slot")
        assert HW * C // 4 % 16 == 0, (C, HW, "image")
        for p in range(0, HW, unit):
            cnt = min(unit, HW - p)
            assert cnt * C % 64 == 0 and p * C % 64 == 0, (base, C, HW, p)
    assert {32, 64, 128, 256, 512} <= took


def test_dispatch_uses_the_rule():
    text = open(os.path.join(CSRC, "gn.cu")).read()
    body = text[text.index("int ring_units("):]
    body = body[:body.index("\n}\n")]
    assert re.search(r"kind == MASK_POS && !ring_mask_copies_ok\(HW, C\)", body)
    assert "rows = kRingRows * P" in text  # the producer's unit is the rule's
