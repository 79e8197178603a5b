"""The order in which the persistent prefill attention's CTAs take its work items,
on the host: every query tile is taken once, and no CTA's share is far above the mean."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MAIN = r"""
#include <cstdio>
#include <vector>
#include "attn_items.h"
using namespace fpk;
int main() {
  int B, S, H, Hkv, sms;
  while (std::scanf("%d %d %d %d %d", &B, &S, &H, &Hkv, &sms) == 5) {
    const PaPlan p = pa_plan(B, S, H, H / Hkv, sms);
    const int tiles = (S + kPaB - 1) / kPaB, g = std::min(p.items, sms);
    std::vector<int> seen((size_t)B * H * tiles);
    std::vector<double> share(g);
    double sum = 0;
    bool ok = true;
    for (int c = 0; c < g; ++c)
      for (int n = 0, i = pa_item(0, c, g); i < p.items; i = pa_item(++n, c, g)) {
        const PaItem w(i, S, H, Hkv, p);
        for (int j = 0; j < 2; ++j)
          if (w.key_tiles(j)) {
            ok = ok && w.kvh == w.h[j] / (H / Hkv) && w.key_tiles(j) == w.row0(j) / kPaB + 1;
            ++seen[((size_t)w.b * H + w.h[j]) * tiles + w.row0(j) / kPaB];
          }
        const double t = p.pair ? w.tiles() : (w.tiles() + 1) / 2;  // steps of the softmax groups
        share[c] += t;
        sum += t;
      }
    for (int v : seen) ok = ok && v == 1;
    double top = 0;
    for (double v : share) top = std::max(top, v);
    std::printf("%d %d %.4f\n", (int)ok, (p.items + sms - 1) / sms, top / (sum / g));
  }
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("items")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2501_13111_gb300", "csrc"),
                    str(d / "main.cpp"), "-o", str(d / "order")], check=True)

    def run(cases):
        text = "\n".join(" ".join(str(v) for v in c) for c in cases)
        out = subprocess.run([str(d / "order")], input=text, capture_output=True, text=True, check=True).stdout
        return [(bool(int(a)), int(b), float(c)) for a, b, c in (line.split() for line in out.splitlines())]

    return run


HEADS = [(32, 32), (40, 40), (64, 8), (32, 8), (24, 8), (8, 1)]


def test_every_tile_is_taken_once(order):
    cases = [(B, S, H, Hkv, 152) for H, Hkv in HEADS for B in (1, 3, 8, 32) for S in (129, 256, 300, 1000, 1153, 2177)]
    assert all(r[0] for r in order(cases))


def test_shares_are_even_over_many_rounds(order):
    """Prompts of 2 to 64 tiles, from few rounds of the SMs to a hundred.  A share can
    exceed the mean by the longest item (1 of 5 rounds of half its length on average),
    and by the end of a block, which nothing evens out."""
    cases = [(B, 128 * t - 7, H, Hkv, 152) for H, Hkv in HEADS for B in (4, 8, 16, 32) for t in range(2, 65)]
    seen = 0
    for c, (_, rounds, share) in zip(cases, order(cases)):
        if rounds >= 5:
            seen += 1
            assert share <= (1.2 if rounds >= 8 else 1.4), (c, rounds, share)
    assert seen > 800
