"""The instructions of a tensor-core digit product (csrc/digit_plan.cuh, the functions that the kernel's
issue loops are unrolled over), enumerated on the CPU for every slice count and column-tile width.

PTX orders two tcgen05.mma by their issue only if they have the same accumulator and the same shape,
so whatever two instructions add into a common column must have the same accumulator and N; an
exact chunk must keep every level's sum of digit products below 2^24; every kept slice pair is added
once, on its level."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1206_3768_gb300", "csrc")
DRIVER = r"""
#include <cstdio>
#include "digit_plan.cuh"
int main() {
  for (int S = 1; S <= 8; ++S)
    for (int w = 16; w <= digit::WIDEST; w += 16) {
      const int g = digit::group_levels(S, w), U = digit::region_levels(S, g, w);
      const int Ut = digit::region_levels(S, g, digit::widest_with(g));  // the unrolled loop's
      std::printf("plan %d %d %d %d %d %d %d %d\n", S, w, g, U, Ut, digit::zero_slices(g), digit::chunk_blocks(S),
                  digit::block_clocks(S, w));
      for (int s = 0; s < S; ++s)
        for (int i = 0; i < digit::groups(S, g); ++i) {
          const digit::Product q = digit::product(S, g, U, s, i);
          if (q.levels) std::printf("product %d %d %d %d %d\n", s, q.region, q.at, q.levels, q.first);
        }
    }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "plan.cpp").write_text(DRIVER)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "plan.cpp"), "-o", str(d / "plan")], check=True)
    out, cur = {}, None
    for line in subprocess.run([str(d / "plan")], check=True, capture_output=True, text=True).stdout.splitlines():
        kind, *v = line.split()
        v = [int(x) for x in v]
        if kind == "plan":
            cur = out[tuple(v[:2])] = dict(zip(("g", "U", "U_unrolled", "zeros", "chunk", "clocks"), v[2:]), products=[])
        else:
            cur["products"].append(tuple(v))
    assert len(out) == 8 * 4
    return out


def test_products_that_share_a_column_have_one_accumulator_and_shape(plans):
    for (S, w), p in plans.items():
        ranges = {(r, at * w, n * w) for _, r, at, n, _ in p["products"]}
        for r, c, n in ranges:
            assert r in (0, 1) and n % 16 == 0 and 16 <= n <= 256 and 0 <= c and c + n <= 256
            assert (r, c, n) == next(x for x in ranges if x[0] == r and x[1] == c)
            assert not any(r2 == r and c < c2 < c + n for r2, c2, _ in ranges)
        # the first slice reaches (and overwrites) every accumulator
        assert {(r, at * w, n * w) for s, r, at, n, _ in p["products"] if s == 0} == ranges
        # region 1 only where the levels do not fit region 0 (it is the other half of the chunks there)
        assert p["U"] == p["U_unrolled"] and (p["U"] == S) == (S * w <= 256)


def test_every_kept_slice_pair_once_on_its_level(plans):
    for (S, w), p in plans.items():
        pairs = []
        for s, r, at, n, first in p["products"]:
            for i in range(n):
                t, level = first + i, r * p["U"] + at + i
                assert -p["zeros"] <= t < S
                if t >= 0:
                    assert s + t == level
                    pairs.append((s, t))
        assert sorted(pairs) == [(s, t) for s in range(S) for t in range(S - s)]


def test_a_chunk_keeps_every_level_below_2_24(plans):
    for (S, w), p in plans.items():
        most = max(sum((129 if s == 0 else 64) * (129 if l - s == 0 else 64) for s in range(l + 1)) for l in range(S))
        assert p["chunk"] >= 1 and p["chunk"] * 64 * most < 2 ** 24 <= (p["chunk"] + 1) * 64 * most


def test_rings_hold_what_a_block_needs(plans):
    budget, a_tile = 227 * 1024 - 1024 - 512, 128 * 64 * 2
    for (S, w), p in plans.items():
        stage = (S + p["zeros"]) * w * 128
        a_tiles = (budget - 2 * stage) // a_tile  # two stages of B at least
        assert a_tiles >= (p["U"] + 1 if p["U"] < S else 2)
        assert p["clocks"] >= 4 * sum(max(n * w / 2, 32 + n * w / 4) for _, _, _, n, _ in p["products"]) - 1e-9
