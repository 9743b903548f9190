"""How the draining warps of the binary convolution divide the columns of the accumulators
(csrc/drain.cuh): plain arithmetic, compiled for the host and walked as the kernel walks it."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1603_05279_b200", "csrc")

# prints, for every plan, a line per warp: the (item, chunk) pairs it drains of 24 items
PROGRAM = r"""
#include <cstdio>
#include "drain.cuh"
int main() {
  for (int fused = 0; fused < 2; ++fused)
    for (int groups = 1 + fused; groups <= 16; groups += 1 + fused)
      for (int warps = 1; warps <= 3 && warps <= groups / (1 + fused); ++warps)
        for (int many_acc = 2; many_acc < 10; ++many_acc) {
          const int many = many_acc & 1, acc = many_acc / 2;
          const xnor::Drain d = xnor::plan_drain(groups, warps, many, fused, acc);
          for (int e = 0; e < d.split; ++e) {
            std::printf("%d %d %d %d %d %d %d:", fused, groups, warps, many, acc, d.chunk, d.chunks);
            int it = 0;
            for (int c = e;; c += d.split) {
              while (c >= d.chunks) { c = d.carry(c); ++it; }
              if (it >= 24) break;
              std::printf(" %d/%d", it, c);
            }
            std::printf("\n");
          }
        }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    """{(fused, groups, warps, many, accumulators): (groups of a chunk, chunks, [(item, chunk) ... of each warp])}"""
    d = tmp_path_factory.mktemp("drain")
    (d / "walk.cpp").write_text(PROGRAM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-I", CSRC, str(d / "walk.cpp"), "-o", str(d / "walk")], check=True)
    out = {}
    for line in subprocess.run([str(d / "walk")], check=True, capture_output=True, text=True).stdout.splitlines():
        head, _, tail = line.partition(":")
        *key, chunk, chunks = map(int, head.split())
        walk = [tuple(map(int, p.split("/"))) for p in tail.split()]
        out.setdefault(tuple(key), (chunk, chunks, []))[2].append(walk)
    return out


def test_every_chunk_is_drained_once(plans):
    for key, (chunk, chunks, walks) in plans.items():
        assert sorted(p for w in walks for p in w) == [(i, c) for i in range(24) for c in range(chunks)], key
        assert (chunks - 1) * chunk < key[1] <= chunks * chunk, key
        assert key[0] == 0 or chunk % 2 == 0, key


def test_no_warp_has_more_than_an_even_share(plans):
    """Over whole turns a warp drains no more than its share of every item in whole groups (fused: pairs)."""
    for (fused, groups, _, many, acc), (chunk, chunks, walks) in plans.items():
        unit = 2 if fused else 1
        share = -(-groups // unit // len(walks)) * unit
        for w in walks:
            assert sum(min(chunk, groups - c * chunk) for _, c in w) <= 24 * share, (fused, groups, many, acc)


def test_no_warp_waits_for_an_item_it_cannot_tell_from_an_earlier_one(plans):
    """A barrier's parity tells two consecutive uses of an accumulator apart."""
    for key, (_, _, walks) in plans.items():
        for w in walks:
            items = [-1] + sorted({i for i, _ in w})
            assert all(b - a <= key[4] for a, b in zip(items, items[1:])), key
