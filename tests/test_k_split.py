"""The split of K's reduction range (csrc/ksplit.cuh, host arithmetic): the partial sums
sized for a largest range hold those of every shorter one, although fewer
orbitals can need more splits."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2404_09452_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "ksplit.cuh"
using namespace dfjk;
int main(int, char **v) {
  KShape s;
  s.nao = std::atoi(v[1]);
  const int slices = std::atoi(v[2]), block = std::atoi(v[3]), most = std::atoi(v[4]);
  s.ordered = std::atoi(v[5]);
  s.tiles = k_tiles(s.nao, 128, 64);
  s.block_bytes = (size_t)(s.nao + 127) / 128 * 128 * slices * 2 * block;
  s.range_bytes = (size_t)64 << 20;
  const size_t n2 = (size_t)s.nao * s.nao;
  for (int nkb = 1; nkb <= most; ++nkb) {
    const KSplit p = k_split(s, nkb);
    const bool covers = (long long)p.n * p.per >= nkb && (long long)(p.n - 1) * p.per < nkb;
    std::printf("%d %d %zu %zu\n", covers, (int)p.partials, p.n * n2, k_part_doubles(s, nkb));
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("ksplit")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("ordered", [1, 0])
@pytest.mark.parametrize("nao,slices,block", [(1, 6, 1024), (60, 8, 384), (128, 6, 1024), (375, 6, 1024), (450, 6, 1024),
                                              (900, 6, 1024), (900, 8, 384), (1800, 6, 1024), (3000, 6, 1024)])
def test_partials_of_every_shorter_range_fit(program, nao, slices, block, ordered):
    out = subprocess.run([program, str(nao), str(slices), str(block), "700", str(ordered)], check=True, capture_output=True, text=True)
    rows = [[int(x) for x in line.split()] for line in out.stdout.splitlines()]
    assert len(rows) == 700 and all(r[0] for r in rows)
    need, have = 0, 0
    for _, partials, doubles, bound in rows:
        need = max(need, doubles if partials else 0)
        assert bound >= max(need, have)
        have = bound
        assert not ordered or bound * 8 <= 64 << 20


def test_fewer_orbitals_can_need_more_splits(program):
    out = subprocess.run([program, "375", "6", "1024", "98", "1"], check=True, capture_output=True, text=True)
    doubles = [int(line.split()[2]) for line in out.stdout.splitlines()]
    assert doubles[98 - 1] == 25 * 375**2 and doubles[77 - 1] == 26 * 375**2  # 104 and 82 orbitals at 25 atoms
