"""Host tables of the deferred products (csrc/gather_table.hpp), compiled with g++, against brute force: every
place of the contribution buffer belongs to one node, a node's places are ascending (in colour order its
cells then add in the order of the colours), and both numberings of the places name the same (cell, slot)."""
import itertools
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_29621_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "gather_table.hpp"
int main() {
  int nc, nb, n, by_slot;
  if (std::scanf("%d %d %d %d", &nc, &nb, &n, &by_slot) != 4) return 1;
  std::vector<int32_t> cells((size_t)nc * nb), perm(nc), ptr, idx;
  for (auto& v : cells) if (std::scanf("%d", &v) != 1) return 1;
  for (auto& v : perm) if (std::scanf("%d", &v) != 1) return 1;
  const std::vector<int32_t> place = mfns::nodes_by_place(cells, nb, perm, by_slot != 0);
  mfns::gather_table(place, n, ptr, idx);
  for (const std::vector<int32_t>* v : {&place, (const std::vector<int32_t>*)&ptr, (const std::vector<int32_t>*)&idx}) {
    for (int32_t x : *v) std::printf("%d ", x);
    std::printf("\n");
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("gather")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(cells, perm, n, by_slot):
        inp = f"{len(cells)} {cells.shape[1]} {n} {int(by_slot)}\n" + " ".join(map(str, cells.ravel())) + "\n" + \
              " ".join(map(str, perm)) + "\n"
        out = subprocess.run([str(exe)], input=inp, capture_output=True, text=True, check=True).stdout.split("\n")
        return [np.array(line.split(), dtype=int) for line in out[:3]]
    return run


def _lattice(n, k):
    """Nodes per cell of n^3 cells of degree k (x fastest), and the cells' colours (parities)."""
    M = k * n + 1
    box = list(itertools.product(range(n), repeat=3))
    cells = np.array([[((k * c[0] + z) * M + k * c[1] + y) * M + k * c[2] + x
                       for z, y, x in itertools.product(range(k + 1), repeat=3)] for c in box])
    return cells, np.array([sum((v & 1) << i for i, v in enumerate(c[::-1])) for c in box]), M ** 3


@pytest.mark.parametrize("by_slot", [False, True])
@pytest.mark.parametrize("n,k", [(1, 1), (2, 1), (3, 2), (2, 3), (5, 1), (1, 4)])
def test_tables_of_a_lattice(harness, n, k, by_slot):
    cells, colour, nodes = _lattice(n, k)
    perm = np.argsort(colour, kind="stable")
    place, ptr, idx = harness(cells, perm, nodes, by_slot)
    nc, nb = cells.shape
    for e, g in enumerate(place):
        cell, slot = (e % nc, e // nc) if by_slot else (perm[e // nb], e % nb)
        assert cells[cell, slot] == g
    assert ptr[0] == 0 and ptr[-1] == len(idx) == nc * nb and sorted(idx) == list(range(nc * nb))
    for g in range(nodes):
        mine = idx[ptr[g]:ptr[g + 1]]
        assert list(mine) == [e for e in range(nc * nb) if place[e] == g]
        if not by_slot:  # one contribution per cell, cells by colour
            c = perm[mine // nb]
            assert len(set(c)) == len(c) and (np.diff(colour[c]) > 0).all()


def test_nodes_without_a_place_and_shared_masters(harness):
    """Hanging nodes have no place of their own; a cell may name a master twice."""
    cells = np.array([[0, 3, 3, 1], [3, 5, 0, 0]])
    place, ptr, idx = harness(cells, [1, 0], 7, False)
    assert list(place) == [3, 5, 0, 0, 0, 3, 3, 1]
    assert [list(idx[ptr[g]:ptr[g + 1]]) for g in range(7)] == [[2, 3, 4], [7], [], [0, 5, 6], [], [1], []]
