"""The shared-memory layout of the low-order solves and the sizes their launches ask for
(csrc/tri_layout.cuh, compiled for the host): no GPU."""
import itertools
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <vector>
#include "paper_2011_05427_gb300/csrc/tri_layout.cuh"
using namespace trt;
int main()
{
    const int prec[3] = {0, TRT_LO_FP32, TRT_LO_PAIR};
    for (int n = 1; n <= 2048; ++n) {
        const TriLayout y = tri_layout(n);
        std::vector<int> s(n + 1);
        lo_slots(n, s.data());
        std::vector<char> used(y.S, 0);
        int bad = 0;
        for (int v : s) {
            if (v < 0 || v >= y.S || used[v]) bad = 1;
            else used[v] = 1;
        }
        std::printf("%d %d %d %d %zu", n, y.S, y.P, bad, grey_smem(n));
        for (int p : prec) std::printf(" %zu", lo_smem(p, n));
        std::printf("\n");
    }
    // several slabs in one launch: what it asks for
    const int sets[][3] = {%SETS%};
    for (auto &b : sets) {
        std::printf("batch %d %d %d", b[0], b[1], b[2]);
        for (int p : prec) {
            BatchSmem m;
            for (int n : b) m.add(p, n);
            std::printf(" %zu %zu %d", m.lo, m.grey, m.max_nx);
        }
        std::printf("\n");
    }
}
"""
SETS = [(60, 59, 58), (200, 199, 7), (256, 255, 3), (64, 33, 63), (257, 256, 255), (2048, 1, 2),
        (140, 90, 55), (2, 3, 5)]


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("tri")
    (d / "t.cpp").write_text(SRC.replace("%SETS%", ", ".join("{%d, %d, %d}" % s for s in SETS)))
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", ROOT, "-I", "/usr/local/cuda/include",
                           str(d / "t.cpp"), "-o", str(d / "t")])
    lines = subprocess.check_output([str(d / "t")], text=True).splitlines()
    one = {int(x[0]): [int(v) for v in x[1:]] for x in (q.split() for q in lines[:2048])}
    many = [[int(v) for v in q.split()[1:]] for q in lines[2048:]]
    return one, many


def test_slots_and_sizes(sizes):
    """Every row and face of 1 to 2048 cells has a slot of its own, and the arrays of a solve
    (6 of S slots and 3 P values; FP32 refined: 6 in both types; pair: a 7th array) and of the
    grey kernel fit what is asked for, within the 227 KB of a CTA."""
    one, _ = sizes
    for n, (S, P, bad, grey, fp64, fp32, pair) in one.items():
        assert not bad, n
        assert 1 <= P <= 128 and 2 * P <= max(n, 2), n
        assert fp64 >= 8 * (6 * S + 3 * P) and fp32 >= 12 * 6 * S + 4 * 3 * P, n
        assert pair >= 8 * max(7 * S, 6 * S + 3 * P), n
        assert grey >= 8 * (3 * n + 7 * 32 + 6 * S + 3 * P), n
        assert max(grey, fp64, fp32, pair) <= 227 * 1024, n


def test_batch_covers_every_slab(sizes):
    """A launch over slabs of different sizes asks for the most that any of them needs: the
    largest slab's own need is less where its cell count is even and at most 256 and a smaller
    one's is odd."""
    one, many = sizes
    short = 0
    for row, s in itertools.product(many, range(3)):
        ns, (lo, grey, mx) = row[:3], row[3 + 3 * s:6 + 3 * s]
        assert mx == max(ns)
        for n in ns:
            assert lo >= one[n][4 + s] and grey >= one[n][3], (ns, n)
        short += one[mx][4 + s] < lo
    assert short >= 9   # (60, 59, 58), (200, 199, 7) and (256, 255, 3) in every form
