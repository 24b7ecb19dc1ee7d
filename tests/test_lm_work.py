"""The LM head's split of (token chunk, vocabulary item) over the CTAs, as the
kernels compute it, compiled for the host."""
import subprocess

import pytest

from paper_2608_02438_gb300 import build

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <set>
#include <vector>
#include "lm_work.h"

// items of every CTA; checks that each (chunk, item) is taken once and that the
// chunk's CTAs own its first slots
static int check(int G, int NC, int NI)
{
    std::vector<std::vector<int>> seen(NC, std::vector<int>(NI, 0));
    std::vector<std::set<int>> slots(NC);
    std::vector<long> load(G, 0);
    for (int r = 0; r < G; ++r) {
        const xp::LmWork w(r, G, NC);
        for (int g = 0; g < w.groups; ++g) {
            const int c = w.chunk(g);
            if (c < 0 || c >= NC || !slots[c].insert(w.first(g)).second || w.first(g) >= G) return -1;
            for (int it = w.first(g); it < NI; it += w.step(g), ++load[r])
                if (seen[c][it]++) return -2;
        }
    }
    for (int c = 0; c < NC; ++c) {
        const int n = xp::LmWork(0, G, NC).slots(c);
        if ((int)slots[c].size() != n || *slots[c].rbegin() != n - 1) return -3;
        for (int it = 0; it < NI; ++it)
            if (!seen[c][it]) return -4;
    }
    return (int)*std::max_element(load.begin(), load.end());
}

int main()
{
    for (int G : {1, 2, 3, 7, 8, 9, 16, 147, 152})
        for (int NC = 1; NC <= 330; NC += NC < 40 ? 1 : 7)
            for (int NI : {1, 5, G, 594})
                std::printf("%d %d %d %d\n", G, NC, NI, check(G, NC, NI));
    return 0;
}
"""


@pytest.fixture(scope="module")
def loads(tmp_path_factory):
    d = tmp_path_factory.mktemp("lm_work")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + build.CSRC, "-o", str(d / "t"), str(d / "t.cpp")], check=True)
    out = subprocess.run([str(d / "t")], capture_output=True, text=True, check=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_every_item_is_taken_once(loads):
    assert len(loads) > 2000
    for G, NC, NI, load in loads:
        assert load >= 0, (G, NC, NI, load)


# A group of n chunks gives each chunk at least floor(G / n) CTAs, n <= 16: with
# 152 CTAs at most 152 / 14 / 10 - 1 = 8.6 % more than an even share, and one item
# from the remainder per group.
def test_no_token_count_leaves_a_chunk_short_of_ctas(loads):
    for G, NC, NI, load in loads:
        if G == 152 and NI == 594:
            assert load <= 1.086 * NC * NI / G + (NC + 15) // 16, (NC, load, NC * NI / G)
