"""The rule that picks tiles and CTA pairs (host arithmetic): what kglm_configure sets for the
pairs holds for every product that can take them, and the split-K slices are the default
tile's whatever is chosen."""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_22188_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "tiling.h"
using namespace kglm;
int main() {
    const int Ms[] = {1, 127, 128, 129, 256, 300, 1000, 2048, 4100, 8192};
    const int Ns[] = {30, 128, 200, 257, 611, 1000, 2000, 5003, 20000};
    const int Ks[] = {1, 3, 17, 63, 157, 313};
    for (int M : Ms) for (int N : Ns) for (int nkb : Ks) for (int grad : {0, 1, 4, 16}) for (int pair : {-1, 0, 1}) {
        TileShape q{};
        q.M = q.Mb = M; q.N = N; q.nkb = nkb; q.na = q.nb = 1;
        q.max_bn = N > 256 ? 256 : (N + 15) / 16 * 16;
        q.def = grad || N <= 256 ? q.max_bn : 128;
        q.grad_splits = grad;
        q.can_pair = M > 128;
        q.pair = pair;
        const Tiling t = choose_tiling(q);
        q.pair = 0;
        const Tiling off = choose_tiling(q);
        std::printf("%d %d %d %d %d %d %d %d %d %d\n", M, N, nkb, grad, pair, q.can_pair, t.pair, t.splits, off.splits, t.bn);
    }
}
"""


@pytest.fixture(scope="module")
def choices(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiling")
    (d / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(d / "t.cpp"), "-o", str(d / "t")], check=True)
    out = subprocess.run([str(d / "t")], check=True, capture_output=True, text=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


@pytest.mark.parametrize("pair", [0, 1])
def test_pairs_as_configured(choices, pair):
    rows = [r for r in choices if r[4] == pair]
    assert len(rows) > 1000
    wrong = [r for r in rows if r[6] != (pair and r[5])]
    assert not wrong, (len(wrong), wrong[:5])


def test_split_and_width(choices):
    both = set()
    for M, N, nkb, grad, pair, can, got, splits, off, bn in choices:
        assert splits == off and 16 <= bn <= 256 and bn % 16 == 0
        if pair == -1:
            both.add(got)
            assert can or not got
    assert both == {0, 1}                          # the rule takes either where it may choose
