"""The rules that pick a transform's tile (csrc/ntt_rules.h), compiled on the
host: both sides of every line, for launches within and past the tune table."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_04775_gb300", "csrc")
FWD_COLS, FWD_ROWS, INV_ROWS, INV_COLS = range(4)
MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "ntt_rules.h"
int main()
{
    int kind, logN;
    long total;
    while (scanf("%d %d %ld", &kind, &logN, &total) == 3) printf("%d\n", ntt_default_variant(kind, logN, total));
}
"""


@pytest.fixture(scope="module")
def default_variant(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-o", str(d / "rules"), str(d / "main.cpp")], check=True)

    def ask(kind, logN, total):
        out = subprocess.run([str(d / "rules")], input="%d %d %d\n" % (kind, logN, total), capture_output=True,
                             text=True, check=True)
        return int(out.stdout)
    return ask


def threads(v, S):
    ct, le = [16, 8, 4, 4, 8, 4][v], 3 if v == 5 else 4
    return (min(ct, 8) if S >= 9 else ct) << S >> le


@pytest.mark.parametrize("logN", [13, 14, 15, 16, 17])
def test_large_launches_take_large_tiles(default_variant, logN):
    """A rule by elements holds past the 128 limbs that a table has entries for:
    the forward rows leave the one-wave tile, the tile is at least a warp, and
    twice the limbs never go back to the tile of small launches."""
    n = (1 << 26) >> logN
    assert n > 128 or logN > 15
    assert default_variant(FWD_ROWS, logN, n) != 5
    assert default_variant(FWD_COLS, logN, n) != 5
    S_row = {13: 6, 14: 7, 15: 7, 16: 8, 17: 8}[logN]
    for kind, S in ((FWD_ROWS, S_row), (INV_ROWS, S_row), (FWD_COLS, logN - S_row), (INV_COLS, logN - S_row)):
        left = False
        for total in range(1, 1025):
            v = default_variant(kind, logN, total) if total % 31 == 1 or total > 1020 else None
            if v is None:
                continue
            assert threads(v, S) >= 32
            assert not (left and v == 5)
            left = left or v != 5
