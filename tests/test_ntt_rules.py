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
    int kind, logN, fold, operands, tuned;
    long total;
    unsigned char table[129];                        // an installed table: the limb count modulo NVAR
    for (int i = 0; i < 129; ++i) table[i] = (unsigned char)(i % NVAR);
    while (scanf("%d %d %d %ld %d %d", &kind, &logN, &fold, &total, &operands, &tuned) == 6)
        printf("%d\n", ntt_variant(table, 129, tuned, kind, logN, fold, (int)total, operands));
}
"""


@pytest.fixture(scope="module")
def variant(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-o", str(d / "rules"), str(d / "main.cpp")], check=True)

    def ask(kind, logN, totals, operands=False, tuned=False, fold=True):
        """The variant for one limb count, or for each of several."""
        many = [totals] if isinstance(totals, int) else list(totals)
        out = subprocess.run([str(d / "rules")], capture_output=True, text=True, check=True,
                             input="".join("%d %d %d %d %d %d\n" % (kind, logN, fold, t, operands, tuned)
                                           for t in many))
        got = [int(x) for x in out.stdout.split()]
        assert len(got) == len(many)
        return got[0] if isinstance(totals, int) else got
    return ask


def threads(v, S):
    ct, le = [16, 8, 4, 4, 8, 4][v], 3 if v == 5 else 4
    return (min(ct, 8) if S >= 9 else ct) << S >> le


@pytest.mark.parametrize("logN", [13, 14, 15, 16, 17])
def test_large_launches_take_large_tiles(variant, logN):
    """A rule by elements holds past the 128 limbs that a table has entries for:
    the forward rows leave the one-wave tile, the tile is at least a warp, and
    twice the limbs never go back to the tile of small launches."""
    n = (1 << 22) >> logN            # 64 limbs of logN = 16
    S_row = {13: 6, 14: 7, 15: 7, 16: 8, 17: 8}[logN]
    for kind, S, op in ((FWD_ROWS, S_row, 0), (FWD_ROWS, S_row, 1), (INV_ROWS, S_row, 0), (FWD_COLS, logN - S_row, 0),
                        (INV_COLS, logN - S_row, 0)):
        got = variant(kind, logN, range(1, 1025), op)
        assert min(threads(v, S) for v in got) >= 32
        if 5 in got and got[-1] != 5:
            first = next(i for i, v in enumerate(got) if v != 5)
            assert 5 not in got[first:]
        assert got[n - 1] != 5


@pytest.mark.parametrize("fold", [True, False])
def test_lines(variant, fold):
    """The last limb count of the small-launch tile at logN = 16 and 17, per pass."""
    def last(kind, logN, operands=False):
        got = variant(kind, logN, range(1, 201), operands, fold=fold)
        return got.index(next(v for v in got if v != 5)) if set(got) != {5} else None

    assert [last(k, 16) for k in range(4)] == [22, 28 if fold else 32, 32, 23]
    assert [last(k, 17) for k in range(4)] == [11, 14 if fold else 16, 16, 11]
    assert last(FWD_ROWS, 16, True) == (56 if fold else None)


@pytest.mark.parametrize("logN", [13, 14, 15, 16, 17])
def test_an_installed_table_decides_every_pass(variant, logN):
    """Every entry is what runs, with and without an epilogue that reads
    operands, and the last one past the table's end; an entry equal to the
    default's leaves the default."""
    for kind in range(4):
        plain, own = variant(kind, logN, range(0, 300)), variant(kind, logN, range(0, 300), True)
        for operands in (False, True):
            got = variant(kind, logN, range(0, 300), operands, tuned=True)
            for i, v in enumerate(got):
                entry = min(i, 128) % 6
                assert v == (own[i] if operands and entry == plain[min(i, 128)] else entry)
