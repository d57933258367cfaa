"""GPU parity of the transforms on both sides of the lines where the default
tile changes, also past the 128 limbs that a tune table has entries for, against
a fixed tile, and the tile that the context reports there."""
import numpy as np
import pytest

import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes, to_device, to_host  # noqa: E402


# limbs of one polynomial, polynomials: on both sides of 22, 23, 28, 32 and 44
# limbs of logN = 16 (12 of logN = 17), and of 128 limbs
@pytest.mark.parametrize("logN,n,batches", [
    (16, 11, (2, 4, 5)), (16, 23, (1,)), (16, 24, (1,)), (16, 14, (2,)), (16, 29, (1,)), (16, 16, (2,)), (16, 33, (1,)),
    (17, 11, (1,)), (17, 12, (1,)), (17, 13, (1,)), (14, 16, (8, 14, 15)), (13, 20, (6, 7, 23))])
@pytest.mark.parametrize("bits", [54, 61])          # folding arithmetic, Shoup products
def test_both_sides_of_the_lines(logN, n, batches, bits):
    q = find_primes(logN, bits, n)
    g = Context(logN, q, find_primes(logN, bits, 1, exclude=q), n if n <= 8 else 4)
    st = si.Stream(2200 + n + bits)
    one = si.uniform_poly(st, q, g.N)
    for batch in batches:
        a = np.stack([np.roll(one, 17 * b, axis=1) for b in range(batch)])
        got = []
        default = g.tune_table()
        for table in (default, bytes([1]) * len(default)):
            g.set_tune_table(table)
            d, e = to_device(a), to_device(a)
            g.ntt(d, 0, n, batch)
            g.intt(e, 0, n, batch)
            got.append((to_host(d), to_host(e)))
        g.set_tune_table(default)
        assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1]), batch
    g.close()


@pytest.mark.parametrize("logN,limbs", [(13, 480), (14, 240)])
def test_reported_tile_past_the_table(logN, limbs):
    """A launch of more limbs than the table holds goes by its own size: the
    forward rows of 60 limbs of logN = 16 (and as many elements) leave the tile
    with eight elements per thread, whose target is 8 resident CTAs of 4 rows."""
    q = find_primes(logN, 54, 2)
    g = Context(logN, q[:1], q[1:], 1)
    small = g.ntt_tile(1, 60)
    assert g.ntt_tile(1, limbs) != small and g.ntt_tile(1, limbs) >> 8 == (8 if logN == 13 else 4)
    table = g.tune_table()
    g.set_tune_table(bytes([2]) * len(table))       # an installed table: its last entry beyond it
    assert g.ntt_tile(1, limbs) == g.ntt_tile(1, 128)
    g.set_tune_table(table)                          # the default one put back
    assert g.ntt_tile(1, limbs) != small and g.ntt_tile(1, 60) == small
    g.close()


def test_reported_tile_is_the_one_that_runs():
    """(tile width << 8) | resident CTAs: a context with Shoup arithmetic runs the
    wide tile as eight columns; 512-element columns (logN = 17) come eight at
    most, 64-element rows (logN = 13) keep the threads per SM; logN = 12 has one
    tile, of which two fit."""
    def tiles(logN, bits, v):
        q = find_primes(logN, bits, 2)
        g = Context(logN, q[:1], q[1:], 1)
        g.set_tune_table(bytes([v]) * len(g.tune_table()))
        got = [g.ntt_tile(k, 30) for k in range(4)]
        g.close()
        return [(t >> 8, t & 255) for t in got]

    assert tiles(16, 54, 0) == [(16, 3)] * 4
    assert tiles(16, 61, 0) == [(8, 6)] * 4
    assert tiles(16, 61, 3) == [(4, 12)] * 4
    assert tiles(16, 61, 4) == [(8, 8), (8, 6), (8, 6), (8, 6)]
    assert tiles(17, 54, 0) == [(8, 3), (16, 3), (16, 3), (8, 3)]
    assert tiles(13, 54, 5) == [(4, 16), (4, 32), (4, 32), (4, 16)]
    assert tiles(12, 54, 0) == [(1, 2)] * 4
