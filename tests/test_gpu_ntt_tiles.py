"""GPU parity of the NTT tiles with eight elements per thread, where they can
go wrong: passes whose stage counts leave each kind of last register round
(logN 13: 7 + 6 stages, 15: 8 + 7, 16: 8 + 8, 17: 9 + 8), primes that leave the
lazy ranges no room (61 bits, residues at q - 1) and ordinary ones, and the two
sides of the default choice by launch size."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes, to_device, to_host  # noqa: E402

EIGHT = 5       # the variant with eight elements per thread


@pytest.mark.parametrize("logN", [13, 15, 16, 17])
@pytest.mark.parametrize("bits", [40, 61])
def test_eight_elements_against_the_oracle(logN, bits):
    primes = find_primes(logN, bits, 3)
    g, o = Context(logN, primes[:2], primes[2:], 1), oracle.Context(logN, primes[:2], primes[2:], 1)
    g.set_tune_table(bytes([EIGHT]) * len(g.tune_table()))
    a = si.uniform_poly(si.Stream(1500 + logN), primes, o.N)
    a[1] = primes[1] - 1                     # every residue at its largest
    a[2, ::2] = primes[2] - 1
    idx = np.arange(3, dtype=np.int32)
    ev, co = o.ntt_limbs(a, idx), o.intt_limbs(a, idx)
    d = to_device(a)
    g.ntt(d, 0, 3)
    assert np.array_equal(to_host(d).reshape(a.shape), ev)
    d = to_device(a)
    g.intt(d, 0, 3)
    assert np.array_equal(to_host(d).reshape(a.shape), co)
    g.close()


@pytest.mark.parametrize("logN,n,batch", [(16, 30, 1), (16, 31, 1), (14, 30, 4), (14, 31, 4), (17, 15, 1), (17, 16, 1)])
def test_default_variant_gives_the_same_residues(logN, n, batch):
    """Both sides of the size where the default variant changes, against a fixed variant."""
    primes = find_primes(logN, 54, 31)
    g = Context(logN, primes, find_primes(logN, 60, 1), 8)
    st = si.Stream(1600 + n)
    a = np.stack([si.uniform_poly(st, primes[:n], g.N) for _ in range(batch)])
    got = []
    default = g.tune_table()
    for table in (default, bytes([2]) * len(default)):
        g.set_tune_table(table)
        d, e = to_device(a), to_device(a)
        g.ntt(d, 0, n, batch)
        g.intt(e, 0, n, batch)
        got.append((to_host(d), to_host(e)))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    g.close()
