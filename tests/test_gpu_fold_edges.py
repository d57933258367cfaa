"""GPU parity of the transforms where the folding arithmetic begins and ends:
primes 2^k - d of the smallest and largest sizes and on both sides of the light
and heavy ranges (58, 59 bits), d just below 2^28 (folding) and just above
(Shoup products), with residues at q - 1; every tile variant, every kind of
pass.  A context mixing both kinds of prime takes Shoup products throughout."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, to_device, to_host  # noqa: E402


def prime_near(logN, k, d, step):
    """The prime 1 modulo 2N nearest 2^k - d, walking up (step 1) or down (-1)."""
    m = 2 << logN
    x = (1 << k) - d
    x += (1 - x) % m if step > 0 else -((x - 1) % m)
    while not oracle.is_prime(x):
        x += step * m
    return x


def check(logN, primes):
    g, o = Context(logN, primes[:-1], primes[-1:], 1), oracle.Context(logN, primes[:-1], primes[-1:], 1)
    n = len(primes)
    a = si.uniform_poly(si.Stream(1900 + logN + primes[0] % 1000), primes, o.N)
    for i in range(n):
        a[i, i::3] = primes[i] - 1
    idx = np.arange(n, dtype=np.int32)
    ev, co = o.ntt_limbs(a, idx), o.intt_limbs(a, idx)
    size = len(g.tune_table())
    for v in range(6):
        g.set_tune_table(bytes([v]) * size)
        d, e = to_device(a), to_device(a)
        g.ntt(d, 0, n)
        g.intt(e, 0, n)
        assert np.array_equal(to_host(d).reshape(a.shape), ev), "forward, variant %d" % v
        assert np.array_equal(to_host(e).reshape(a.shape), co), "inverse, variant %d" % v
    g.close()


@pytest.mark.parametrize("logN", [12, 13, 15, 16, 17])
@pytest.mark.parametrize("inside", [True, False])
def test_edges(logN, inside):
    d, step = ((1 << 28) - 1, 1) if inside else ((1 << 28) + 1, -1)
    check(logN, [prime_near(logN, k, d, step) for k in (50, 58, 59, 60)])


def test_mixed_context():
    check(16, [prime_near(16, 54, 1, -1), prime_near(16, 61, 1, -1), prime_near(16, 40, 1, -1)])
