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


@pytest.mark.parametrize("k,d", [(50, 1 << 20), (50, 1 << 25), (53, 1 << 26), (53, (1 << 28) - 1), (54, 1),
                                 (54, (1 << 28) - 1), (59, 1), (60, (1 << 28) - 1)])
@pytest.mark.parametrize("nearest", [False, True])
def test_conversions(k, d, nearest):
    """Key switches whose conversions fold, on both sides of the size of d where
    they stop (53 bits: between 2^26 and 2^28; 50 bits: 2^20 and 2^25)."""
    q, step = [], -1 if d == 1 else 1
    while len(q) < 5:
        q.append(prime_near(12, k, (1 << k) - q[-1] - 2 * step if q else d, step))
    p = [prime_near(12, 60, 1, -1)]
    while len(p) < 2 or p[-1] in q:
        p.append(prime_near(12, 60, (1 << 60) - p[-1] + 2, -1))
    p = [x for x in p if x not in q][:2]
    g, o = Context(12, q, p, 2), oracle.Context(12, q, p, 2)
    assert g.tensor_bconv
    g.set_rounding(nearest)
    o.set_rounding(nearest)
    st = si.Stream(1950 + k)
    a = np.stack([si.uniform_poly(st, q, o.N) for _ in range(2)])
    b = np.stack([si.uniform_poly(st, q, o.N) for _ in range(2)])
    a[:, :, ::5] = np.array(q, dtype=np.uint64)[:, None] - 1
    key = np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(2)])
    out = torch.empty_like(to_device(a))
    g.hmult(to_device(a), to_device(b), 5, g.relin_key(to_device(key)), out)
    assert np.array_equal(to_host(out).reshape(a.shape), o.hmult(a, b, key))
    g.close()
