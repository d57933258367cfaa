"""Every form of the tensor-core conversion's epilogue against the oracle, on
sets that the rule for small conversions does not send to the integer kernel
(the launch trace says which kernel ran): primes below 2^48 among the targets
(any prime), all of at least 2^48 without folding transforms, folding
transforms whose conversion cannot fold, and folding conversions, on both
sides of the size of d = 2^k - q where each begins and ends; floor and nearest;
ragged last digits; the largest number of sources; uniform residues and all of
them at q - 1."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import (Context, find_primes, to_device, to_host, trace_enable, trace_read,  # noqa: E402
                                    trace_reset)

LOGN = 12


def below(k, d, step, n, exclude=()):
    """n primes 1 modulo 2N from 2^k - d on, upward (step 1) or downward (-1)."""
    m, out = 2 << LOGN, []
    x = (1 << k) - d
    x += (1 - x) % m if step > 0 else -((x - 1) % m)
    while len(out) < n:
        if oracle.is_prime(x) and x not in exclude:
            out.append(x)
        x += step * m
    return out


def check(q, p, dnum, levels, nearest):
    g, o = Context(LOGN, q, p, dnum), oracle.Context(LOGN, q, p, dnum)
    g.set_rounding(nearest)
    o.set_rounding(nearest)
    st = si.Stream(2300 + len(q) + q[0] % 997)
    key = np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(dnum)])
    rlk = g.relin_key(to_device(key))
    for nl in levels:
        a, b = (np.stack([si.uniform_poly(st, q[:nl], o.N) for _ in range(2)]) for _ in range(2))
        top = np.stack([np.full(o.N, x - 1, dtype=np.uint64) for x in q[:nl]])
        for x, y in ((a, b), (np.stack([top, top]), a)):
            out = torch.empty_like(to_device(x))
            trace_reset()
            trace_enable(True)
            g.hmult(to_device(x), to_device(y), nl, rlk, out)
            trace_enable(False)
            ran = trace_read()
            assert "k_bconv_tc" in ran and "k_bconv" not in ran, sorted(ran)
            assert np.array_equal(to_host(out).reshape(x.shape), o.hmult(x, y, key)), "%d limbs" % nl
        # the conversions by themselves, on the largest sources
        ext = torch.zeros(g.beta(nl) * (nl + o.nk) * o.N, dtype=torch.int64, device="cuda")
        g.modup(to_device(top), nl, ext)
        assert np.array_equal(to_host(ext).reshape(g.beta(nl), nl + o.nk, o.N), o.modup(top)), "modup, %d limbs" % nl
        wide = np.stack([np.full(o.N, x - 1, dtype=np.uint64) for x in list(q[:nl]) + list(p)])
        down = torch.zeros(nl * o.N, dtype=torch.int64, device="cuda")
        g.moddown(to_device(wide), nl, down)
        assert np.array_equal(to_host(down).reshape(nl, o.N), o.moddown(wide)), "moddown, %d limbs" % nl
    assert g.status() == 0
    g.close()


@pytest.mark.parametrize("bits,pbits", [(40, 50), (47, 47), (48, 48), (49, 49), (60, 61), (61, 61), (54, 60)])
@pytest.mark.parametrize("nearest", [False, True])
def test_prime_sizes(bits, pbits, nearest):
    """40/50 to 48 bits: any prime; 49 and 61: at least 2^48; 54/60: folding."""
    q = find_primes(LOGN, bits, 14)
    check(q, find_primes(LOGN, pbits, 4, exclude=q), 4, (14, 13, 10), nearest)


@pytest.mark.parametrize("k,d,step", [(50, 1 << 20, 1), (50, 1 << 25, 1), (53, 1 << 26, 1), (53, (1 << 28) - 1, 1), (54, 1, -1),
                                      (54, (1 << 28) - 1, 1), (54, (1 << 28) + 1, -1), (59, 1, -1), (60, (1 << 28) - 1, 1)])
@pytest.mark.parametrize("nearest", [False, True])
def test_folding_limits(k, d, step, nearest):
    """The conversion folds up to a d that depends on k (53 bits: between 2^26 and
    2^28; 50 bits: 2^20 and 2^25), the transforms below 2^28."""
    q = below(k, d, step, 14)
    check(q, below(60, 1, -1, 4, exclude=q), 4, (14, 13), nearest)


@pytest.mark.parametrize("bits,pbits", [(40, 50), (61, 61), (54, 60)])
@pytest.mark.parametrize("nearest", [False, True])
def test_most_sources(bits, pbits, nearest):
    """Sixteen sources in both conversions, the most that the byte sums hold."""
    q = find_primes(LOGN, bits, 32)
    check(q, find_primes(LOGN, pbits, 16, exclude=q), 2, (32, 17), nearest)
