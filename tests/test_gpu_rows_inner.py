"""GPU parity of the key switch whose row pass, inner product and inverse row
pass are one kernel, on both sides of the size where it starts (11 limbs of
logN = 16, here 22 of logN = 15) and of the digit count where it stops (5): an
odd and an even number of digits, ragged last digits, 60-bit primes (the
accumulators' general reduction), keys that are not 16-byte aligned, operands
that are not (the tensor product fused into the first inverse pass), and the
dropped limb of HMult fused with Rescale.  Passes of 7 and 8 row stages."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes, to_device, to_host  # noqa: E402


def offset(a, words):
    """A device copy of `a` that starts `words` words into its allocation."""
    buf = torch.empty(a.size + words, dtype=torch.int64, device="cuda")
    buf[words:] = to_device(a).flatten()
    return buf[words:]


@pytest.mark.parametrize("logN,L,K,dnum,bits,levels", [
    (15, 12, 10, 2, 54, (11, 12)), (15, 15, 12, 5, 60, (10, 13, 15)), (15, 18, 12, 6, 54, (18, 10)),
    (16, 6, 6, 3, 54, (6, 5, 1)), (15, 16, 16, 1, 59, (16, 7))])
def test_key_switch(logN, L, K, dnum, bits, levels):
    q = find_primes(logN, bits, L)
    p = find_primes(logN, 60, K, exclude=q)
    g, o = Context(logN, q, p, dnum), oracle.Context(logN, q, p, dnum)
    st = si.Stream(2000 + 7 * logN + L)
    key = np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(dnum)])
    rlk, rk = g.relin_key(offset(key, 1)), g.rotation_key(to_device(key), 3)
    for nl in levels:
        a, b = (np.stack([si.uniform_poly(st, q[:nl], o.N) for _ in range(2)]) for _ in range(2))
        a[:, :, ::7] = np.array(q[:nl], dtype=np.uint64)[:, None] - 1
        ref = o.hmult(a, b, key)
        out = torch.empty_like(to_device(a))
        g.hmult(to_device(a), to_device(b), nl, rlk, out)
        assert np.array_equal(to_host(out).reshape(a.shape), ref), "hmult, %d limbs" % nl
        g.rotate(to_device(a), nl, 3, rk, out)
        assert np.array_equal(to_host(out).reshape(a.shape), o.rotate(a, 3, key)), "rotate, %d limbs" % nl
        if nl > 1:
            res = torch.empty(2 * (nl - 1) * o.N, dtype=torch.int64, device="cuda")
            want = o.rescale(ref)
            for w in (0, 1):
                g.hmult_rescale(offset(a, w), to_device(b), nl, rlk, res)
                assert np.array_equal(to_host(res).reshape(want.shape), want), "hmult_rescale, %d limbs, %d" % (nl, w)
    g.close()
