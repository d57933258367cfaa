"""GPU parity of key switches whose conversions go to the integer kernel because
they are small, on both sides of the rule (16, ten or six targets, eight at logN =
12) and with ragged last digits, whose jobs share a launch of the largest source
count: single operations, a batch and round-to-nearest."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import OP_HMULT, Batch, Context, Op, find_primes, to_device, to_host  # noqa: E402


@pytest.mark.parametrize("logN,L,K,dnum,levels", [
    (12, 10, 4, 3, (1, 4, 5, 8, 9, 10)), (13, 14, 5, 3, (4, 6, 11, 14)), (14, 7, 3, 3, (3, 4, 7)),
    (13, 12, 12, 1, (12, 7)), (13, 26, 13, 2, (13, 2)), (13, 20, 4, 5, (16, 17))])
@pytest.mark.parametrize("nearest", [False, True])
def test_small_conversions(logN, L, K, dnum, levels, nearest):
    q = find_primes(logN, 54, L)
    p = find_primes(logN, 60, K, exclude=q)
    g, o = Context(logN, q, p, dnum), oracle.Context(logN, q, p, dnum)
    g.set_rounding(nearest)
    o.set_rounding(nearest)
    st = si.Stream(2100 + logN + L)
    key = np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(dnum)])
    rlk = g.relin_key(to_device(key))
    ops, refs = [], []
    for nl in levels:
        a, b = (np.stack([si.uniform_poly(st, q[:nl], o.N) for _ in range(2)]) for _ in range(2))
        da, db = to_device(a), to_device(b)
        out = torch.empty_like(da)
        g.hmult(da, db, nl, rlk, out)
        refs.append(o.hmult(a, b, key))
        assert np.array_equal(to_host(out).reshape(a.shape), refs[-1]), "%d limbs" % nl
        ops.append(Op(OP_HMULT, da, nl, torch.empty_like(da), b=db, key=rlk))
    for part in (ops[:1], ops):                 # a batch of one (small) and of all
        Batch(g, part).run()
        for op, ref in zip(part, refs):
            assert np.array_equal(to_host(op.out).reshape(ref.shape), ref)
    g.close()
