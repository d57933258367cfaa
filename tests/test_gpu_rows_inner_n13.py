"""GPU parity of the fused row pass and inner product with several digits at
logN = 13 (six row stages), which only batches reach: 88 extended limbs or
more.  Two to five digits, ragged last ones, ops at uneven levels, products and
rotations, 54- and 60-bit primes."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import (OP_HMULT, OP_ROTATE, Batch, Context, Op, find_primes, to_device, to_host,  # noqa: E402
                                    trace_enable, trace_read, trace_reset)


@pytest.mark.parametrize("L,K,dnum,bits", [(12, 6, 2, 54), (14, 5, 3, 60), (13, 4, 4, 54), (14, 3, 5, 54)])
def test_batch(L, K, dnum, bits):
    q = find_primes(13, bits, L)
    p = find_primes(13, 60, K, exclude=q)
    g, o = Context(13, q, p, dnum), oracle.Context(13, q, p, dnum)
    st = si.Stream(2400 + L + dnum)
    key = np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(dnum)])
    dk = to_device(key)
    rlk, rk = g.relin_key(dk), g.rotation_key(dk, 3)
    ops, refs = [], []
    for i, nl in enumerate((L, L - 1, L, L - 2, L, L, L)):
        a, b = (np.stack([si.uniform_poly(st, q[:nl], o.N) for _ in range(2)]) for _ in range(2))
        a[:, :, ::7] = np.array(q[:nl], dtype=np.uint64)[:, None] - 1
        da = to_device(a)
        if i % 2:
            ops.append(Op(OP_ROTATE, da, nl, torch.empty_like(da), key=rk, steps=3))
            refs.append(o.rotate(a, 3, key))
        else:
            ops.append(Op(OP_HMULT, da, nl, torch.empty_like(da), b=to_device(b), key=rlk))
            refs.append(o.hmult(a, b, key))
    assert sum(op.n_limbs + K for op in ops) >= 88
    batch = Batch(g, ops)
    trace_reset()
    trace_enable(True)
    batch.run()
    trace_enable(False)
    assert "k_rows_inner" in trace_read()
    for op, ref in zip(ops, refs):
        assert np.array_equal(to_host(op.out).reshape(ref.shape), ref)
    g.close()
