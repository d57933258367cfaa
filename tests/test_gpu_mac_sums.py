"""GPU parity of the plaintext multiply-accumulate's two accumulators at the
line between them: n products of k-bit residues go by column sums up to
n = 2^(63 - k), by 128-bit sums above.  A linear transform of n diagonals with
no giant step is one such sum (and past 32 terms two, the second adding to the
first); plaintexts hold the largest residues."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes, to_device, to_host  # noqa: E402


@pytest.mark.parametrize("bits,n", [(61, 4), (61, 5), (60, 8), (60, 9), (57, 33), (40, 3), (54, 1)])
def test_sum_of_products(bits, n):
    q = find_primes(12, bits, 2)
    p = find_primes(12, bits, 1, exclude=q)
    g, o = Context(12, q, p, 2), oracle.Context(12, q, p, 2)
    st = si.Stream(1800 + 64 * bits + n)
    a = np.stack([si.uniform_poly(st, q, o.N) for _ in range(2)])
    a[0, :, ::3] = np.array(q, dtype=np.uint64)[:, None] - 1
    pts = [si.uniform_poly(st, q, o.N) for _ in range(n)]
    for t in pts:
        t[:, : o.N // 2] = np.array(q, dtype=np.uint64)[:, None] - 1
    keys = {b: np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(2)])
            for b in range(1, n)}
    da = to_device(a)
    out = torch.empty_like(da)
    g.linear_transform(da, 2, list(range(n)), [to_device(t) for t in pts], 64,
                       [g.rotation_key(to_device(k), b) for b, k in keys.items()], out)
    assert np.array_equal(to_host(out).reshape(a.shape), o.linear_transform(a, list(range(n)), pts, 64, keys))
    g.close()
