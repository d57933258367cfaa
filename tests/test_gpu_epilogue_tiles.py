"""GPU parity of the forward row passes with fused epilogues (ModDown, hoisted
ModDown, Rescale, the fused HMult + Rescale) on both sides of the size from
which their tiles run within 64 registers: 28 and 30 limbs of logN = 16 in one
launch, every tile against the eight-element one."""
import numpy as np
import pytest

import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes, to_device, to_host  # noqa: E402


@pytest.mark.parametrize("nl", [14, 15])
@pytest.mark.parametrize("bits", [54, 61])          # folding arithmetic, Shoup products
def test_epilogue_tiles(nl, bits):
    q = find_primes(16, bits, 16)
    g = Context(16, q, find_primes(16, 61 if bits == 61 else 60, 4, exclude=q), 4)
    st = si.Stream(1900 + nl)
    ct = [np.stack([si.uniform_poly(st, q[:nl], g.N) for _ in range(2)]) for _ in range(2)]
    key = np.stack([np.stack([si.uniform_poly(st, list(g.q) + list(g.p), g.N) for _ in range(2)]) for _ in range(4)])
    wide = np.stack([si.uniform_poly(st, q, g.N) for _ in range(2)])
    a, b, w, k = to_device(ct[0]), to_device(ct[1]), to_device(wide), to_device(key)
    rlk, rk = g.relin_key(k), [g.rotation_key(k, s) for s in (1, 5)]
    got = []
    for v in (5, 0, 1, 2, 3, 4):
        g.set_tune_table(bytes([v]) * len(g.tune_table()))
        out = [torch.empty_like(a) for _ in range(4)]
        lower = [torch.empty((2, n - 1, g.N), dtype=torch.int64, device="cuda") for n in (nl, nl, 16)]
        g.hmult(a, b, nl, rlk, out[0])
        g.rotate(a, nl, 5, rk[1], out[1])
        g.rotate_hoisted(a, nl, [1, 5], rk, out[2:])
        g.hmult_rescale(a, b, nl, rlk, lower[0])
        g.rescale(a, nl, lower[1])
        g.rescale(w, 16, lower[2])
        got.append([to_host(x) for x in out + lower])
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)
    g.close()
