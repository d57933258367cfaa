"""GPU parity of hoisted rotations run several at a time: counts around the
group sizes at each level (3 rotations at 12 limbs, where the scratch pool
bounds them, 4 below, for the MID set), both rounding modes, the integer
conversion (digits above 16 primes), and outputs that overlap one another,
which are written in order."""
import numpy as np
import pytest

import oracle
import seeded_inputs as si

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2507_04775_gb300 import Context, find_primes, to_device, to_host  # noqa: E402

P = si.MID


def make(nq=P.nq, nk=P.nk, dnum=P.dnum):
    q = find_primes(P.logN, P.q_bits, nq)
    p = find_primes(P.logN, P.p_bits, nk, exclude=q)
    return Context(P.logN, q, p, dnum), oracle.Context(P.logN, q, p, dnum)


def rand_key(st, o):
    return np.stack([np.stack([si.uniform_poly(st, o.primes, o.N) for _ in range(2)]) for _ in range(o.dnum)])


@pytest.mark.parametrize("nl,n_rot", [(12, 3), (12, 4), (7, 4), (7, 6), (5, 1), (1, 9)])
@pytest.mark.parametrize("nearest", [False, True])
def test_groups(nl, n_rot, nearest):
    g, o = make()
    g.set_rounding(nearest)
    o.set_rounding(nearest)
    st = si.Stream(1700 + 16 * nl + n_rot)
    a = np.stack([si.uniform_poly(st, o.primes[:nl], o.N) for _ in range(2)])
    steps = [(-1) ** k * (3 * k + 1) for k in range(n_rot)]
    keys = [rand_key(st, o) for _ in steps]
    da = to_device(a)
    outs = [torch.empty_like(da) for _ in steps]
    g.rotate_hoisted(da, nl, steps, [g.rotation_key(to_device(k), s) for k, s in zip(keys, steps)], outs)
    ref = o.rotate_hoisted(a, steps, keys)
    for k in range(n_rot):
        assert np.array_equal(to_host(outs[k]).reshape(a.shape), ref[k]), "rotation %d" % k
    g.close()


def test_integer_conversion():
    g, o = make(18, 18, 1)
    st = si.Stream(1790)
    a = np.stack([si.uniform_poly(st, o.primes[:18], o.N) for _ in range(2)])
    steps, keys = [1, 2, 3], [rand_key(st, o) for _ in range(3)]
    da = to_device(a)
    outs = [torch.empty_like(da) for _ in steps]
    g.rotate_hoisted(da, 18, steps, [g.rotation_key(to_device(k), s) for k, s in zip(keys, steps)], outs)
    for x, y in zip(outs, o.rotate_hoisted(a, steps, keys)):
        assert np.array_equal(to_host(x).reshape(a.shape), y)
    g.close()


def test_overlapping_outputs_are_written_in_order():
    g, o = make()
    nl, st = 4, si.Stream(1791)
    a = np.stack([si.uniform_poly(st, o.primes[:nl], o.N) for _ in range(2)])
    steps, keys = [1, 2, 3], [rand_key(st, o) for _ in range(3)]
    da = to_device(a)
    buf = torch.empty(3 * a.size // 2, dtype=torch.int64, device="cuda")
    shared, shifted = buf[:a.size], buf[a.size // 2:]
    rks = [g.rotation_key(to_device(k), s) for k, s in zip(keys, steps)]
    g.rotate_hoisted(da, nl, steps, rks, [shared, shared, shifted])
    ref = o.rotate_hoisted(a, steps, keys)
    assert np.array_equal(to_host(shifted).reshape(a.shape), ref[2])
    assert np.array_equal(to_host(shared[:a.size // 2]).reshape(a.shape[1:]), ref[1][0])
    g.close()
