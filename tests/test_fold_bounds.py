"""The ranges of the folding transforms, stage by stage, in whole numbers: every
sum stays below 2^64, every subtraction has a large enough multiple of q, and
every transform ends in the range its consumer takes, for each size of prime
that folds (50 to 60 bits, 2^k - q up to 2^28), each pass length and both tile
widths.  The schedule mirrors ntt_round in csrc/ntt.cuh."""
import pytest

LIMIT = 1 << 64


def rounds(S, LE, inv):
    out = []
    for rho in range(-(-S // LE)):
        partial = rho == -(-S // LE) - 1 and S % LE
        out.append(LE - S % LE if partial else 0)
    return out


class Prime:
    def __init__(self, k, d):
        self.k, self.d, self.q = k, d, (1 << k) - d
        self.heavy = k > 58
        self.bt = (2 << k) + (2 * d << 32)
        self.big = (self.bt // self.q + 1) * self.q
        self.K = (3 << 61) // self.q * self.q if k <= 58 else ((9 << 59) // self.q + 1) * self.q

    def fold(self, b):
        assert b <= LIMIT
        return min(b, (2 << self.k) + ((b - 1) >> (self.k + 1)) * 2 * self.d)

    def fold_2q(self, b):
        assert b <= LIMIT
        return (1 << self.k) + ((b - 1) >> self.k) * self.d

    def mul(self, b):
        assert b <= LIMIT       # the product takes any 64-bit value
        hi = ((1 << 32) * self.q + ((b - 1) >> 32) * self.q) >> (self.k + 1)
        assert hi < 1 << 32
        t = (2 << self.k) + hi * 2 * self.d
        assert t <= self.bt
        return t


def forward(p, S, LE, bound, first):
    x = [bound] * (1 << LE)
    for rho, A0 in enumerate(rounds(S, LE, False)):
        x = [max(x)] * len(x)                                   # an exchange
        for a in range(A0, LE):
            n, h = a - A0, (1 << LE) >> (a + 1)
            if (n == 0 and not (first and rho == 0)) or (n == 2 and p.heavy):
                x = [p.fold(b) if not r & h else b for r, b in enumerate(x)]
            y = list(x)
            for r in range(len(x)):
                if not r & h:
                    t = p.mul(x[r + h])
                    assert t <= p.big
                    y[r], y[r + h] = x[r] + t, x[r] + p.big
                    assert max(y[r], y[r + h]) <= LIMIT
            x = y
    return max(x)


def inverse(p, S, LE, bound, scaled):
    x = [bound] * (1 << LE)
    R = rounds(S, LE, True)
    for rho, A0 in enumerate(R):
        x = [max(x)] * len(x)
        for a in range(A0, LE):
            n, h = a - A0, 1 << a
            if n == 2 and p.heavy:
                x = [p.fold(b) if not r & (2 << A0) else b for r, b in enumerate(x)]
            if n == 3:
                x = [p.fold(b) if (p.heavy and r & 2 and not r & 4) or (not p.heavy and r & 1 and not r & 6) else b
                     for r, b in enumerate(x)]
            y = list(x)
            for r in range(len(x)):
                if not r & h:
                    assert x[r + h] <= p.K and x[r] + p.K <= LIMIT and x[r] + x[r + h] <= LIMIT
                    y[r], y[r + h] = x[r] + x[r + h], p.mul(x[r] + p.K)
            x = y
        if not (scaled and rho == len(R) - 1):
            x = [p.fold(b) for b in x]
    return max(x)


@pytest.mark.parametrize("k", range(50, 61))
@pytest.mark.parametrize("d", [1, (1 << 28) - 1])
@pytest.mark.parametrize("LE", [3, 4])
def test_ranges(k, d, LE):
    p = Prime(k, d)
    for cols, rows in ((7, 6), (7, 7), (8, 7), (8, 8), (9, 8)):
        b = forward(p, cols, LE, 4 * p.q, True)
        b = forward(p, rows, LE, b, False)
        assert p.fold_2q(b) <= 2 * p.q
        b = inverse(p, rows, LE, 2 * p.q, False)
        inverse(p, cols, LE, b, True)
    if LE == 3:                                                  # logN = 12: one pass
        assert p.fold_2q(forward(p, 12, LE, 4 * p.q, True)) <= 2 * p.q
        inverse(p, 12, LE, 2 * p.q, True)
