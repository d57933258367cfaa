"""The work that programs written on this framework give it, as cases to time.

A case is one call, or a short fixed sequence of calls, through the public
Python API of ``paper_2507_04775_gb300``.  Parameter sets are those of
``seeded_inputs.py``, the tests and ``bench.py``; ``draw`` varies ring degree,
level, digit count, prime sizes and rounding over the ranges that the API
takes.  Ciphertexts, plaintexts and keys are uniform residues: RLWE samples
look like that, and no kernel's work depends on the values.  Every output is
whole residues.
"""
from __future__ import annotations

import functools
from collections import OrderedDict

import numpy as np
import torch

import paper_2507_04775_gb300 as fides
from paper_2507_04775_gb300 import bootstrap


def _set(kind, logN, L, K, dnum, qb, pb, level, **more):
    return dict(kind=kind, logN=logN, L=L, K=K, dnum=dnum, qb=qb, pb=pb, level=level,
                nearest=more.pop("nearest", False), **more)


def listed():
    return [
        # one product at the smallest parameters (bounded-depth circuits, the
        # SMALL set): the call is nothing but latency
        dict(_set("hmult", 12, 3, 1, 3, 40, 50, 3), name="hmult_n12_l3"),
        # a rotation in a mid-size ring, a ragged last digit (7 limbs, digits of 3)
        dict(_set("rotate", 14, 7, 3, 3, 54, 60, 7, steps=5), name="rotate_n14_l7"),
        # encoding and decoding: transforms into and out of evaluation form,
        # three polynomials at a time
        dict(_set("ntt", 15, 14, 7, 2, 54, 60, 14, batch=3), name="ntt_n15_l14_b3"),
        # slot-wise arithmetic at the top level: plaintext product, sum,
        # constant product, difference
        dict(_set("elementwise", 16, 30, 10, 3, 54, 60, 30), name="elementwise_n16_l30"),
        # a weighted sum's step: plaintext product, then Rescale, mid chain
        dict(_set("ptmult_rescale", 16, 30, 10, 3, 54, 60, 21), name="ptmult_rescale_n16_l21"),
        # a rotation part-way down the chain (last digit of 7 limbs), rounding
        # to nearest as precise programs set it
        dict(_set("rotate", 16, 30, 10, 3, 54, 60, 17, steps=1024, nearest=True), name="rotate_n16_l17_nearest"),
        # the product that every circuit is made of, at the top level
        dict(_set("hmult", 16, 30, 10, 3, 54, 60, 30), name="hmult_n16_l30"),
        # product and Rescale in one call, the set of the paper's operation table
        dict(_set("hmult_rescale", 16, 30, 8, 4, 59, 60, 30), name="hmult_rescale_n16_l30_d4"),
        # the largest ring and key
        dict(_set("hmult", 17, 36, 9, 4, 54, 60, 36), name="hmult_n17_l36"),
        # a matrix-vector product: hoisted baby steps, plaintext sums, giant steps
        dict(_set("lintrans", 16, 30, 10, 3, 54, 60, 15, n_diag=32, n1=8), name="lintrans_n16_l15_d32"),
        # many users' products and rotations at uneven levels, planned once and
        # replayed as a graph
        dict(_set("batch", 16, 30, 10, 3, 54, 60, 30, n_ct=12), name="batch_n16_ct12"),
        # a whole bootstrap of a sparsely packed ciphertext (64 slots)
        dict(_set("bootstrap", 16, 30, 10, 3, 54, 60, 1, slots=64), name="bootstrap_n16_s64"),
    ]


_SINGLE = ("hmult", "hmult", "hmult_rescale", "rotate", "rotate", "keyswitch")


def draw(rng):
    kind = rng.choice(("single", "single", "single", "ntt", "elementwise", "ptmult_rescale", "lintrans", "batch",
                       "bootstrap"))
    logN = rng.choice((12, 13, 14, 15, 16, 16, 16, 17))
    L = rng.randint(2, 36) if logN > 12 else rng.randint(2, 14)
    dnum = rng.randint(1, min(6, L))
    alpha = -(-L // dnum)
    if alpha > 32 or (alpha > 16 and rng.random() < 0.7):   # mostly digits of up to 16 primes, as large sets have
        dnum, alpha = 3, -(-L // 3)
    K = min(alpha, 20)
    qb, pb = rng.choice(((40, 50), (50, 60), (54, 60), (54, 60), (59, 60), (60, 61)))
    level = rng.randint(2, L)
    nearest = rng.random() < 0.3
    if kind == "single":
        kind = rng.choice(_SINGLE)
        c = _set(kind, logN, L, K, dnum, qb, pb, level, nearest=nearest)
        if kind == "rotate":
            c["steps"] = rng.choice((1, -1)) * rng.randint(1, (1 << (logN - 1)) - 1)
        return c
    if kind == "ntt":
        return _set(kind, logN, L, K, dnum, qb, pb, level, batch=rng.randint(1, 6))
    if kind in ("elementwise", "ptmult_rescale"):
        return _set(kind, logN, L, K, dnum, qb, pb, level, nearest=nearest)
    if kind == "lintrans":
        return _set(kind, min(logN, 16), min(L, 20), min(K, 10), max(2, min(dnum, min(L, 20))), qb, pb,
                    min(level, min(L, 20)), nearest=nearest, n_diag=rng.randint(2, 40), n1=rng.choice((2, 4, 8)))
    if kind == "batch":
        return _set(kind, min(logN, 16), L, K, dnum, qb, pb, L, nearest=nearest, n_ct=rng.randint(2, 14))
    return _set("bootstrap", rng.choice((12, 13)), 30, 10, 3, 54, 60, 1, nearest=nearest,
                slots=rng.choice((32, 64, 128, 256, 512)))


# ---------------------------------------------------------------------------
# What a program keeps: contexts (one per parameter set) and bootstrapping
# plans, made once and used for every input.
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _primes(kind, logN, L, K, qb, pb):
    # a bootstrapping chain starts with a prime of the special primes' size
    head = fides.find_primes(logN, 60, 1) if kind == "bootstrap" else []
    q = head + fides.find_primes(logN, qb, L - len(head), exclude=head)
    p = fides.find_primes(logN, pb, K, exclude=q)
    return tuple(q), tuple(p)


def _case_primes(case):
    kind = "bootstrap" if case["kind"] == "bootstrap" else ""
    return _primes(kind, case["logN"], case["L"], case["K"], case["qb"], case["pb"])


_contexts = OrderedDict()


def _context(case):
    q, p = _case_primes(case)
    key = (case["logN"], q, p, case["dnum"], case["nearest"])
    if key not in _contexts:
        ctx = fides.Context(case["logN"], q, p, case["dnum"])
        ctx.set_rounding(case["nearest"])
        _contexts[key] = ctx
        while len(_contexts) > 4:
            _contexts.popitem(last=False)
    _contexts.move_to_end(key)
    return _contexts[key]


@functools.lru_cache(maxsize=4)
def _boot_plan(N, q, slots):
    return bootstrap.plan(N, q, 2.0 ** 50, slots=slots)


# ---------------------------------------------------------------------------
# Inputs: uniform residues from the seed, made on the GPU.
# ---------------------------------------------------------------------------
class _Draws:
    def __init__(self, seed, N, device="cuda"):
        self.N, self.device = N, device
        self.g = torch.Generator(device=device)
        self.g.manual_seed(seed)

    def residues(self, primes, *lead):
        """[*lead][len(primes)][N], limb i uniform modulo primes[i]."""
        x = torch.randint(0, 1 << 62, (*lead, len(primes), self.N), generator=self.g, device=self.device)
        return x.remainder_(torch.tensor(primes, dtype=torch.int64, device=self.device)[:, None])

    def key(self, case, q, p):
        return self.residues(q + p, case["dnum"], 2)


def _batch_plan(case):
    """Levels and rotation steps of the batch's ciphertexts: uneven, fixed by the sizes."""
    n, L = case["n_ct"], case["L"]
    low = max(2, L // 8)
    return [(low + (i * 7 + 3) % (L - low + 1), 1 << (i % 8)) for i in range(n)]


def _lt_steps(case):
    n1, d = case["n1"], case["n_diag"]
    return list(range(1, min(n1, d))) + [n1 * g for g in range(1, -(-d // n1))]


def _inputs(case, seed, device="cuda"):
    """The case's input tensors, by name."""
    q, p = _case_primes(case)
    q, p = list(q), list(p)
    kind, nl = case["kind"], case["level"]
    D = _Draws(seed, 1 << case["logN"], device)
    x = {}
    if kind == "ntt":
        x["a"] = D.residues(q[:nl], case["batch"])
        x["b"] = D.residues(q[:nl], case["batch"])
    elif kind == "keyswitch":
        x["a"] = D.residues(q[:nl])
        x["key"] = D.key(case, q, p)
    elif kind == "lintrans":
        x["a"] = D.residues(q[:nl], 2)
        x["pts"] = [D.residues(q[:nl]) for _ in range(case["n_diag"])]
        x["keys"] = [D.key(case, q, p) for _ in _lt_steps(case)]
    elif kind == "batch":
        plan = _batch_plan(case)
        x["a"] = [D.residues(q[:l], 2) for l, _ in plan]
        x["b"] = [D.residues(q[:l], 2) for l, _ in plan]
        x["key"] = D.key(case, q, p)
        x["rot"] = {s: D.key(case, q, p) for s in sorted({s for _, s in plan})}
    elif kind == "bootstrap":
        x["a"] = D.residues(q[:1], 2)
        prog = _boot_plan(1 << case["logN"], tuple(q), case["slots"])
        x["key"] = D.key(case, q, p)
        x["conj"] = D.key(case, q, p)
        x["rot"] = [D.key(case, q, p) for _ in prog.rot_steps]
    else:
        x["a"] = D.residues(q[:nl], 2)
        if kind in ("hmult", "hmult_rescale", "elementwise"):
            x["b"] = D.residues(q[:nl], 2)
        if kind in ("hmult", "hmult_rescale", "rotate"):
            x["key"] = D.key(case, q, p)
        if kind in ("elementwise", "ptmult_rescale"):
            x["pt"] = D.residues(q[:nl])
    return x


_K = 0x1234567890AB     # the scalar constant of the element-wise case


def prepare(case, seed):
    ctx = _context(case)
    x = _inputs(case, seed)
    kind, nl, N = case["kind"], case["level"], ctx.N

    def buf(*shape):
        return torch.empty(*shape, N, dtype=torch.int64, device="cuda")

    s = {"kind": kind, "ctx": ctx, "nl": nl, "x": x}
    if kind in ("hmult", "hmult_rescale"):
        s["rlk"] = ctx.relin_key(x["key"])
        s["out"] = buf(2, nl - (kind == "hmult_rescale"))
    elif kind == "rotate":
        s["steps"], s["rk"], s["out"] = case["steps"], ctx.rotation_key(x["key"], case["steps"]), buf(2, nl)
    elif kind == "keyswitch":
        s["evk"], s["out"] = ctx.relin_key(x["key"]), [buf(nl), buf(nl)]
    elif kind == "ntt":
        s["batch"] = case["batch"]
    elif kind == "elementwise":
        s["out"] = [buf(2, nl) for _ in range(4)]
    elif kind == "ptmult_rescale":
        s["prod"], s["out"] = buf(2, nl), buf(2, nl - 1)
    elif kind == "lintrans":
        s["diag"], s["n1"] = list(range(case["n_diag"])), case["n1"]
        s["keys"] = [ctx.rotation_key(t, k) for t, k in zip(x["keys"], _lt_steps(case))]
        # one work buffer kept for every transform of this size: at most
        # n1 - 1 rotations and two more ciphertexts
        s["work"], s["out"] = buf((case["n1"] + 1) * 2 * nl), buf(2, nl)
    elif kind == "batch":
        rlk = ctx.relin_key(x["key"])
        rot = {k: ctx.rotation_key(t, k) for k, t in x["rot"].items()}
        ops, s["out"] = [], []
        for (l, step), a, b in zip(_batch_plan(case), x["a"], x["b"]):
            m, r = buf(2, l), buf(2, l)
            ops.append(fides.Op(fides.OP_HMULT, a, l, m, b=b, key=rlk, stage=0))
            ops.append(fides.Op(fides.OP_ROTATE, m, l, r, key=rot[step], steps=step, stage=1))
            s["out"] += [m, r]
        s["batch"] = fides.Batch(ctx, ops)
        st = torch.cuda.Stream()
        st.wait_stream(torch.cuda.current_stream())
        s["batch"].capture(st)
        torch.cuda.current_stream().wait_stream(st)
    else:
        prog = _boot_plan(N, tuple(ctx.q), case["slots"])
        s["prog"] = bootstrap.DeviceProgram(ctx, prog, ctx.relin_key(x["key"]), ctx.conjugation_key(x["conj"]),
                                            [ctx.rotation_key(t, k) for t, k in zip(x["rot"], prog.rot_steps)])
        s["out"] = buf(2, s["prog"].out_limbs)
    return s


def run(s):
    kind, ctx, nl, x = s["kind"], s["ctx"], s["nl"], s["x"]
    if kind == "hmult":
        ctx.hmult(x["a"], x["b"], nl, s["rlk"], s["out"])
    elif kind == "hmult_rescale":
        ctx.hmult_rescale(x["a"], x["b"], nl, s["rlk"], s["out"])
    elif kind == "rotate":
        ctx.rotate(x["a"], nl, s["steps"], s["rk"], s["out"])
    elif kind == "keyswitch":
        ctx.keyswitch(x["a"], nl, s["evk"], s["out"][0], s["out"][1])
    elif kind == "ntt":
        # in place, as the API has it: a goes into evaluation form, b out of it
        ctx.ntt(x["a"], 0, nl, s["batch"])
        ctx.intt(x["b"], 0, nl, s["batch"])
        return [x["a"], x["b"]]
    elif kind == "elementwise":
        o = s["out"]
        ctx.ptmult(x["a"], x["pt"], nl, o[0])
        ctx.hadd(o[0], x["b"], nl, o[1])
        ctx.scalar_mult(x["b"], _K, nl, o[2])
        ctx.hsub(x["a"], o[2], nl, o[3])
    elif kind == "ptmult_rescale":
        ctx.ptmult(x["a"], x["pt"], nl, s["prod"])
        ctx.rescale(s["prod"], nl, s["out"])
    elif kind == "lintrans":
        ctx.linear_transform(x["a"], nl, s["diag"], x["pts"], s["n1"], s["keys"], s["out"], work=s["work"])
    elif kind == "batch":
        s["batch"].run()
    else:
        s["prog"].run(x["a"], s["out"], 2.0 ** 50)
    return s["out"]


# ---------------------------------------------------------------------------
# Work that one pass cannot do without: each input and key limb in use read
# once, each output written once; two operations for every 64-bit modular
# product of the transforms, conversions and products.
# ---------------------------------------------------------------------------
class _Work:
    def __init__(self, case):
        self.N, self.logN = 1 << case["logN"], case["logN"]
        self.K, self.alpha = case["K"], -(-case["L"] // case["dnum"])
        self.words = self.products = 0

    def limbs(self, n):
        self.words += n * self.N

    def ntt(self, n):
        self.products += n * (self.N // 2) * self.logN

    def slot(self, n):
        self.products += n * self.N

    def modup(self, nl):
        ne, beta = nl + self.K, -(-nl // self.alpha)
        self.ntt(nl + beta * ne - nl)
        self.slot(nl * (ne - min(self.alpha, nl)))

    def tail(self, nl, key=True):
        """Inner product with one key and both ModDowns."""
        ne, beta = nl + self.K, -(-nl // self.alpha)
        if key:
            self.limbs(beta * 2 * ne)
        self.slot(2 * beta * ne + 2 * self.K * nl + 2 * nl)
        self.ntt(2 * (self.K + nl))

    def rescale(self, nl):
        self.ntt(2 + 2 * (nl - 1))
        self.slot(2 * (nl - 1))

    def lintrans(self, nl, n_diag, baby, giant, key=True):
        if baby:
            self.modup(nl)
        for _ in range(baby):
            self.tail(nl, key)
        for _ in range(giant):
            self.modup(nl)
            self.tail(nl, key)
        self.limbs(n_diag * nl)
        self.slot(2 * n_diag * nl)

    def total(self):
        return {"bytes": 8.0 * self.words, "flops": 2.0 * self.products}


def work(case):
    w, kind, nl = _Work(case), case["kind"], case["level"]
    if kind in ("hmult", "hmult_rescale"):
        out = nl - (kind == "hmult_rescale")
        w.limbs(4 * nl + 2 * out)
        w.slot(4 * nl)
        w.modup(nl)
        w.tail(nl)
    elif kind == "rotate":
        w.limbs(4 * nl)
        w.modup(nl)
        w.tail(nl)
    elif kind == "keyswitch":
        w.limbs(3 * nl)
        w.modup(nl)
        w.tail(nl)
    elif kind == "ntt":
        w.limbs(4 * nl * case["batch"])
        w.ntt(2 * nl * case["batch"])
    elif kind == "elementwise":
        w.limbs(5 * nl + 4 * 2 * nl)
        w.slot(4 * nl)
    elif kind == "ptmult_rescale":
        w.limbs(3 * nl + 2 * (nl - 1))
        w.slot(2 * nl)
        w.rescale(nl)
    elif kind == "lintrans":
        w.limbs(4 * nl)
        n1, d = case["n1"], case["n_diag"]
        w.lintrans(nl, d, min(n1, d) - 1, -(-d // n1) - 1)
    elif kind == "batch":
        steps = set()
        for l, step in _batch_plan(case):
            w.limbs(4 * l + 2 * l + 2 * l)
            w.slot(4 * l)
            for _ in range(2):
                w.modup(l)
                w.tail(l, key=False)
            steps.add(step)
        w.limbs((1 + len(steps)) * case["dnum"] * 2 * (case["L"] + case["K"]))
    else:
        q, _ = _case_primes(case)
        prog = _boot_plan(w.N, q, case["slots"])
        level, seen = {prog.in_reg: 1}, []
        for op, dst, a, b, arg in prog.instr:
            name = _INSTRUCTIONS[op]
            la = level.get(a, 0)
            out = {"MODRAISE": arg, "DROP": arg, "RESCALE": la - 1, "CMAC": b}.get(name, la)
            level[dst] = out
            if name == "MODRAISE":
                w.ntt(2 + 2 * out)
            elif name == "RESCALE":
                w.rescale(la)
            elif name in ("HMULT", "CONJ", "ROT"):
                w.slot(4 * la if name == "HMULT" else 0)
                w.modup(la)
                w.tail(la, key=False)
            elif name == "LT":
                t = prog.lts[arg]
                idx, n1 = t["diag_idx"], t["n1"]
                w.lintrans(la, len(idx), len({i % n1 for i in idx} - {0}), len({i // n1 for i in idx} - {0}), key=False)
        w.limbs((2 + len(prog.rot_steps)) * case["dnum"] * 2 * (case["L"] + case["K"]))
        w.limbs(2 + 2 * level[prog.out_reg])
    return w.total()


_INSTRUCTIONS = dict(enumerate(("", "MODRAISE", "LT", "RESCALE", "DROP", "HADD", "HSUB", "HMULT", "CONJ", "MULI",
                                  "CMULT", "CADD", "COPY", "CMAC", "ROT")))


# ---------------------------------------------------------------------------
# The same results from plain 64-bit torch arithmetic: textbook transforms and
# the definitions of the operations.
# ---------------------------------------------------------------------------
def _mul_small(a, b, q):
    """a b mod q for a < q < 2^62 and b < 2^31: the FP64 quotient is within one."""
    r = a * b - (a.double() * b.double() / q.double()).to(torch.int64) * q
    r = torch.where(r < 0, r + q, r)
    r = torch.where(r < 0, r + q, r)
    return torch.where(r >= q, r - q, r)


def _mul(a, b, q):
    a, b = torch.broadcast_tensors(a, b)
    hi = _mul_small(_mul_small(a, b >> 30, q), torch.full_like(a, 1 << 30), q)
    r = hi + _mul_small(a, b & ((1 << 30) - 1), q)
    return torch.where(r >= q, r - q, r)


@functools.lru_cache(maxsize=None)
def _psi(logN, q):
    """A primitive 2N-th root of unity: from the smallest generator modulo q."""
    rest, factors = q - 1, {2}
    while rest % 2 == 0:
        rest //= 2
    d = np.arange(3, 1 << 24, 2, dtype=np.int64)
    for f in d[rest % d == 0].tolist():
        while rest % f == 0:
            factors.add(f)
            rest //= f
    if rest > 1:
        factors.add(rest)
    g = next(g for g in range(2, q) if all(pow(g, (q - 1) // f, q) != 1 for f in factors))
    return pow(g, (q - 1) >> (logN + 1), q)


class _Plain:
    def __init__(self, case, device):
        q, p = _case_primes(case)
        self.q, self.p, self.logN, self.N = list(q), list(p), case["logN"], 1 << case["logN"]
        self.alpha, self.nearest, self.dev = -(-case["L"] // case["dnum"]), case["nearest"], device
        r = np.arange(self.N)
        rev = np.zeros(self.N, dtype=np.int64)
        for i in range(self.logN):
            rev |= ((r >> i) & 1) << (self.logN - 1 - i)
        self.rev, self.tw = torch.from_numpy(rev).to(device), {}

    def col(self, values):
        return torch.tensor([int(v) for v in values], dtype=torch.int64, device=self.dev)[:, None]

    def powers(self, q, inverse):
        key = (q, inverse)
        if key not in self.tw:
            w = _psi(self.logN, q)
            w = pow(w, -1, q) if inverse else w
            t, qq = torch.ones(1, dtype=torch.int64, device=self.dev), torch.tensor(q, device=self.dev)
            for i in range(self.logN):
                t = torch.cat([t, _mul(t, torch.full_like(t, pow(w, 1 << i, q)), qq)])
            self.tw[key] = t[self.rev]
        return self.tw[key]

    def ntt(self, x, primes):
        w = torch.stack([self.powers(q, False) for q in primes])
        q, m, x = self.col(primes)[:, None], 1, x.clone()
        while m < self.N:
            v = x.view(len(primes), m, 2, -1)
            t = _mul(v[:, :, 1], w[:, m:2 * m, None], q)
            a = v[:, :, 0]
            x = torch.stack([(a + t) % q, (a - t) % q], 2).reshape(len(primes), -1)
            m *= 2
        return x

    def intt(self, x, primes):
        w = torch.stack([self.powers(q, True) for q in primes])
        q, m, x = self.col(primes)[:, None], self.N // 2, x.clone()
        while m >= 1:
            v = x.view(len(primes), m, 2, -1)
            a, b = v[:, :, 0], v[:, :, 1]
            x = torch.stack([(a + b) % q, _mul((a - b) % q, w[:, m:2 * m, None], q)], 2).reshape(len(primes), -1)
            m //= 2
        return _mul(x, self.col([pow(self.N, -1, q) for q in primes]), self.col(primes))

    def convert(self, x, src, dst, centred=False):
        """Fast base conversion of coefficient-form limbs modulo src to dst."""
        v, P = [], 1
        for s in src:
            P *= s
        for i, s in enumerate(src):
            v.append(_mul(x[i], torch.tensor(pow(P // s, -1, s), device=self.dev), torch.tensor(s, device=self.dev)))
        y = []
        for d in dst:
            dq, acc = torch.tensor(d, device=self.dev), torch.zeros_like(x[0])
            for i, s in enumerate(src):
                acc = (acc + _mul(v[i] % dq, torch.tensor(P // s % d, device=self.dev), dq)) % dq
                if centred:
                    acc = torch.where(v[i] > (s - 1) // 2, (acc - P % d) % dq, acc)
            y.append(acc)
        return torch.stack(y)

    def modup(self, d):
        nl = len(d)
        q = self.q[:nl]
        c, ext = self.intt(d, q), []
        for lo in range(0, nl, self.alpha):
            hi = min(lo + self.alpha, nl)
            to = q[:lo] + q[hi:] + self.p
            e = self.ntt(self.convert(c[lo:hi], q[lo:hi], to), to)
            ext.append(torch.cat([e[:lo], d[lo:hi], e[lo:]]))
        return ext

    def moddown(self, x):
        nl = len(x) - len(self.p)
        q, P = self.q[:nl], 1
        for s in self.p:
            P *= s
        t = self.ntt(self.convert(self.intt(x[nl:], self.p), self.p, q, self.nearest), q)
        qq = self.col(q)
        return _mul((x[:nl] - t) % qq, self.col([pow(P, -1, s) for s in q]), qq)

    def inner(self, ext, key, nl):
        primes = self.q[:nl] + self.p
        qq, L = self.col(primes), len(self.q)
        acc = []
        for t in range(2):
            a = 0
            for e, k in zip(ext, key):
                a = (a + _mul(e, torch.cat([k[t, :nl], k[t, L:]]), qq)) % qq
            acc.append(a)
        return acc

    def keyswitch(self, d, key):
        return [self.moddown(a) for a in self.inner(self.modup(d), key, len(d))]

    def hmult(self, a, b, key):
        nl = a.shape[1]
        qq = self.col(self.q[:nl])
        k0, k1 = self.keyswitch(_mul(a[1], b[1], qq), key)
        d1 = (_mul(a[0], b[1], qq) + _mul(a[1], b[0], qq)) % qq
        return torch.stack([(_mul(a[0], b[0], qq) + k0) % qq, (d1 + k1) % qq])

    def sigma(self, x, steps):
        g = pow(5, steps % (self.N // 2), 2 * self.N)
        return x[..., self.rev[(((2 * self.rev + 1) * g) % (2 * self.N) - 1) // 2]]

    def rotate(self, a, steps, key):
        k0, k1 = self.keyswitch(self.sigma(a[1], steps), key)
        qq = self.col(self.q[:a.shape[1]])
        return torch.stack([(self.sigma(a[0], steps) + k0) % qq, k1])

    def hoisted(self, a, steps, keys):
        nl = a.shape[1]
        qq, ext, out = self.col(self.q[:nl]), self.modup(a[1]), []
        for s, k in zip(steps, keys):
            k0, k1 = [self.moddown(t) for t in self.inner([self.sigma(e, s) for e in ext], k, nl)]
            out.append(torch.stack([(self.sigma(a[0], s) + k0) % qq, k1]))
        return out

    def rescale(self, x):
        l = x.shape[1] - 1
        q, ql, out = self.q[:l], self.q[l], []
        qq = self.col(q)
        for c in x:
            r = self.intt(c[l:], [ql])
            r = torch.where(r > (ql - 1) // 2, r - ql, r) if self.nearest else r
            t = self.ntt((r % qq).contiguous(), q)
            out.append(_mul((c[:l] - t) % qq, self.col([pow(ql, -1, s) for s in q]), qq))
        return torch.stack(out)


def exact(case, seed):
    kind, nl = case["kind"], case["level"]
    if kind == "bootstrap":
        return None         # some 200 key switches: minutes
    device = "cuda" if torch.cuda.is_available() else "cpu"
    x, P = _inputs(case, seed, device), _Plain(case, device)
    q = P.q[:nl]
    qq = P.col(q)
    if kind == "hmult":
        return P.hmult(x["a"], x["b"], x["key"])
    if kind == "hmult_rescale":
        return P.rescale(P.hmult(x["a"], x["b"], x["key"]))
    if kind == "rotate":
        return P.rotate(x["a"], case["steps"], x["key"])
    if kind == "keyswitch":
        return P.keyswitch(x["a"], x["key"])
    if kind == "ntt":
        return [torch.stack([P.ntt(t, q) for t in x["a"]]), torch.stack([P.intt(t, q) for t in x["b"]])]
    if kind == "elementwise":
        o0 = _mul(x["a"], x["pt"], qq)
        o2 = _mul(x["b"], P.col([_K % s for s in q]), qq)
        return [o0, (o0 + x["b"]) % qq, o2, (x["a"] - o2) % qq]
    if kind == "ptmult_rescale":
        return P.rescale(_mul(x["a"], x["pt"], qq))
    if kind == "batch":
        out = []
        for (l, step), a, b in zip(_batch_plan(case), x["a"], x["b"]):
            m = P.hmult(a, b, x["key"])
            out += [m, P.rotate(m, step, x["rot"][step])]
        return out
    n1, d = case["n1"], case["n_diag"]
    steps = _lt_steps(case)
    keys = dict(zip(steps, x["keys"]))
    baby = list(range(1, min(n1, d)))
    rot = [x["a"]] + P.hoisted(x["a"], baby, [keys[b] for b in baby])
    y = 0
    for g in range(-(-d // n1)):
        inner = 0
        for i in range(g * n1, min(d, (g + 1) * n1)):
            inner = (inner + _mul(rot[i % n1], x["pts"][i], qq)) % qq
        y = (y + (P.rotate(inner, n1 * g, keys[n1 * g]) if g else inner)) % qq
    return y
