"""w = A z + B^T p of the FP32-cycle FGMRES step, restated on the host in numpy float32: A z
is a pair of floats, B^T p an FP64 sum left as three floats that add up to it (24 + 24 + 5
bits), and their sum, kept as a pair, lies within 2^-47 of the exact sum of the two also
where they cancel -- which a B^T p rounded to a pair first does not reach."""
from fractions import Fraction

import numpy as np

F = np.float32


def two_sum(a, b):
    t = F(a + b)
    q = F(t - a)
    return t, F(F(a - F(t - q)) + F(b - q))


def norm_pair(S, s):
    hi = F(S + s)
    return hi, F(s - F(hi - S))


def split(v, parts):
    out = []
    for _ in range(parts):
        out.append(F(v))
        v = v - float(out[-1])
    return out, v


def join(a, t):
    (b0, b1, b2), rest = split(t, 3)
    assert rest == 0.0
    s, e1 = two_sum(a[0], b0)
    l, e2 = two_sum(a[1], b1)
    m, e3 = two_sum(e1, l)
    hi, e4 = two_sum(s, m)
    return norm_pair(hi, F(e4 + F(F(e2 + e3) + b2)))


def join_pairs(a, t):
    (b0, b1), _ = split(t, 2)
    s, e = two_sum(a[0], b0)
    return norm_pair(s, F(a[1] + F(e + b1)))


def error(w, a, t):
    want = Fraction(float(a[0])) + Fraction(float(a[1])) + Fraction(t)
    got = Fraction(float(w[0])) + Fraction(float(w[1]))
    return float(abs(got - want) / abs(want)) if want else float(abs(got))


def draws(cancel):
    rng = np.random.default_rng(4)
    for _ in range(4000):
        t = float(rng.standard_normal() * 10.0 ** rng.uniform(-12, 12))
        v = -t * (1.0 + float(rng.standard_normal()) * 2.0 ** -cancel) if cancel else \
            float(rng.standard_normal() * 10.0 ** rng.uniform(-12, 12))
        yield tuple(split(v, 2)[0]), t


def test_join_keeps_fp64_sums():
    for cancel in (0, 1, 10, 23, 30, 40):
        assert max(error(join(a, t), a, t) for a, t in draws(cancel)) <= 2.0 ** -47


def test_pairs_alone_would_not():
    assert max(error(join_pairs(a, t), a, t) for a, t in draws(30)) > 2.0 ** -30
