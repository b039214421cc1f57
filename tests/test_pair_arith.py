"""Host emulation of the float-pair arithmetic of large FP64 Phi launches
(df_pair.cuh: pair_factor, pair_mul, PairProduct; df_walk.cuh: df_cut, df_dot,
df_divide, df_fma2, the escapes' bound; phi_kernels.cuh: df_add), operation for
operation in numpy float32, against exact rationals.

u = 2^-24.  A factor's pair is within 2^-49 and each product adds at most 2^-47.  The
quotient is within 3e-13 (40 u^2 for four ranks per lane, 5 u^2 for each of five
exchanges, 10 u^2 for cuts and division).  A sum of n terms v pi rounds its
remainders' sum C, at most (2 + n) u of the sum itself, three times per term and
one FMA more: (3 n (2 + n) + n) u^2, 3.1e-12 for the 16 terms between two moves to
FP64 if all roundings had one sign; they do not, and the entries are asked to be
within the 1e-12 that the library's parity tests ask of Phi."""
import struct
from fractions import Fraction

import numpy as np

f32 = np.float32
TOP, LOW, FACTOR_LOW = 60, -80, -100
DF_S, DF_V = 60, 10
DOWN = f32(2.0 ** -60)


def _u2f(u):
    return f32(struct.unpack("<f", struct.pack("<I", u & 0xFFFFFFFF))[0])


def _f2u(f):
    return struct.unpack("<I", struct.pack("<f", f))[0]


def fma(a, b, c):  # the product of two floats is exact in double
    return f32(float(a) * float(b) + float(c))


def exact(p):
    return Fraction(float(p[0])) + Fraction(float(p[1]))


def pair_factor(v, s):
    """(hi, lo) of v 2^s, or "low" / "high"."""
    if v == 0.0:
        return f32(0), f32(0)
    m, e = np.frexp(v)
    es = int(e) - 1 + s
    if v < 2.0 ** -1022 or es < FACTOR_LOW:
        return "low"
    w = float(np.ldexp(v, s))
    if es > TOP or w > 2.0 ** TOP:
        return "high"
    h = f32(w)
    return h, f32(w - float(h))


def pair_mul(a, b):
    p = f32(a[0] * b[0])
    e = fma(a[0], b[0], -p)
    e = fma(a[0], b[1], e)
    e = f32(fma(a[1], b[0], e) * DOWN)
    h = fma(p, DOWN, e)
    return h, f32(e - fma(-DOWN, p, h))


def product(ops):
    """PairProduct::value over factor entries as pair_factor gives them."""
    raw = [{"low": (f32(-2.0 ** -126), f32(0)), "high": (f32(-np.inf), f32(0))}.get(o, o) if isinstance(o, str) else o
           for o in ops]
    with np.errstate(all="ignore"):
        p = raw[0]
        for b in raw[1:]:
            p = pair_mul(p, b)
    esc = any(isinstance(o, str) for o in ops)
    if not esc and p[0] >= f32(2.0 ** LOW):
        return p
    if any(not isinstance(o, str) and o[0] == 0 for o in ops):
        return f32(0), f32(0)
    return "high" if esc and not abs(float(p[0])) < np.inf else "low"


def cut(x, s):
    """df_cut: the leading 48 bits of x 2^s."""
    w = Fraction(x) * Fraction(2) ** s
    if w < Fraction(2) ** -126:
        return f32(0), f32(0)
    bits = struct.unpack("<Q", struct.pack("<d", float(w)))[0]
    H, L = bits >> 32, bits & 0xFFFFFFFF
    e = H >> 20
    if e >= 1023 + 100:
        return f32(np.inf), f32(0)
    h = _u2f((((H << 3) | (L >> 29)) & 0xFFFFFFFF) - (896 << 23))
    v = L & 0x1FFFFFFF
    nb = v.bit_length()
    if nb > 24:
        v = (v >> (nb - 24)) << (nb - 24)
    low = f32(f32(f32(v) * _u2f((e - 1023 + 127) << 23)) * f32(2.0 ** -52))
    t = f32(h + low)
    return t, f32(low - f32(t - h))


def fma2(a, b, S, C):
    t = fma(a[0], b[0], S)
    nz = f32(S - t)
    e = f32(S - f32(t + nz))
    r = fma(a[0], b[0], nz)
    C = fma(a[0], b[1], C)
    C = fma(a[1], b[0], C)
    return t, f32(C + f32(e + r))


def dot(a, b):
    """df_dot: even and odd columns, then their sums."""
    S, C = [], []
    for o in (0, 1):
        x, y = a[o], b[o]
        s = f32(x[0] * y[0])
        c = fma(x[0], y[0], -s)
        c = fma(x[0], y[1], c)
        c = fma(x[1], y[0], c)
        for v in range(2 + o, len(a), 2):
            s, c = fma2(a[v], b[v], s, c)
        S.append(s)
        C.append(c)
    t = f32(S[0] + S[1])
    z = f32(t - S[0])
    c = f32(f32(f32(S[0] - f32(t - z)) + f32(S[1] - z)) + f32(C[0] + C[1]))
    h = f32(t + c)
    return h, f32(c - f32(h - t))


def add_pair(a, b):
    s = f32(a[0] + b[0])
    z = f32(s - a[0])
    e = f32(f32(f32(a[0] - f32(s - z)) + f32(b[0] - z)) + f32(a[1] + b[1]))
    h = f32(s + e)
    return h, f32(e - f32(h - s))


def divide(x, s, eps, rng):
    use = f32(f32(s[0] - eps[0]) + f32(s[1] - eps[1])) >= 0
    m = s if use else eps
    r = f32(1.0 / float(m[0]))
    k = rng.integers(-1, 2)  # the hardware estimate's stated error of one ulp
    r = np.nextafter(r, f32(np.inf)) if k > 0 else np.nextafter(r, f32(0)) if k < 0 else r
    r = fma(r, fma(-m[0], r, f32(1)), r)
    q0 = f32(x[0] * r)
    p = f32(q0 * m[0])
    pe = fma(q0, m[0], -p)
    q1 = f32(f32(f32(f32(x[0] - p) - pe) + fma(-q0, m[1], x[1])) * r)
    h = f32(q0 + q1)
    return h, f32(q1 - f32(h - q0))


def test_products_and_their_window():
    rng = np.random.default_rng(3)
    edge = [0.0, 1.0, np.nextafter(1.0, 0), np.nextafter(1.0, 2), 1.5, 2.0 ** -160, np.nextafter(2.0 ** -160, 0),
            2.0 ** -140, 2.0 ** -139.5, 2.0 ** -70, 1e-310, 1e-200]
    seen = set()
    for _ in range(6000):
        nm1 = int(rng.integers(1, 8))
        vs = [float(rng.choice(edge)) if rng.random() < 0.3 else float(2.0 ** -rng.uniform(0, 170 / nm1)) for _ in range(nm1)]
        got = product([pair_factor(v, TOP) for v in vs])
        want = Fraction(2) ** TOP
        for v in vs:
            want *= Fraction(v)
        if isinstance(got, str):
            seen.add(got)
            if got == "low":    # no product is called low that is not: to a rounding
                assert want < Fraction(2) ** LOW * (1 + Fraction(1, 2 ** 20))
            else:               # only where an entry is above its exponent
                assert max(vs) > 1.0
        elif want == 0:
            seen.add("zero")
            assert got == (0, 0)
        else:
            seen.add("pair")
            bound = nm1 * Fraction(1, 2 ** 49) + (nm1 - 1) * Fraction(1, 2 ** 47)
            assert abs(exact(got) - want) <= bound * want, (vs, nm1)
    assert seen == {"low", "high", "zero", "pair"}


def test_cuts_over_their_whole_range():
    """48 bits from 2^-78 on (below, what a float holds), up to 2^100; counts up to 2^30 whose
    low bits are all in use among them."""
    rng = np.random.default_rng(6)
    for x in [float(2 ** 30 - 2 ** -22), 2.0 ** 17 + 2.0 ** -35, 2.0 ** 29 / 3] + list(2.0 ** rng.uniform(-20, 30, 2000)):
        h, low = cut(float(x), DF_S + DF_V)
        w = Fraction(float(x)) * Fraction(2) ** (DF_S + DF_V)
        assert abs(exact((h, low)) - w) <= w * Fraction(1, 2 ** 47) and abs(float(low)) <= float(np.spacing(h)) / 2
    for x in 2.0 ** rng.uniform(-78, 100, 2000):
        h, low = cut(float(x), 0)
        assert abs(exact((h, low)) - Fraction(float(x))) <= Fraction(float(x)) * Fraction(1, 2 ** 47)
    assert cut(2.0 ** 100, 0)[0] == np.inf and cut(2.0 ** -127, 0) == (0, 0)


def test_quotients_and_sums():
    """One row: 16 nonzeros (the terms between two moves to FP64), ranks over G lanes of
    four; quotients within 3e-13, the row's entries within 1e-12 and 1e-14 in the mean."""
    rng = np.random.default_rng(4)
    eps = 1e-10
    errs = []
    for trial in range(60):
        G = int(rng.choice([1, 2, 4, 8, 32]))
        R = 4 * G
        spread = rng.choice([1.0, 20.0, 60.0])
        b = [float(2.0 ** rng.uniform(-spread / 2, 10)) for _ in range(R)]
        nm1 = int(rng.integers(1, 4))
        bp = [cut(v, DF_S - TOP) for v in b]
        ep = cut(eps, DF_S)
        use = list(range(4)) if R > 8 else list(range(R))  # columns whose sums are followed
        S = {c: (f32(0), f32(0)) for c in use}
        want = {c: Fraction(0) for c in use}
        for _ in range(16):
            fs = [[float(2.0 ** -rng.uniform(0, spread / nm1)) for _ in range(nm1)] for _ in range(R)]
            row = [product([pair_factor(v, TOP) for v in f]) for f in fs]
            assert not any(isinstance(p, str) for p in row)
            x = float(rng.integers(1, 2 ** int(rng.integers(1, 30))))
            lanes = [dot(bp[4 * g:4 * g + 4], row[4 * g:4 * g + 4]) for g in range(G)]
            while len(lanes) > 1:
                lanes = [add_pair(lanes[i], lanes[i + len(lanes) // 2]) for i in range(len(lanes) // 2)]
            v = divide(cut(x, DF_S + DF_V), lanes[0], ep, rng)
            el = [Fraction(1)] * R
            for c in range(R):
                for f in fs[c]:
                    el[c] *= Fraction(f)
            d = max(sum(Fraction(b[c]) * el[c] for c in range(R)), Fraction(eps))
            q = Fraction(x) / d
            assert abs(exact(v) / Fraction(2) ** DF_V - q) <= Fraction(3, 10 ** 13) * q
            for c in use:
                S[c] = fma2(v, row[c], *S[c])
                want[c] += q * el[c]
        for c in use:
            got = (Fraction(float(S[c][0])) + Fraction(float(S[c][1]))) / Fraction(2) ** (TOP + DF_V)
            errs.append(float(abs(got - want[c]) / want[c]))
    assert max(errs) <= 1e-12 and np.mean(errs) <= 1e-14, (max(errs), np.mean(errs))


def test_escapes_bound_is_not_below_what_is_left_out():
    """The float kept with a row's escapes (its low 8 bits hold columns) is not below the
    sum of their quotients, so a column with 2^-25 of it or more lacks at most 2^-55."""
    rng = np.random.default_rng(5)
    for _ in range(300):
        esc, total = 0, Fraction(0)
        for _ in range(int(rng.integers(1, 200))):
            vh = f32(2.0 ** rng.uniform(-20, 50))
            total += Fraction(float(vh)) * (1 + Fraction(1, 2 ** 23))  # its lo part
            s = f32(_u2f(esc & ~0xFF) + f32(vh * f32(1.01)))
            esc = ((_f2u(s) & ~0xFF) + 0x100) | (esc & 0xFF) | int(rng.integers(1, 16))
        assert Fraction(float(_u2f(esc & ~0xFF))) >= total
