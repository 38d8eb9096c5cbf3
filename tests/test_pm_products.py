"""Host check of the products modulo q = 2^b - d and of the transforms' storage order.

pm_mul(a, w) = P + 2^k ql + 4d qh with k = b - 30, v = 2^32 w mod q, w and v cut at bit k, P = a0 wl + a1 vl,
Q = a0 wh + a1 vh = qh 2^32 + ql: replayed with the kernels' 32-bit operand ranges at the extremes and at random for
the moduli of the parameter rule; congruence, the bound that a context checks its transforms against, and the folds.
eval_pos (the evaluation domain's storage order) and the exchanges that the transforms keep inside a warp are walked
for every shape.
"""

import random

import pytest

from oracle.params import Params


def s32(x):
    assert -(1 << 31) <= x < (1 << 31), x
    return x


def u32(x):
    assert 0 <= x < (1 << 32), x
    return x


def entry(w, q, b):
    k = b - 30
    v = (w << 32) % q
    return w & ((1 << k) - 1), w >> k, v & ((1 << k) - 1), v >> k


def pm_mul(a, w, q, b):
    wl, wh, vl, vh = (u32(x) for x in entry(w, q, b))
    s32(wh), s32(vh), s32(vl)
    a0, a1 = u32(a & 0xFFFFFFFF), s32(a >> 32)
    Q = a0 * wh + a1 * vh
    assert abs(Q) < 1 << 63
    ql, qh = u32(Q & 0xFFFFFFFF), s32(Q >> 32)
    d4 = s32(4 * ((1 << b) - q))
    T = a0 * wl + a1 * vl + (ql << (b - 30)) + qh * d4
    assert abs(T) < 1 << 63
    return T


def stage_bound(b, d):
    return 3 * 2 ** 29 * 4 * d + 5 * 2 ** (b + 1)


def fold(x, b, d):
    h = x >> b
    return s32(h) * d + (x & ((1 << b) - 1))


@pytest.mark.parametrize("bits", [45, 50, 55])
@pytest.mark.parametrize("N,L", [(1024, 1), (16384, 8), (32768, 16)])
def test_products_are_congruent_and_bounded(bits, N, L):
    prm = Params(N=N, L=L, alpha=2, prime_bits=bits)
    rng = random.Random(bits * N + L)
    big = (1 << 63) - 1
    for q in prm.q + prm.p + prm.b:
        d = (1 << bits) - q
        assert 0 < d < 1 << 27
        words = [0, 1, q - 1, big, -big - 1, (1 << 32) - 1, 1 << 32, -1] + [rng.randrange(-big, big) for _ in range(40)]
        ws = [0, 1, q - 1, (1 << 32) - 1, q >> 1] + [rng.randrange(q) for _ in range(10)]
        for a in words:
            y = fold(a, bits, d)
            assert (y - a) % q == 0 and -(d << (63 - bits)) <= y < (1 << bits) + (d << (63 - bits))
            y += q if y < 0 else 0
            assert 0 <= y < 2 * q
            for w in ws:
                T = pm_mul(a, w, q, bits)
                assert (T - a * w) % q == 0 and abs(T) <= stage_bound(bits, d)


class Sum:
    """One extension sum as ext_pm.cu computes it: digits y cut at bit hs, constants at bit k, wide sums P and Q."""

    def __init__(self, b):
        self.b, self.k, self.hs = b, b - 28, (b + 2) // 2

    def digits(self, ys):
        out = []
        for y in ys:
            y0, y1 = u32(y & ((1 << self.hs) - 1)), s32(y >> self.hs)
            out.append((y0, y1))
        return out

    def fold(self, ys, v, consts, cv, T, extra=None):
        """sum y c + v cv (+ a 64-bit word times a twist constant): congruent, every partial sum below 2^63."""
        m, P, Q = (1 << self.k) - 1, 0, 0

        def acc(a, c):
            nonlocal P, Q
            P += a * s32(c & m)
            Q += a * s32(c >> self.k)
            assert abs(P) < 1 << 63 and abs(Q) < 1 << 63
        if extra:
            a, w = extra
            acc(u32(a & 0xFFFFFFFF), w)
            acc(s32(a >> 32), (w << 32) % T)
        acc(v, cv)
        for (y0, y1), c in zip(self.digits(ys), consts):
            acc(y0, c)
            acc(y1, (c << self.hs) % T)
        d16 = s32(16 * ((1 << self.b) - T))
        r = P + ((Q & 0xFFFFFFFF) << self.k) + s32(Q >> 32) * d16
        assert abs(r) < 1 << 62
        return r

    def round(self, ys, guard):
        z = sum(ys) + (1 << (self.b - 1))
        frac = z & ((1 << self.b) - 1)
        return z >> self.b, guard <= frac < (1 << self.b) - guard


@pytest.mark.parametrize("bits", [45, 50, 55])
@pytest.mark.parametrize("N,L", [(1024, 1), (16384, 8), (32768, 16)])
def test_extension_sums_are_exact(bits, N, L):
    """The lift's digits, overflow count and sums, and scale-and-round's with its twist word, at the extremes of their
    operands and near the centring boundary: the guarded count is the true one and the result congruent."""
    from fractions import Fraction
    prm = Params(N=N, L=L, alpha=2, prime_bits=bits)
    S, rng = Sum(bits), random.Random(bits + N)
    src, dst = prm.q, prm.b
    Q = 1
    for q in src:
        Q *= q
    dmax = max((1 << bits) - q for q in prm.q + prm.p + prm.b)
    hat = [pow(Q // q, -1, q) for q in src]
    y_up = (1 << bits) + (dmax << (S.hs + 1)) + (1 << (S.hs + bits - 27))
    y_sc = (1 << bits) + (dmax << (63 - bits))

    def guard(y):
        ds = max((1 << bits) - q for q in src)
        return len(src) * y * ds // ((1 << bits) - ds) + len(src) + 2
    xs = [0, 1, Q - 1, Q // 2, Q // 2 + 1, Q // 2 + Q // (1 << 40)] + [rng.randrange(Q) for _ in range(6)]
    hit = 0
    for x in xs:
        ys = []
        for q, h in zip(src, hat):
            r, d = x % q, (1 << bits) - q
            x0, x1 = u32(r & ((1 << S.hs) - 1)), u32(r >> S.hs)
            hv = (h << S.hs) % q
            q2 = x0 * (h >> S.k) + x1 * (hv >> S.k)
            m = (1 << S.k) - 1
            y = ((q2 & ((1 << 28) - 1)) << S.k) + x0 * (h & m) + x1 * (hv & m) + u32(q2 >> 28) * d
            assert 0 <= y <= y_up and (y - r * h) % q == 0
            ys.append(y)
        v, ok = S.round(ys, guard(y_up))
        true_v = (sum(Fraction(y, q) for y, q in zip(ys, src)) + Fraction(1, 2)).__floor__()
        centred = x if x <= Q // 2 else x - Q
        if ok:
            assert v == true_v
            hit += 1
            for T in dst[:3] + dst[-1:]:
                got = S.fold(ys, v, [(Q // q) % T for q in src], -Q % T, T)
                assert bits > 52 or 0 <= got < 1 << 60   # what the forward transform's bound starts from
                assert (got - centred) % T == 0
    assert hit >= 8
    # scale-and-round's first sum: folded digits (signed) and a full signed tensor word
    for T in dst[:2]:
        for lim in (0, 1):
            ys = [(y_sc - 1) if lim else -(dmax << (63 - bits)) for _ in src]
            for a in ((1 << 63) - 1, -(1 << 63), 0):
                cs, cv, w = [T - 1] * len(src), T - 1, T - 1
                v = S.round(ys, guard(y_sc))[0]
                got = S.fold(ys, v, cs, cv, T, (a, w))
                assert (got - (sum(y * c for y, c in zip(ys, cs)) + v * cv + a * w)) % T == 0


def eval_pos(w):
    return (w & ~1022) | ((w & 30) << 5) | ((w >> 4) & 62)


def test_storage_order_is_a_permutation_with_contiguous_lanes():
    assert sorted(eval_pos(w) for w in range(4096)) == list(range(4096))
    for e in (3, 4, 5):
        E = 1 << e
        for base in range(0, 4096, E):
            for j in range(E // 2):
                p = eval_pos(base) + 64 * j
                assert p % 2 == 0 and (eval_pos(base + 2 * j), eval_pos(base + 2 * j + 1)) == (p, p + 1)
        for warp in range(4096 // (32 * E)):   # one 16-byte access of a warp: runs of at least 128 bytes
            pos = sorted(eval_pos((32 * warp + t) * E) for t in range(32))
            runs = 1 + sum(1 for a, b in zip(pos, pos[1:]) if b != a + 2)
            assert runs * 4 <= 16 and all(p % 16 == 0 for i, p in enumerate(pos) if i == 0 or p != pos[i - 1] + 2)


@pytest.mark.parametrize("m", [10, 11, 12, 13, 14])
@pytest.mark.parametrize("e", [3, 4, 5])
def test_warp_exchanges_stay_inside_the_warp(m, e):
    """Passes with a low window of at most 5 bits on both sides of an exchange only synchronise the warp."""
    n = (m + e - 1) // e
    fwd = [max(m - (p + 1) * e, 0) for p in range(n)]
    inv = [p * e if (p + 1) * e <= m else m - e for p in range(n)]

    def words(W, warp):
        return {((t & ((1 << W) - 1)) | ((t >> W) << (W + e))) + (i << W)
                for t in range(32 * warp, 32 * warp + 32) for i in range(1 << e)}
    for lo in (fwd, inv):
        for a, b in zip(lo, lo[1:]):
            if a <= 5 and b <= 5:
                for warp in range((1 << (m - e)) // 32):
                    assert words(a, warp) == words(b, warp)


@pytest.mark.parametrize("bits", [45, 50, 55])
def test_product_of_two_run_time_factors(bits):
    """pm_mul_var: the 128-bit product of factors below 2^(bits+1) folded to a canonical residue."""
    rng = random.Random(bits)
    for N, L in [(1024, 1), (32768, 16)]:
        q = Params(N=N, L=L, alpha=1, prime_bits=bits).b[-1]
        d, s, M = (1 << bits) - q, bits - 32, (1 << 32) - 1
        top_v = (1 << (bits + 1)) - 1
        for a, b in [(0, 0), (top_v, top_v), (q - 1, q - 1), (top_v, 1)] + [(rng.randrange(top_v), rng.randrange(top_v)) for _ in range(50)]:
            a0, a1, b0, b1 = a & M, a >> 32, b & M, b >> 32
            lo = a0 * b0
            m = a1 * b0 + (lo >> 32) + a0 * b1
            top = a1 * b1 + (m >> 32)
            assert m < 1 << 64 and top < 1 << 64
            h0, h1 = ((m & M) | (top & M) << 32) >> s & M, u32(top >> s)
            g = h1 * d
            assert g < 1 << 64
            r = ((m & ((1 << s) - 1)) << 32 | lo & M) + ((g & ((1 << s) - 1)) << 32) + h0 * d + u32(g >> s) * d
            assert r < 1 << 63 and (r - a * b) % q == 0


@pytest.mark.parametrize("bits", [45, 50, 51, 55])
@pytest.mark.parametrize("terms", [1, 2, 8, 16])
def test_limb_sums_fold_to_the_sum_of_products(bits, terms):
    """pm_fold3 on the three limb sums of x y (x below 2^(bits+1), y below 2^bits; with (x0 + x1)(y0 + y1) as well):
    no sum wraps, the fold is congruent and below 2^62."""
    rng = random.Random(bits + terms)
    q = Params(N=32768, L=16, alpha=2, prime_bits=bits).b[-1]
    d, hs, s, M = (1 << bits) - q, (bits + 2) // 2, bits - 32, (1 << 32) - 1
    mask = (1 << hs) - 1
    for case in range(40):
        xs = [(2 << bits) - 1 if case == 0 else rng.randrange(2 << bits) for _ in range(terms)]
        ys = [(2 << bits) - 1 if case == 0 and terms <= 2 else q - 1 if case == 0 else rng.randrange(q) for _ in range(terms)]
        p00 = pm = p11 = pk = 0
        for x, y in zip(xs, ys):
            x0, x1, y0, y1 = u32(x & mask), u32(x >> hs), u32(y & mask), u32(y >> hs)
            p00, pm, p11 = p00 + x0 * y0, pm + x0 * y1 + x1 * y0, p11 + x1 * y1
            pk += u32(x0 + x1) * u32(y0 + y1)
        assert pk - p00 - p11 == pm
        if terms <= 8:
            assert pk < 1 << 64
        assert max(p00, pm, p11) <= 1 << 61 and p11 << (2 * hs - bits) <= 1 << 60
        H = (pm >> (bits - hs)) + (p11 << (2 * hs - bits))
        g = u32(H >> 32) * d
        r = p00 + ((pm & ((1 << (bits - hs)) - 1)) << hs) + ((g & ((1 << s) - 1)) << 32) + (H & M) * d + u32(g >> s) * d
        assert r < 1 << 62 and (r - sum(x * y for x, y in zip(xs, ys))) % q == 0
