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
