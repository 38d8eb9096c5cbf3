"""GPU: the guarded extensions where their rounded count is not certain, word for word against the oracle.

Operands a = (a0, a1) and b = (1, 0) or (0, 1) make the tensors (a0, a1, 0) and (0, a0, a1), so that a's words put both the lift and scale-and-round
(which extends the centred [t d]_Q) at, or one off, half of Q, where the guarded forms hand over to mixed radix: the one
for moduli 2^b - d (45 to 55 bits; two passes with a mark above 8 primes) and the general one (below 45 bits; two passes
from 10 primes), and mixed radix alone where it can be chosen.
"""

import pytest
import torch

from oracle import bfv
from oracle.params import Params
from tests.gpu_util import assert_ct_equal, cts_to_device, need_gpu

pytestmark = pytest.mark.gpu


def boundary_words(prm):
    """Words whose centred [t x]_Q, or which themselves, lie at or next to half of Q, and ordinary ones."""
    Q, t = prm.Q, prm.t
    h, inv = (Q - 1) // 2, pow(prm.t, -1, prm.Q)
    near = [(inv * (h + j)) % Q for j in (0, 1, -1, 2, -2)]
    for x in near:
        r = t * x % Q
        assert abs(2 * r - Q) <= 5
    return near + [h, h + 1, h - 1, 0, 1, Q - 1, 1234567 * t % Q]


@pytest.mark.parametrize("bits", [44, 45, 50, 55])
@pytest.mark.parametrize("L,alpha", [(1, 1), (3, 1), (8, 1), (9, 2), (10, 1), (16, 1)])
def test_products_at_the_rounding_boundaries(bits, L, alpha):
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    cfg = dict(N=1024, L=L, alpha=alpha, prime_bits=bits)
    prm, ctx = Params(**cfg), bfhe.Context(**cfg)
    ctx.keygen(5)
    keys = bfv.keygen(prm, 5)
    w = boundary_words(prm)
    n = len(w)
    a = ([w[k % n] for k in range(prm.N)], [w[(k // n + 3 * k) % n] for k in range(prm.N)])
    one, zero = [1] + [0] * (prm.N - 1), [0] * prm.N
    left, right = [a, (one, zero), a], [(one, zero), a, (zero, one)]
    want = [bfv.mul_relin(prm, keys, x, y) for x, y in zip(left, right)]
    da, db = cts_to_device(prm, left), cts_to_device(prm, right)
    assert_ct_equal(prm, ctx.mul_relin(da, db), want, "default, %d bits, L = %d" % (bits, L))
    for on in (False, True):
        if on and bits > 50:
            continue   # refused above 2^50
        ctx.set_fast_extension(on)
        assert_ct_equal(prm, ctx.mul_relin(da, db), want, "setting %s, %d bits, L = %d" % (on, bits, L))
    ctx.check()
    ctx.close()


@pytest.mark.parametrize("bits", [44, 45, 50, 55])
@pytest.mark.parametrize("L,t", [(1, 65537), (3, 12289), (8, 65537), (16, 65537), (3, 2)])
def test_decryption_at_the_rounding_boundaries(bits, L, t):
    """c1 = 0, so that c0 alone is rounded: words on both sides of a half of a plaintext step, and at the ends."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    cfg = dict(N=1024, L=L, alpha=1, t=t, prime_bits=bits)
    prm, ctx = Params(**cfg), bfhe.Context(**cfg)
    ctx.keygen(5)
    keys = bfv.keygen(prm, 5)
    Q = prm.Q
    w = [0, 1, Q - 1, Q // 2, Q // 2 + 1]
    for m in (0, 1, t // 2, t - 1):
        w += [((2 * m + 1) * Q // (2 * t) + j) % Q for j in (-1, 0, 1, 2)]
    ct = ([w[k % len(w)] for k in range(prm.N)], [0] * prm.N)
    want = torch.tensor(bfv.decrypt_poly(prm, keys, ct))
    dct = cts_to_device(prm, [ct])
    assert torch.equal(ctx.decrypt_poly(dct)[0].cpu(), want)
    ctx.set_fast_extension(False)
    assert torch.equal(ctx.decrypt_poly(dct)[0].cpu(), want)
    ctx.close()
