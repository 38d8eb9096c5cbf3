"""GPU: the multiply and the transforms on both sides of the rule that takes products modulo 2^b - d (45 to 55 bits)
against the oracle, word for word."""

import numpy as np
import pytest
import torch

from oracle import bfv
from oracle.params import Params
from paper_2204_12201_gb300 import inputs
from tests.gpu_util import assert_ct_equal, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [44, 45, 50, 55, 56])
@pytest.mark.parametrize("N,L,alpha", [(1024, 3, 1), (2048, 9, 2)])
def test_multiply_at_the_edges_of_the_product_rule(bits, N, L, alpha):
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    cfg = dict(N=N, L=L, alpha=alpha, prime_bits=bits)
    prm, ctx = Params(**cfg), bfhe.Context(**cfg)
    ctx.keygen(5)
    keys = bfv.keygen(prm, 5)
    y = inputs.slots(bits, 2, N)
    ct = ctx.encrypt(torch.from_numpy(y).cuda(), 7)
    a, b = (bfv.encrypt(prm, keys, [int(v) for v in y[i]], 7, i) for i in range(2))
    assert_ct_equal(prm, ct, [a, b], "encrypt")
    prod = ctx.mul_relin(ct[:1].contiguous(), ct[1:].contiguous())
    assert_ct_equal(prm, prod, [bfv.mul_relin(prm, keys, a, b)], "mul_relin")
    assert np.array_equal(ctx.decrypt(ct).cpu().numpy(), y)
    # the transform pair is the identity at the residues' extremes
    q = torch.tensor(ctx.primes[:L], device="cuda").view(1, L, 1)
    x = torch.randint(0, 1 << 62, (3, L, N), device="cuda") % q
    x[0] = q[0] - 1
    x[1] = 0
    z = ctx.ntt(x.clone())
    assert bool((z >= 0).all()) and bool((z < q).all())
    assert torch.equal(ctx.ntt(z.clone(), inverse=True), x)
    ctx.check()
    ctx.close()


@pytest.mark.parametrize("bits", [45, 50, 55])
@pytest.mark.parametrize("L,alpha", [(1, 1), (2, 1), (7, 2), (8, 1), (9, 1), (12, 1), (13, 1), (15, 2), (16, 1)])
def test_extension_forms_agree(bits, L, alpha):
    """The multiply with the extensions for moduli 2^b - d (the default) and with mixed radix alone, on uniform
    residues with every eighth coefficient at, or one off, the centring boundary, zero or the largest integer."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    N = 1024
    ctx = bfhe.Context(N=N, L=L, alpha=alpha, prime_bits=bits)
    ctx.keygen(9)
    Q = 1
    for p in ctx.primes[:L]:
        Q *= p
    g = torch.Generator(device="cuda").manual_seed(L)
    q = torch.tensor(ctx.primes[:L], device="cuda").view(1, 1, L, 1)
    a, b = (torch.randint(0, 1 << 62, (3, 2, L, N), device="cuda", generator=g) % q for _ in range(2))
    for t, x in enumerate([Q // 2, Q // 2 + 1, 0, 1, Q - 1, Q // 2 - 1]):
        a[0, :, :, t::8] = torch.tensor([x % p for p in ctx.primes[:L]], device="cuda").view(1, L, 1)
    new = [ctx.mul_relin(a, b), ctx.mul_relin(a, a)]
    assert ctx.lib.bfhe_set_fast_extension(ctx.h, 0) == 0
    old = [ctx.mul_relin(a, b), ctx.mul_relin(a, a)]
    for x, y in zip(new, old):
        assert torch.equal(x, y)
    ctx.check()
    ctx.close()


@pytest.mark.parametrize("bits,t", [(45, 65537), (50, 65537), (55, 65537), (50, 12289), (50, 2)])
@pytest.mark.parametrize("N,L", [(1024, 1), (1024, 8), (2048, 16)])
def test_decryption_forms_agree(bits, t, N, L):
    """Decryption's last step as folded sums and by mixed radix, on uniform residues and on words whose plaintext
    lies at a rounding boundary; the plain product (inverse of an evaluation-domain product) against slot products."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    ctx = bfhe.Context(N=N, L=L, alpha=1, t=t, prime_bits=bits)
    ctx.keygen(4)
    Q = 1
    for p in ctx.primes[:L]:
        Q *= p
    g = torch.Generator(device="cuda").manual_seed(bits + L)
    q = torch.tensor(ctx.primes[:L], device="cuda").view(1, 1, L, 1)
    ct = torch.randint(0, 1 << 62, (3, 2, L, N), device="cuda", generator=g) % q
    ct[1:, 1] = 0   # c1 = 0: c0 alone is decrypted, k/t Q + a half either side
    for m, x in enumerate([0, 1, Q - 1, Q // (2 * t), Q // (2 * t) + 1, Q // 2, Q // 2 + 1, 3 * Q // (2 * t)]):
        ct[1, 0, :, m::8] = torch.tensor([x % p for p in ctx.primes[:L]], device="cuda").view(L, 1)
    new = ctx.decrypt_poly(ct)
    assert ctx.lib.bfhe_set_fast_extension(ctx.h, 0) == 0
    assert torch.equal(new, ctx.decrypt_poly(ct))
    assert ctx.lib.bfhe_set_fast_extension(ctx.h, 1) in (0, -1)
    assert bool((new >= 0).all()) and bool((new < t).all())
    if t != 2 and L == 8:
        y = torch.from_numpy(inputs.slots(3, 2, N, hi=t)).cuda()
        w = torch.from_numpy(inputs.slots(5, 2, N, hi=t)).cuda()
        assert torch.equal(ctx.decrypt(ctx.mul_plain(ctx.encrypt(y, 1), w)), y * w % t)
    ctx.check()
    ctx.close()
