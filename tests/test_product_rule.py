"""Which parameter sets take products modulo 2^b - d: the rule, evaluated by the library, over the supported sets."""

import ctypes
import os

import pytest
import torch

from paper_2204_12201_gb300 import bfhe, build, inputs
from tests.gpu_util import need_gpu

# (bits, log2 N, special primes) -> the least number of data primes at which the transforms' growth bound fails; where a
# set with 45 to 55 bits is not named, it never does
FAILS_FROM = {(54, 15, 1): 22, (54, 15, 2): 21, (55, 14, 1): 29, (55, 14, 2): 28, (55, 15, 1): 11, (55, 15, 2): 10}


def bounded(bits, logN, d):
    if not os.path.exists(build.lib_path()):
        build.build()
    fn = ctypes.CDLL(build.lib_path())._Z10pm_boundedjjm   # pm_bounded(uint32_t, uint32_t, uint64_t)
    fn.argtypes, fn.restype = [ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint64], ctypes.c_bool
    return fn(bits, logN, d)


def largest_d(bits, logN, L, alpha):
    if not os.path.exists(build.lib_path()):
        build.build()
    return max((1 << bits) - q for q in bfhe.param_primes(1 << logN, L, alpha, prime_bits=bits)[0])


@pytest.mark.parametrize("bits", range(44, 57))
def test_sets_that_take_the_products(bits):
    for logN in range(10, 16):
        for alpha in (1, 2):
            first = FAILS_FROM.get((bits, logN, alpha), 33)
            for L in {1, 8, 16, 32, min(first, 32), min(first, 33) - 1}:
                want = 45 <= bits <= 55 and L < first
                assert bounded(bits, logN, largest_d(bits, logN, L, alpha)) == want, (bits, logN, L, alpha)


@pytest.mark.parametrize("bits,logN,L,alpha", [(45, 15, 32, 2), (50, 15, 16, 2), (52, 15, 32, 2), (55, 15, 10, 1), (55, 14, 16, 2)])
def test_the_rule_covers_every_stage(bits, logN, L, alpha):
    """Where the rule holds, the sum of the start and of one product's bound per stage stays a signed 64-bit word: the
    product of a word a below 2^63 is P + 2^k ql + 4d qh with |P| < 2^32 2^k + 2^31 2^k, ql < 2^32, |qh| < 3 2^29."""
    d, k = largest_d(bits, logN, L, alpha), bits - 30
    product = 3 * 2 ** (31 + k) + 2 ** (32 + k) + 4 * d * 3 * 2 ** 29
    assert bounded(bits, logN, d)
    forward = 2 ** 60 if bits <= 52 else 2 ** (bits + 1) + d * 2 ** (63 - bits)
    inverse = 32 * (2 ** bits + d * 2 ** (63 - bits))   # the first pass adds words with w = 1
    assert max(forward, inverse) + logN * product < 2 ** 63


@pytest.mark.gpu
@pytest.mark.parametrize("L", [10, 11])
def test_both_sides_of_the_rule_at_the_largest_ring(L):
    """55 bits at N = 32768: 10 data primes are the last set with the products, 11 take the general kernels.  Transforms of
    the residues' extremes are inverted, and ciphertext and plain products decrypt to the slots' products."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    N = 32768
    assert bounded(55, 15, largest_d(55, 15, L, 1)) == (L == 10)
    ctx = bfhe.Context(N=N, L=L, alpha=1, prime_bits=55)
    ctx.keygen(3)
    q = torch.tensor(ctx.primes[:L], device="cuda").view(1, L, 1)
    x = torch.randint(0, 1 << 62, (4, L, N), device="cuda", generator=torch.Generator(device="cuda").manual_seed(L)) % q
    x[0] = q[0] - 1
    x[1] = (q[0] - 1) * (torch.arange(N, device="cuda") % 2)
    x[2, :, 1:] = 0
    z = ctx.ntt(x.clone())
    assert bool((z >= 0).all()) and bool((z < q).all())
    assert torch.equal(z[2], x[2, :, :1].expand(L, N))   # a constant evaluates to itself everywhere
    assert torch.equal(ctx.ntt(z.clone(), inverse=True), x)
    y = torch.from_numpy(inputs.slots(7, 3, N)).cuda()
    ct = ctx.encrypt(y, 5)
    a, b, w = ct[:1].contiguous(), ct[1:2].contiguous(), y[2:3]
    assert torch.equal(ctx.decrypt(ctx.mul_relin(a, b)), y[:1] * y[1:2] % ctx.t)
    assert torch.equal(ctx.decrypt(ctx.mul_relin(a, a)), y[:1] * y[:1] % ctx.t)
    assert torch.equal(ctx.decrypt(ctx.mul_plain(b, w)), y[1:2] * w % ctx.t)
    ctx.check()
    ctx.close()
