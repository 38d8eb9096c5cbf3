"""GPU: the linear kernels on buffers of both alignments."""

import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_linear_calls_on_buffers_aligned_to_one_word():
    """The row kernels take two words per access on 16-byte aligned buffers and one otherwise: same results."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    ctx = bfhe.Context(N=1024, L=3, alpha=1)
    n, s = 3, 4
    shape = (n, 2, ctx.L, ctx.N)
    words = n * 2 * ctx.L * ctx.N
    g = torch.Generator(device="cuda").manual_seed(5)
    q = torch.tensor(ctx.primes[:ctx.L], device="cuda").view(1, 1, ctx.L, 1)

    def off(t):   # the same words at an odd word offset
        flat = torch.empty(t.numel() + 1, dtype=torch.int64, device="cuda")[1:]
        flat.copy_(t.reshape(-1))
        return flat.view(t.shape)
    a, b = (torch.randint(0, 1 << 62, shape, device="cuda", generator=g) % q for _ in range(2))
    bits = torch.randint(0, 1 << 62, (s,) + shape, device="cuda", generator=g) % q
    want = [ctx.add(a, b), ctx.sub(a, b), ctx.add_const(a, 7), ctx.const_sub(7, a), ctx.mul_scalar(a, 12345),
            ctx.bits_to_mod(bits)]
    oa, ob, obits = off(a), off(b), off(bits)
    assert oa.data_ptr() % 16 == 8
    out = torch.empty(words + 1, dtype=torch.int64, device="cuda")[1:].view(shape)
    got = [ctx.add(oa, ob, out=out).clone(), ctx.sub(oa, b, out=out).clone(), ctx.add_const(oa, 7), ctx.const_sub(7, oa, out=out).clone(),
           ctx.mul_scalar(oa, 12345, out=out).clone(), ctx.bits_to_mod(obits, out=out).clone()]
    for x, y in zip(want, got):
        assert torch.equal(x, y)
    ref = (a.cpu() + b.cpu()) % q.cpu()
    assert torch.equal(want[0].cpu(), ref)
    ctx.close()


def test_gates_on_buffers_aligned_to_one_word():
    """Every gate with the equation fused into the multiply (16-byte aligned buffers) and as a kernel of its own."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    for alpha, bits in ((1, 50), (2, 55), (1, 40)):
        ctx = bfhe.Context(N=1024, L=2, alpha=alpha, prime_bits=bits)
        ctx.keygen(3)
        n = 3
        x, y, z = (ctx.encrypt(torch.randint(0, 2, (n, ctx.N), device="cuda"), s) for s in (1, 2, 3))
        px, py, pz = (ctx.decrypt(t) for t in (x, y, z))
        flat = torch.empty(x.numel() + 1, dtype=torch.int64, device="cuda")[1:].view(x.shape)
        want = {bfhe.AND: px & py, bfhe.OR: px | py, bfhe.XOR: px ^ py, bfhe.NAND: 1 - (px & py), bfhe.NOR: 1 - (px | py),
                bfhe.XNOR: 1 - (px ^ py), bfhe.MUX: torch.where(px == 1, py, pz)}
        for gate, w in want.items():
            got = ctx.bit_gate(gate, x, y, z)
            assert torch.equal(got, ctx.bit_gate(gate, x, y, z, out=flat))
            if bits >= 50:   # noise budget for one product
                assert torch.equal(ctx.decrypt(got), w)
        ctx.close()
