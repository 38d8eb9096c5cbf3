"""GPU: calls whose kernels overlap their predecessors' tails give what separately synchronised calls give."""

import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,L,n", [(1024, 2, 1), (4096, 2, 3), (16384, 8, 1), (32768, 3, 2)])
def test_back_to_back_calls_equal_synchronised_ones(N, L, n):
    """Products, linear calls, memory copies and torch operations on one stream, each reading what the one before it
    wrote (buffers reused), 20 rounds, against the same calls with the device idle in between."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    ctx = bfhe.Context(N=N, L=L, alpha=1)
    ctx.keygen(2)
    g = torch.Generator(device="cuda").manual_seed(N)
    a0 = ctx.encrypt(torch.randint(0, ctx.t, (n, N), device="cuda", generator=g), 1)
    b0 = ctx.encrypt(torch.randint(0, ctx.t, (n, N), device="cuda", generator=g), 2)

    def rounds(step):
        a, b, o = a0.clone(), b0.clone(), torch.empty_like(a0)
        for _ in range(20):
            for f in (lambda: ctx.mul_relin(a, b, out=o), lambda: ctx.add(o, a, out=a), lambda: ctx.mul_relin(a, a, out=o),
                      lambda: b.copy_(o), lambda: ctx.sub(b, a, out=b), lambda: ctx.bit_gate(bfhe.XOR, a, b, out=o),
                      lambda: a.copy_(o)):
                f()
                step()
        return a, b, ctx.decrypt(a)
    want = rounds(torch.cuda.synchronize)
    for _ in range(3):
        for x, y in zip(want, rounds(lambda: None)):
            assert torch.equal(x, y)
    ctx.close()
