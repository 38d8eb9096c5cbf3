"""A circuit recorded as a CUDA graph works in the context's scratch arena, which a larger call on the same context frees."""

import pytest
import torch

from paper_2204_12201_gb300 import circuits
from tests.gpu_util import need_gpu


def test_replay_records_again_when_the_arena_has_moved():
    """Host side alone: a graph whose arena is gone is never launched."""
    log = []

    class Graph:
        def __init__(self, gen):
            self.gen = gen

        def replay(self):
            log.append((self.gen, ctx.scratch_generation))

    class Ctx:
        scratch_generation = 1

    ctx = Ctx()
    c = object.__new__(circuits.Compiled)
    c.ctx, c.graph, c.generation = ctx, Graph(1), 1

    def capture():
        c.graph, c.generation = Graph(ctx.scratch_generation), ctx.scratch_generation
    c.capture = capture
    c.replay()
    ctx.scratch_generation = 2
    c.replay()
    c.replay()
    ctx.scratch_generation = 5
    c.replay()
    assert log == [(1, 1), (2, 2), (2, 2), (5, 5)]


@pytest.mark.gpu
def test_replay_after_a_larger_call():
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    N = 1024
    ctx = bfhe.Context(N=N, L=3, alpha=1)
    assert ctx.scratch_generation == 0
    ctx.keygen(1)
    net = circuits.Netlist()
    a, b = net.inputs(2), net.inputs(2)
    out = net.less_than(a, b)
    comp = circuits.Compiled(ctx, net, 1)
    bits = torch.randint(0, 2, (4, N), device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    comp.set_inputs(ctx.encrypt(bits, 5).view(4, 1, 2, ctx.L, N))
    comp.capture()
    first, gen = comp.graph, ctx.scratch_generation
    comp.replay()
    want = comp.out([out]).clone()
    assert comp.graph is first and ctx.scratch_generation == gen == comp.generation
    ctx.reserve(64)   # a larger arena in another place
    assert ctx.scratch_generation == gen + 1
    for _ in range(2):
        comp.wires[net.n_inputs:].zero_()
        comp.replay()
        assert torch.equal(comp.out([out]), want)
    assert comp.graph is not first and comp.generation == gen + 1
    ctx.close()
