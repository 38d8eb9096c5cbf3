"""GPU: bfhe_set_fast_extension restores what bfhe_fast_extension returned."""

import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits,on", [(45, True), (50, True), (52, False), (55, False)])
def test_writing_back_the_setting_changes_nothing(bits, on):
    """At 9 data primes the guarded form for moduli 2^b - d takes scale-and-round in two launches, mixed radix in one, so
    the launches of a multiply tell which one runs: the guarded one before and after the setting is read and written
    back, above 2^50 too, where the setting is off and cannot be switched on."""
    need_gpu()
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    ctx = bfhe.Context(N=1024, L=9, alpha=1, prime_bits=bits)
    ctx.keygen(1)
    ct = ctx.encrypt(torch.randint(0, ctx.t, (2, ctx.N), device="cuda"), 2)

    def launches():
        n = bfhe.launch_count()
        ctx.mul_relin(ct[:1].contiguous(), ct[1:].contiguous())
        return bfhe.launch_count() - n
    guarded = launches()
    assert ctx.fast_extension == on
    ctx.set_fast_extension(ctx.fast_extension)
    assert launches() == guarded and ctx.fast_extension == on
    if on:   # both ways, then what it was
        ctx.set_fast_extension(False)
        assert launches() == guarded - 1 and not ctx.fast_extension
        ctx.set_fast_extension(True)
        assert launches() == guarded and ctx.fast_extension
    else:
        with pytest.raises(bfhe.BfheError):
            ctx.set_fast_extension(True)
        ctx.set_fast_extension(False)
        assert launches() == guarded and not ctx.fast_extension
    ctx.close()
