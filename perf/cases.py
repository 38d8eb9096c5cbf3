"""The work this library is timed on: calls of its public entry points (`bfhe.Context`, `circuits.Compiled`) over
the range of ring degrees, prime counts and batch sizes that its workloads use.

A case is a dict: `op` (what is called), the parameters (`N`, `L` data primes, `alpha` special primes, `bits` of
every prime, plaintext modulus 65537) and the batch `n`; `s` is a number of bits (bit-level operands, the bridge),
`mode` the bridge's accounting mode (0: one product per candidate and bit, 1: selection by public bits).
"""

import math

import numpy as np
import torch

from paper_2204_12201_gb300 import bfhe, circuits

T = 65537


def listed():
    return [
        # one gate on one pair of ciphertexts: the smallest multiplying call (bit-level code run one gate at a time)
        dict(name="gate_n4096_l2_x1", op="gate", N=4096, L=2, alpha=1, bits=50, n=1),
        # the small workload: 64 independent pairs at N = 4096
        dict(name="mul_n4096_l2_x64", op="mul", N=4096, L=2, alpha=1, bits=50, n=64),
        # the headline product: a batch of 64 pairs at N = 16384, 8 primes
        dict(name="mul_n16384_l8_x64", op="mul", N=16384, L=8, alpha=1, bits=50, n=64),
        # one step of the genotype job's Fermat chains: 156 candidates x 3 scores squared in one call
        dict(name="sqr_n16384_l8_x468", op="sqr", N=16384, L=8, alpha=1, bits=50, n=468),
        # the bridge workload's product: the largest ring, 16 + 2 primes, a small batch
        dict(name="mul_n32768_l16_x8", op="mul", N=32768, L=16, alpha=2, bits=50, n=8),
        # odd sizes: an odd number of primes above 50 bits, a ragged batch
        dict(name="mul_n8192_l5_b55_x7", op="mul", N=8192, L=5, alpha=1, bits=55, n=7),
        # a 16-bit comparator, all gates of a depth level in one launch, replayed as a CUDA graph
        dict(name="lt16_n8192_l4_x1", op="circuit", N=8192, L=4, alpha=1, bits=50, n=1, s=16),
        # SecureMod -> SecureUint<4> of three scores, with the products the paper counts
        dict(name="m2b_paper_n16384_l8_s4_x3", op="mod_to_bits", N=16384, L=8, alpha=1, bits=50, n=3, s=4, mode=0),
        # the same bridge at the largest ring, by selection
        dict(name="m2b_select_n32768_l16_s3_x1", op="mod_to_bits", N=32768, L=16, alpha=2, bits=50, n=1, s=3, mode=1),
        # SecureMod dot products: 32 tag vectors encrypted, weighted by public vectors for 3 classes, summed
        dict(name="dot_n16384_l8_x32", op="dot", N=16384, L=8, alpha=1, bits=50, n=32),
        # results read back
        dict(name="decrypt_n16384_l8_x64", op="decrypt", N=16384, L=8, alpha=1, bits=50, n=64),
        # SecureUint -> SecureMod of 64 nine-bit sums (additions only)
        dict(name="b2m_n4096_l2_s9_x64", op="bits_to_mod", N=4096, L=2, alpha=1, bits=50, n=64, s=9),
    ]


def draw(rng):
    """One more call of the same ranges; no costlier than the largest listed one."""
    most = max(work(c)["flops"] for c in listed())
    logn = rng.choice([12, 13, 14, 14, 15])
    few, many = {12: (1, 4), 13: (2, 6), 14: (3, 10), 15: (2, 16)}[logn]
    op = rng.choice(["mul", "mul", "mul", "sqr", "sqr", "gate", "circuit", "mod_to_bits", "dot", "decrypt", "bits_to_mod"])
    c = dict(op=op, N=1 << logn, L=rng.randint(few, many), alpha=rng.choice([1, 1, 2]),
             bits=rng.choice([50, 50, 50, 50, 45, 55]), n=round(2 ** rng.uniform(0, 9)))
    if op == "circuit":
        c.update(n=rng.randint(1, 4), s=rng.choice([8, 12, 16]))
    if op == "mod_to_bits":
        c.update(n=rng.randint(1, 4), s=rng.randint(2, 4), mode=rng.randint(0, 1))
    if op == "dot":
        c.update(n=1 << rng.randint(2, 5))
    if op == "bits_to_mod":
        c.update(s=rng.randint(2, 16), n=round(2 ** rng.uniform(0, 6)))
    while c["n"] > 1 and (work(c)["flops"] > most or work(c)["bytes"] > 4e9):
        c["n"] //= 2
    return c


def _slots(case, seed, n, hi):
    return np.random.Generator(np.random.PCG64(seed)).integers(0, hi, size=(n, case["N"]), dtype=np.int64)


def _netlist(case):
    net = circuits.Netlist()
    a, b = net.inputs(case["s"]), net.inputs(case["s"])
    return net, net.less_than(a, b)


def prepare(case, seed):
    """A context with its keys, room reserved for the batch, and encrypted operands."""
    op, n = case["op"], case["n"]
    seed %= 1 << 31
    ctx = bfhe.Context(N=case["N"], L=case["L"], alpha=case["alpha"], t=T, prime_bits=case["bits"])
    ctx.keygen(seed + 1)
    st = dict(op=op, ctx=ctx, case=case, seed=seed)

    def enc(k, hi=T, salt=0):
        return ctx.encrypt(torch.from_numpy(_slots(case, seed + salt, k, hi)).cuda(), seed + salt)

    if op in ("mul", "sqr", "gate"):
        ctx.reserve(n)
        st["a"] = enc(n, 2 if op == "gate" else T)
        if op != "sqr":
            st["b"] = enc(n, 2 if op == "gate" else T, 1)
    elif op == "circuit":
        net, out = _netlist(case)
        st["out"] = [out]
        st["cts"] = enc(2 * case["s"] * n, 2).view(2 * case["s"], n, 2, ctx.L, ctx.N)
        st["circ"] = circuits.Compiled(ctx, net, n)
        st["circ"].set_inputs(st["cts"])
        st["circ"].capture()
    elif op == "mod_to_bits":
        st["x"] = enc(n, 1 << case["s"])
    elif op == "dot":
        # tag genotypes in {0, 1, 2} and 6-bit weights for three classes
        st["slots"] = torch.from_numpy(_slots(case, seed, n, 3)).cuda()
        st["weights"] = torch.from_numpy(_slots(case, seed + 1, 3 * n, 64)).cuda()
    elif op == "decrypt":
        st["a"] = enc(n)
    elif op == "bits_to_mod":
        st["bits"] = enc(case["s"] * n, 2).view(case["s"], n, 2, ctx.L, ctx.N)
    else:
        raise ValueError(op)
    return st


def run(st):
    op, ctx = st["op"], st["ctx"]
    if op == "mul":
        return ctx.mul_relin(st["a"], st["b"])
    if op == "sqr":
        return ctx.mul_relin(st["a"], st["a"])
    if op == "gate":
        return ctx.bit_gate(bfhe.XOR, st["a"], st["b"])
    if op == "circuit":
        st["circ"].set_inputs(st["cts"])
        st["circ"].replay()
        return st["circ"].out(st["out"])
    if op == "mod_to_bits":
        s = st["case"]["s"]
        return ctx.mod_to_bits(st["x"], s, 0, (1 << s) - 1, st["case"]["mode"])
    if op == "dot":
        n = st["case"]["n"]
        x = ctx.mul_plain(ctx.encrypt(st["slots"], st["seed"]).repeat(3, 1, 1, 1), st["weights"])
        x = x.view(3, n, 2, ctx.L, ctx.N)
        while x.shape[1] > 1:
            h = x.shape[1] // 2
            x = ctx.add(x[:, :h].contiguous(), x[:, h:].contiguous())
        return x.view(3, 2, ctx.L, ctx.N)
    if op == "decrypt":
        return ctx.decrypt(st["a"])
    return ctx.bits_to_mod(st["bits"])


def _mul_modmuls(case, square):
    """64-bit modular multiplies of one relinearised product (K = L + 1 auxiliary primes)."""
    N, L, A = case["N"], case["L"], case["alpha"]
    K, QP, slots = L + 1, L + A, 2 if square else 4
    ntt = ((slots + 3) * (L + K) + (L + 2) * QP) * (N // 2) * int(math.log2(N))
    modup = slots * N * (L * (L - 1) // 2 + K * (L - 1))
    scale = 3 * N * (2 * L + 3 * K + L * (L - 1) // 2 + K * (L - 1) + K * (K - 1) // 2 + L * (K - 1))
    return ntt + modup + scale + 4 * (L + K) * N + 2 * L * QP * N + 2 * N * (L * A + L + A)


def work(case):
    """Bytes: operands, keys and results once.  flops: two per 64-bit modular multiply or addition."""
    op, N, L, A, n = case["op"], case["N"], case["L"], case["alpha"], case["n"]
    ct, key = 16 * L * N, 16 * L * (L + A) * N
    ntt = (N // 2) * int(math.log2(N))
    if op in ("mul", "sqr", "gate"):
        return dict(bytes=n * ct * (2 if op == "sqr" else 3) + key, flops=2 * n * _mul_modmuls(case, op == "sqr"))
    if op == "circuit":
        net, _ = _netlist(case)
        return dict(bytes=(2 * case["s"] + 1) * n * ct + key, flops=2 * n * net.n_mul * _mul_modmuls(case, False))
    if op == "mod_to_bits":
        m, s = n << case["s"], case["s"]
        per = 16 * _mul_modmuls(case, True) + (s * _mul_modmuls(case, False) if case["mode"] == 0 else 0)
        return dict(bytes=(s + 1) * n * ct + key, flops=2 * m * per)
    if op == "dot":
        m = 3 * n
        return dict(bytes=8 * N * (n + m) + 3 * ct + 16 * L * N,
                    flops=2 * (n * (3 * L * ntt + ntt + 2 * L * N) + m * (5 * L * ntt + ntt + 2 * L * N) + 3 * n * 2 * L * N))
    if op == "decrypt":
        return dict(bytes=n * (ct + 8 * N) + 8 * L * N,
                    flops=2 * n * (2 * L * ntt + ntt + N * (L * (L - 1) // 2 + 4 * L)))
    return dict(bytes=(case["s"] + 1) * n * ct, flops=4 * (case["s"] - 1) * n * 2 * L * N)


def exact(case, seed):
    """Decryption returns the encrypted slots; every other output is a ciphertext (residues of whole numbers)."""
    if case["op"] != "decrypt":
        return None
    return torch.from_numpy(_slots(case, seed % (1 << 31), case["n"], T))
