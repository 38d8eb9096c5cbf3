#!/usr/bin/env python
"""Benchmark of the bridged-FHE hot path on GB300: one JSON line on rank 0.

A step is one pass of the whole hot path over one batch: the genotype-shaped
job at N = 16384 (8 data primes of 50 bits + 1 special, t = 65537):
encrypt 32 tag-genotype slot vectors (2000 targets x 8 individuals packed in
16000 of the 16384 slots), SecureMod dot products with 6-bit public weights
for 3 classes (mul_plain + adds), the bridge SecureMod -> SecureUint<12>
(Eq. 2 / Listings 7-8, paper mode: every candidate c in 0..4095 runs 16
chained squarings and 12 ANDs), a levelised 3-way argmax circuit over the
bits, and decryption of the two index bits.  The metric counts the
relinearised ciphertext multiplies the step performs (op counter) per
second.  Extra keys report the batched-vs-per-op mul_relin rate at
N = 16384, bit-gates/s of the 16-bit comparator and 16x16 multiplier
circuits at N = 8192 (eager and CUDA-graph), the modmul probe, and the
serving loop's p50/p99 latency and throughput against one-request-at-a-time
per-op launches at two arrival rates.

--impl reference times the CPU oracle (the plain arbitrary-precision BFV the
library is checked against) on the host cores instead.
"""

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "mul_relin/sec at N=16384 and bit-gates/sec, batched vs per-op, bit-exact; % roofline"
UNIT = "mul_relin/s"
WL = dict(N=16384, L=8, alpha=1, t=65537)
N_IND, N_TARGETS, N_TAGS, N_CLASSES, S_BITS = 8, 2000, 32, 3, 12
WORKLOAD = ("genotype-shaped job: BFV N=16384, 8x50-bit data primes + 1 special, t=65537; "
            "2000 targets x 8 individuals slot-packed, 32 tag ciphertexts, 3-class 6-bit-weight "
            "SecureMod dot products, mod_to_bits s=12 over c in 0..4095 (paper mode), 3-way argmax "
            "circuit, decrypt")
CPU_SAMPLE_N = 16384


# --------------------------------------------------------------------------- helpers
def base_config():
    """The workload fields both arms report."""
    return {"workload": WORKLOAD, "N": WL["N"], "L": WL["L"], "alpha": WL["alpha"], "t": WL["t"]}


def combine_ranks(dist, ms, units, device):
    """Max over ranks of the timed-region duration and the units all ranks processed."""
    if dist is None:
        return ms, units
    import torch
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    u = torch.tensor([units], dtype=torch.int64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t.item()), int(u.item())

def ntt_traffic_per_limb(kernel):
    """DRAM bytes per limb of the dominant kernel from the committed ncu summary, or None when the
    kernel's sources changed since those counters were taken (the summary records their hash)."""
    import hashlib
    here = os.path.dirname(os.path.abspath(__file__))
    path = os.path.join(here, "profiles", "%s_traffic_genotype_N16384.md" % kernel)
    if not os.path.exists(path):
        return None
    h = hashlib.sha256()
    csrc = os.path.join(here, "paper_2204_12201_gb300", "csrc")
    with open(os.path.join(csrc, "ntt.cu"), "rb") as fh:
        h.update(fh.read())
    # the device modular arithmetic the transforms use (one section of common.cuh)
    with open(os.path.join(csrc, "common.cuh"), "rb") as fh:
        text = fh.read()
    a = text.index(b"// ---") if b"// ---" in text else 0
    b = text.index(b"exact base extension tables") if b"exact base extension tables" in text else len(text)
    h.update(text[a:b])
    fields = {}
    with open(path) as fh:
        for line in fh:
            if line.startswith("- `") and ": `" in line:
                k, v = line[2:].strip().split(": ", 1)
                fields[k.strip("`")] = v.split("`")[1]
    if fields.get("sources_sha256") != h.hexdigest():
        return None
    return float(fields["dram_bytes_per_limb"])


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "sm_max_mhz": 2070.0}, "fallback"


def alu_peak_modmul_per_s(sms, mhz, slots=10):
    """Derived integer-pipe peak: 64 32-bit IMAD issue slots per SM per clock; a product modulo 2^b - d takes
    10 of them (five 32x32->64 wide multiply-adds at 2 slots).  A 64-bit Shoup product, which the library's
    probe times, takes 16 (four wide products of the high half, and one wide + two narrow products for each
    of the two low halves)."""
    return sms * 64.0 * mhz * 1e6 / slots


def kernel_rooflines(prof, alu_peak, hbm_gbs):
    """Per kernel class: its roofline time is the slower of the algorithmic modmuls at the integer-pipe peak
    and the algorithmic DRAM bytes at the measured copy bandwidth; frac = that time / the measured time."""
    out = {}
    for k, (ms, _, work, nbytes) in prof.items():
        if ms <= 0:
            continue
        t_alu, t_hbm = work / alu_peak, nbytes / (hbm_gbs * 1e9)
        out[k] = {"bound": "alu" if t_alu >= t_hbm else "hbm", "frac": round(max(t_alu, t_hbm) / (ms / 1e3), 3),
                  "alu_frac": round(t_alu / (ms / 1e3), 3), "hbm_frac": round(t_hbm / (ms / 1e3), 3)}
    return out


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons while running."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.proc = None
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(gpu_index), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        self.proc.wait()
        self.f.flush()
        self.f.seek(0)
        rows = [r.split(",") for r in self.f.read().strip().splitlines() if r.strip()]
        os.unlink(self.f.name)
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            try:
                sm.append(float(r[1]))
                mx.append(float(r[2]))
            except (ValueError, IndexError):
                continue
            for name, v in zip(names, r[5:9]):
                if v.strip().lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# --------------------------------------------------------------------------- CPU oracle leg
def _oracle_mul_relin(args):
    """One oracle mul_relin on random ciphertexts and a random-key stand-in; returns seconds."""
    N, L, alpha, seed = args
    import random
    sys.path.insert(0, ROOT)
    from oracle import bfv
    from oracle.params import Params
    prm = Params(N=N, L=L, alpha=alpha)
    rng = random.Random(seed)
    Q, PQ = prm.Q, prm.P * prm.Q
    ct = lambda: ([rng.randrange(Q) for _ in range(N)], [rng.randrange(Q) for _ in range(N)])
    a, b = ct(), ct()
    rlk = [([rng.randrange(PQ) for _ in range(N)], [rng.randrange(PQ) for _ in range(N)]) for _ in range(L)]
    keys = bfv.Keys([0] * N, None, None, rlk)
    t0 = time.perf_counter()
    bfv.mul_relin(prm, keys, a, b)
    return time.perf_counter() - t0


def cpu_pool_start(n_procs, N=CPU_SAMPLE_N):
    import multiprocessing as mp
    ctx = mp.get_context("spawn")
    pool = ctx.Pool(n_procs)
    res = pool.map_async(_oracle_mul_relin, [(N, WL["L"], WL["alpha"], 100 + i) for i in range(n_procs)])
    return pool, res


def cpu_pool_finish(pool, res, n_procs, wall0):
    times = res.get()
    wall = time.perf_counter() - wall0
    pool.close()
    pool.join()
    return {"value": n_procs / max(times), "unit": UNIT, "cores": n_procs, "kind": "oracle",
            "sample": "%d oracle mul_relin at N=16384, L=8, alpha=1 (random ciphertexts, random-key "
                      "stand-in), one per process in parallel; rate = count / slowest process" % n_procs,
            "per_op_s": round(statistics.mean(times), 2), "wall_s": round(wall, 1)}


def host_cores():
    try:
        return len(os.sched_getaffinity(0))
    except AttributeError:
        return os.cpu_count() or 1


# --------------------------------------------------------------------------- reference arm
def run_reference(args, rank, world):
    if rank != 0:
        return 0
    n_procs = max(1, min(16, host_cores()))
    import multiprocessing as mp
    pool = mp.get_context("spawn").Pool(n_procs)
    for w in range(args.warmup):   # untimed: module import and a small op per process
        pool.map(_oracle_mul_relin, [(1024, 2, 1, 900 + w * 100 + i) for i in range(n_procs)])
    t0 = time.perf_counter()
    done = 0
    for s in range(args.steps):
        pool.map(_oracle_mul_relin, [(CPU_SAMPLE_N, WL["L"], WL["alpha"], s * 100 + i) for i in range(n_procs)])
        done += n_procs
    el = time.perf_counter() - t0
    pool.close()
    pool.join()
    v = done / el
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": el / args.steps * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int (exact)",
            "data": "synthetic",
            "config": {**base_config(), "parallelism": "host cores"},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": n_procs, "kind": "oracle",
                             "sample": "the step's multiply: %d oracle mul_relin at N=%d, L=%d, alpha=%d per step "
                                       "(random ciphertexts, random-key stand-in), one per process"
                                       % (n_procs, CPU_SAMPLE_N, WL["L"], WL["alpha"])},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# --------------------------------------------------------------------------- extras
def config1_extras(torch, bfhe, circuits, timed):
    """The small workload (N = 4096, 2 data primes + 1 special, t = 65537): 64 independent ciphertext pairs
    through add and mul_relin, the 8-bit ripple-carry adder over 64 batched operand pairs (bits as 0/1
    ciphertexts; 15 multiplies per adder), then bits_to_mod (Listing 5) on the 64 nine-bit sums."""
    from paper_2204_12201_gb300 import inputs
    ctx = bfhe.Context(N=4096, L=2, alpha=1)
    ctx.keygen(11)
    N, n = 4096, 64
    a = ctx.encrypt(torch.from_numpy(inputs.slots(501, n, N)).cuda(), 501)
    b = ctx.encrypt(torch.from_numpy(inputs.slots(502, n, N)).cuda(), 502)
    o = torch.empty_like(a)
    r = {"ciphertext_pairs": n}
    r["add_per_s"] = n / timed(lambda: ctx.add(a, b, out=o), 20) * 1e3
    r["mul_relin_per_s"] = n / timed(lambda: ctx.mul_relin(a, b, out=o), 10) * 1e3
    net = circuits.Netlist()
    x, y = net.inputs(8), net.inputs(8)
    sum_w = net.ripple_add(x, y)
    X, Y = inputs.slots(503, n, N, hi=256), inputs.slots(504, n, N, hi=256)
    planes = torch.from_numpy(__import__("numpy").concatenate([inputs.bit_planes(X, 8), inputs.bit_planes(Y, 8)]))
    comp = circuits.Compiled(ctx, net, n)
    comp.set_inputs(ctx.encrypt(planes.reshape(-1, N).cuda(), 505).view(16, n, 2, 2, N))
    ms_e = timed(comp.run, 3)
    comp.capture()
    ms_g = timed(comp.replay, 5)
    r["adder8_gates"] = net.n_mul
    r["adder8_bit_gates_per_s_eager"] = net.n_mul * n / ms_e * 1e3
    r["adder8_bit_gates_per_s_graph"] = net.n_mul * n / ms_g * 1e3
    bits = comp.out(sum_w).contiguous()
    m = torch.empty_like(a)
    r["bits_to_mod_per_s"] = n / timed(lambda: ctx.bits_to_mod(bits, out=m), 20) * 1e3
    ok = bool((ctx.decrypt(m).cpu() == torch.from_numpy(X + Y)).all())
    r["adder_and_bits_to_mod_decrypt_correctly"] = ok
    del comp
    ctx.close()
    return r


def config3_extras(torch, bfhe, timed):
    """The bridge workload (N = 32768, 16 data primes + 2 special, t = 65537): batched mul_relin and squarings,
    and one SecureMod -> SecureUint<8> conversion (Eq. 2, Listings 7-8, paper mode) of a slot-packed x in
    [0, 255] over c in 0..255: 256 chains of 16 squarings and 8 ANDs each (6,144 multiplies), with its
    candidate tiles eager and replayed from a CUDA graph."""
    from paper_2204_12201_gb300 import inputs
    ctx = bfhe.Context(N=32768, L=16, alpha=2)
    ctx.keygen(13)
    N, B = 32768, 16
    a = ctx.encrypt(torch.from_numpy(inputs.slots(801, B, N)).cuda(), 801)
    b = ctx.encrypt(torch.from_numpy(inputs.slots(802, B, N)).cuda(), 802)
    o = torch.empty_like(a)
    r = {"batch": B, "base_extension": "guarded fast" if ctx.fast_extension else "exact"}
    r["mul_relin_batched_per_s"] = B / timed(lambda: ctx.mul_relin(a, b, out=o), 3) * 1e3
    r["squarings_batched_per_s"] = B / timed(lambda: ctx.mul_relin(a, a, out=o), 3) * 1e3
    del a, b, o
    xs = inputs.slots(701, 1, N, hi=256)
    x = ctx.encrypt(torch.from_numpy(xs).cuda(), 701)
    bits = torch.empty(8, 1, 2, 16, N, dtype=torch.int64, device="cuda")
    conv = {}
    for graph in (False, True):
        ctx.set_graph_tiles(graph)
        ms = timed(lambda: ctx.mod_to_bits(x, 8, 0, 255, bfhe.PAPER, out=bits), 2)
        conv["graph" if graph else "eager"] = {"ms": round(ms, 1), "conversions_per_s": 1e3 / ms,
                                               "mul_relin_per_s": 256 * 24 / ms * 1e3}
    ctx.set_graph_tiles(False)
    ok = all(bool((ctx.decrypt(bits[k].contiguous()).cpu().numpy() == ((xs >> k) & 1)).all()) for k in range(8))
    r["mod_to_bits_c0_255"] = conv
    r["mod_to_bits_decrypts_correctly"] = ok
    ctx.close()
    return r


def extras(torch, bfhe, circuits, ctx16):
    out = {}
    N = ctx16.N
    # batched vs per-op mul_relin at N = 16384
    B = 64
    a = ctx16.encrypt(torch.randint(0, 65537, (B, N), dtype=torch.int64, device="cuda"), 7)
    b = ctx16.encrypt(torch.randint(0, 65537, (B, N), dtype=torch.int64, device="cuda"), 8)
    o = torch.empty_like(a)

    def timed(fn, reps):
        fn()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            fn()
        e1.record()
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / reps

    ms_b = timed(lambda: ctx16.mul_relin(a, b, out=o), 5)
    # the same batched multiply with each base extension forced (same words, other speed)
    default = ctx16.fast_extension
    for fast in (False, True):
        ctx16.set_fast_extension(fast)
        ms_x = timed(lambda: ctx16.mul_relin(a, b, out=o), 5)
        out["mul_relin_batched_%s_extension_per_s" % ("fast" if fast else "exact")] = B / ms_x * 1e3
    ctx16.set_fast_extension(default)
    ms_p = timed(lambda: [ctx16.mul_relin(a[i:i + 1], b[i:i + 1], out=o[i:i + 1]) for i in range(B)], 3)
    out["mul_relin_batched_per_s"] = B / ms_b * 1e3
    out["mul_relin_per_op_per_s"] = B / ms_p * 1e3
    # graph-captured per-op sequence
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        with torch.cuda.graph(g, stream=s):
            for i in range(B):
                ctx16.mul_relin(a[i:i + 1], b[i:i + 1], out=o[i:i + 1])
    torch.cuda.current_stream().wait_stream(s)
    ms_g = timed(g.replay, 3)
    out["mul_relin_per_op_graph_per_s"] = B / ms_g * 1e3
    del g
    # bit-level circuits at N = 8192, L = 4
    ctx8 = bfhe.Context(N=8192, L=4, alpha=1)
    ctx8.keygen(3)
    rng = torch.Generator().manual_seed(5)
    for name, build in (("lt16", lambda n: [n.less_than(n.inputs(16), n.inputs(16))]),
                        ("mul16", lambda n: n.multiply(n.inputs(16), n.inputs(16)))):
        net = circuits.Netlist()
        build(net)
        comp = circuits.Compiled(ctx8, net, 1)
        ops = torch.randint(0, 2, (net.n_inputs, 8192), generator=rng, dtype=torch.int64).cuda()
        comp.set_inputs(ctx8.encrypt(ops, 9).view(net.n_inputs, 1, 2, 4, 8192))
        ms_e = timed(comp.run, 2)
        comp.capture()
        ms_gr = timed(comp.replay, 3)
        out["bit_gates_per_s_%s_eager" % name] = net.n_mul / ms_e * 1e3
        out["bit_gates_per_s_%s_graph" % name] = net.n_mul / ms_gr * 1e3
        out["%s_gates" % name] = net.n_mul
        del comp
        # the per-op baseline: one gate per call (one multiply launch sequence per gate)
        po = circuits.Compiled(ctx8, net, 1, per_op=True)
        po.set_inputs(ctx8.encrypt(ops, 9).view(net.n_inputs, 1, 2, 4, 8192))
        out["bit_gates_per_s_%s_per_op" % name] = net.n_mul / timed(po.run, 1) * 1e3
        del po
    ctx8.close()
    out["modmul_probe_per_s"] = bfhe.probe_modmul(torch.cuda.current_device())
    # Fibonacci (Listings 3 and 4), 8-bit words, 10 iterations, one input per slot, at the paper's
    # ring degree N = 32768: bit-level vs bridged, both with 28 data primes (an insecure, test-only modulus
    # large enough for the bit-level program's multiplicative depth of 36, so that both decrypt)
    from paper_2204_12201_gb300 import workloads
    ctx32 = bfhe.Context(N=32768, L=28, alpha=1)
    ctx32.keygen(4)
    vals = torch.randint(0, 12, (1, 32768), generator=rng, dtype=torch.int64).cuda()
    fib = [0, 1]
    while len(fib) < 10:
        fib.append(fib[-1] + fib[-2])
    fib += [0, 0]                      # inputs 10 and 11 are never reached in 10 iterations
    want = torch.tensor(fib, dtype=torch.int64, device="cuda")[vals]
    fo = {}
    for kind in ("bits", "bridged"):
        job = workloads.FibonacciJob(ctx32, kind, 8, 10)
        job.set_inputs(vals, 12)
        ms_e = timed(job.run, 2)
        ok = bool(torch.equal(job.decrypt(), want))
        job.circ.capture()
        ms_gr = timed(job.circ.replay, 2)
        fo[kind] = {"ms_eager": round(ms_e, 2), "ms_graph": round(ms_gr, 2), "mul_relin": job.net.n_mul,
                    "mul_levels": job.circ.depth, "instances_per_run": 32768, "decrypts_correctly": ok}
        del job
    ctx32.close()
    # the same bit-level program at t = 2 (no batching: one instance per ciphertext, XOR free)
    ctx2 = bfhe.Context(N=32768, L=16, alpha=1, t=2)
    ctx2.keygen(4)
    job = workloads.FibonacciJob(ctx2, "bits", 8, 10, n=1)
    job.set_inputs(vals[:, :1].contiguous(), 12)
    ms_e = timed(job.run, 2)
    ok = bool(torch.equal(job.decrypt(), want[:, :1]))
    job.circ.capture()
    ms_gr = timed(job.circ.replay, 2)
    fo["bits_t2"] = {"ms_eager": round(ms_e, 2), "ms_graph": round(ms_gr, 2), "mul_relin": job.net.n_mul,
                     "mul_levels": job.circ.depth, "instances_per_run": 1, "decrypts_correctly": ok}
    del job
    ctx2.close()
    both = fo["bits"]["decrypts_correctly"] and fo["bridged"]["decrypts_correctly"]
    # a speed ratio is reported only where both programs decrypt to the right values
    fo["bridged_speedup_graph"] = round(fo["bits"]["ms_graph"] / fo["bridged"]["ms_graph"], 2) if both else None
    fo["moduli"] = {"bits": "28 x 50-bit data primes", "bridged": "28 x 50-bit data primes",
                    "bits_t2": "16 x 50-bit data primes"}
    out["fibonacci_n32768_8bit_10iter"] = fo
    out["config1_n4096_l2"] = config1_extras(torch, bfhe, circuits, timed)
    out["config3_n32768_l16"] = config3_extras(torch, bfhe, timed)
    # serving: a Poisson stream of mixed requests (N in {4096, 8192, 16384}, 1..16 squarings,
    # 1..64 ciphertexts), continuous batching vs one request at a time with per-op launches
    from paper_2204_12201_gb300 import serving
    sv = {}
    for rate in (20.0, 200.0):
        r = serving.demo(n_req=60, rate=rate, seed=11)
        sv["rate_%d" % int(rate)] = {k: {kk: (round(vv, 4) if isinstance(vv, float) else vv) for kk, vv in v.items()}
                                     for k, v in r.items() if isinstance(v, dict)}
    out["serving"] = sv
    return {k: (round(v, 1) if isinstance(v, float) else v) for k, v in out.items()}


# --------------------------------------------------------------------------- profiling cases
def run_case(args):
    """One small, self-contained launch sequence for capturing one kernel family under ncu (no JSON line):
    `ntt`: forward + inverse over polys x L limbs; `mul`: batched mul_relin of n pairs. The measured rounds
    sit inside the NVTX range "bfhe_cases", so that ncu can skip the set-up (keygen, encryption) with
    --nvtx --nvtx-include "bfhe_cases/"."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import bfhe
    ctx = bfhe.Context(N=args.N, L=args.L, alpha=args.alpha)
    if args.case == "ntt":
        x = torch.randint(0, 1 << 40, (args.polys, args.L, args.N), dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("bfhe_cases")
        for _ in range(args.rounds):
            ctx.ntt(x)
            ctx.ntt(x, inverse=True)
    else:
        ctx.keygen(1)
        g = torch.Generator().manual_seed(3)
        ys = torch.randint(0, 65537, (2 * args.n, args.N), generator=g, dtype=torch.int64).cuda()
        ct = ctx.encrypt(ys, 5)
        x, y = ct[: args.n].contiguous(), ct[args.n:].contiguous()
        out = torch.empty_like(x)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("bfhe_cases")
        for _ in range(args.rounds):
            ctx.mul_relin(x, y if args.case == "mul" else x, out=out)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    ctx.close()
    print("case %s ok" % args.case)
    return 0


# --------------------------------------------------------------------------- main
def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu", action="store_true", help="skip the oracle CPU leg")
    ap.add_argument("--no-extras", action="store_true")
    ap.add_argument("--case", choices=["ntt", "mul", "square"],
                    help="run one small profiling case instead of the benchmark (see run_case)")
    ap.add_argument("--N", type=int, default=16384)
    ap.add_argument("--L", type=int, default=8)
    ap.add_argument("--alpha", type=int, default=1)
    ap.add_argument("--polys", type=int, default=256)
    ap.add_argument("--n", type=int, default=32)
    ap.add_argument("--rounds", type=int, default=3)
    args = ap.parse_args()
    if args.case:
        return run_case(args)
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        return run_reference(args, rank, world)
    args.warmup = max(3, args.warmup)

    # the oracle leg starts first (spawned processes, before any GPU call) and runs on the host
    # cores while the GPU sets up and warms up; it is collected before the timed region
    cpu = None
    n_cpu = 0
    if rank == 0 and world == 1 and not args.no_cpu:
        n_cpu = max(1, min(16, host_cores() - 2))
        wall0 = time.perf_counter()
        cpu = cpu_pool_start(n_cpu) + (wall0,)

    import numpy as np
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2204_12201_gb300 import autotune, bfhe, circuits, workloads

    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    tuned = autotune.tune(ring_degrees=(4096, 8192, 16384, 32768))   # NTT shapes and multiply tiles
    ctx = bfhe.Context(N=WL["N"], L=WL["L"], alpha=WL["alpha"], t=WL["t"], device=local)
    ctx.keygen(1 + rank)
    job = workloads.GenotypeJob(ctx, n_tags=N_TAGS, s_bits=S_BITS)
    Gs, Ws = workloads.genotype_inputs(1004 + rank, WL["N"], N_IND, N_TARGETS, N_TAGS, N_CLASSES)
    G_dev = torch.from_numpy(Gs).cuda()
    W_dev = torch.from_numpy(Ws).cuda()
    for w in range(args.warmup):
        job.run(G_dev, W_dev, seed=10 + w)
    torch.cuda.synchronize()
    cpu_line = None
    if cpu is not None:
        cpu_line = cpu_pool_finish(cpu[0], cpu[1], n_cpu, cpu[2])

    # ---------------- timed region: K steps, inputs resident in HBM
    ctx.op_counts(reset=True)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    clocks = Clocks(local)
    launches0 = bfhe.launch_count()
    ctx.profile(True)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for s in range(args.steps):
        res = job.run(G_dev, W_dev, seed=100 + s)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    prof = ctx.profile_read()
    ctx.profile(False)
    launches = bfhe.launch_count() - launches0
    clk = clocks.stop()
    n_add, n_sub, n_mul, n_pmul = ctx.op_counts(reset=True)
    ms, total_mul = combine_ranks(dist, ms, n_mul, "cuda")
    value = total_mul / (ms / 1e3)

    # ---------------- e2e: the same job from host buffers (pinned), copies inside the timed region
    G_h = torch.from_numpy(Gs).pin_memory()
    W_h = torch.from_numpy(Ws).pin_memory()
    out_h = torch.empty((2, WL["N"]), dtype=torch.int64).pin_memory()
    torch.cuda.synchronize()
    ctx.op_counts(reset=True)
    t0 = time.perf_counter()
    g_d = G_h.to("cuda", non_blocking=True)
    w_d = W_h.to("cuda", non_blocking=True)
    r = job.run(g_d, w_d, seed=500)
    out_h.copy_(r, non_blocking=True)
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    e2e_mul = ctx.op_counts(reset=True)[2]
    e2e = {"value": e2e_mul / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(Gs.nbytes + Ws.nbytes),
           "d2h_bytes_per_step": int(out_h.numel() * 8)}

    # ---------------- roofline of the dominant kernel class
    peaks, src = measured_peaks()
    props = torch.cuda.get_device_properties(local)
    peak = alu_peak_modmul_per_s(props.multi_processor_count, peaks.get("sm_max_mhz", 2070.0))
    dom = max(prof, key=lambda k: prof[k][0])
    d_ms, d_launch, d_work, _ = prof[dom]
    achieved = d_work / (d_ms / 1e3)
    traffic = None
    if dom.startswith("ntt"):
        per_limb = ntt_traffic_per_limb("k_" + dom)
        if per_limb is not None:
            limbs_per_launch = d_work / max(1, d_launch) / (WL["N"] // 2 * (WL["N"].bit_length() - 1))
            traffic = per_limb * limbs_per_launch
    hbm = None
    if traffic is not None and peaks.get("hbm_gbs"):
        gbs = traffic / (d_ms / max(1, d_launch) / 1e3) / 1e9
        hbm = {"achieved_gbs": gbs, "peak_gbs": peaks["hbm_gbs"], "frac": gbs / peaks["hbm_gbs"]}
    roofline = {"bound": "alu", "kernel": dom, "achieved": achieved, "peak": peak, "unit": "modmul/s",
                "frac": achieved / peak, "traffic": traffic, "traffic_unit": "bytes per launch",
                "hbm_side": hbm,
                "frac_of_shoup_peak": achieved / (peak * 10 / 16),
                "peak_source": "derived: %d SMs x 64 IMAD/clk x %.0f MHz / 10 IMAD slots per product "
                               "modulo 2^b - d (clock from MEASURED_PEAKS.json, %s)"
                               % (props.multi_processor_count, peaks.get("sm_max_mhz", 2070.0), src),
                "avg_launch_ms": d_ms / max(1, d_launch), "launches": d_launch,
                "kernel_share": {k: round(v[0] / max(1e-9, sum(x[0] for x in prof.values())), 3)
                                 for k, v in prof.items()},
                "kernel_alu_frac": {k: round(v[2] / (v[0] / 1e3) / peak, 3) for k, v in prof.items() if v[0] > 0},
                "kernel_roofline": kernel_rooflines(prof, peak, peaks.get("hbm_gbs", 6800.0))}

    ext = {} if args.no_extras else extras(torch, bfhe, circuits, ctx)
    if ext.get("modmul_probe_per_s"):
        # the same rate against the library's own measured probe of Shoup products (all SMs), whose peak is 10/16 of it
        roofline["probe_modmul_per_s"] = ext["modmul_probe_per_s"]
        roofline["frac_of_probe"] = achieved / ext["modmul_probe_per_s"]
    # what the headline counts: mostly Fermat squarings and paper-mode ANDs of the bridge
    e = WL["t"] - 1
    chains = N_CLASSES * (1 << S_BITS)
    mix = {"squarings": chains * (e.bit_length() - 1), "odd_step_products": chains * (bin(e).count("1") - 1),
           "paper_mode_ands": chains * S_BITS, "argmax_circuit_products": job.circuit_muls,
           "general_batched_mul_relin_per_s_same_params": ext.get("mul_relin_batched_per_s")}
    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
                "config": {**base_config(), "mul_relin_per_step": n_mul // args.steps, "mul_relin_mix": mix,
                           "base_extension": "guarded fast, exact fallback" if ctx.fast_extension else "exact Garner",
                           "parallelism": "replicas" if world > 1 else "single",
                           "autotuned": {str(k): {"ntt_fwd": v["fwd"], "ntt_inv": v["inv"], "mul_tile": v["tile"]}
                                         for k, v in tuned.items()},
                           "l2": "no flush: per-step working set > 10 GB >> 129 MB L2"},
                "gpu_launches": int(launches), "clocks": clk, "e2e": e2e, "roofline": roofline,
                "cpu_baseline": cpu_line, "ops_per_step": {"add": n_add // args.steps, "sub": n_sub // args.steps,
                                                            "mul": n_mul // args.steps, "plain_mul": n_pmul // args.steps},
                "extras": ext}
        print(json.dumps(line), flush=True)
    ctx.close()
    if dist:
        dist.barrier()
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
