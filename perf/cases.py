"""The work that users of the library have it do, as timed and compared cases.

A case is one call (or one batch call) of the public interface
(`paper_2603_16692_gb300.ks`, the binding of include/ks.h) over the parameter range of the
repository's benchmark, batch and selector sweep: N = 2^12..2^17, L up to 60, dnum 1..10.
The operations are what a CKKS program calls: the KeySwitch itself, HMUL and HROT (which
contain one), at the top level or at a lower one with the top level's key, from device or
from pinned host buffers, alone or as an uneven batch.

Inputs are canonical residues, uniform mod each prime: that is the distribution of
ciphertexts and of evaluation keys (an RLWE key's words are uniform to the eye), so the
keys are drawn directly. The primes are those of the repository's workloads (50-bit
ciphertext primes, 60-bit special primes, all 1 mod 2N). Every output is a whole number
(a residue), so results are compared bit for bit.
"""
import math

import torch

from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W


def listed():
    """Sizes: the repository's three plain workloads (2, 2^13, 7), (2, 2^15, 10) and
    (4, 2^16, 35), the largest point of its sweep (10, 2^17, 60), and points with ragged
    digits inside the range of its batch. plan "auto" is what a program gets that names no
    plan; "tuned" is one that ran the autotuner once when it made its context."""
    return [
        # one pass per NTT, a handful of microseconds per kernel: launches and latency
        dict(name="switch_2^12", op="switch", dnum=2, logn=12, L=3, level=3, plan="auto"),
        # the smallest plain workload: every launch is a fraction of a wave
        dict(name="switch_2^13", op="switch", dnum=2, logn=13, L=7, level=7, plan="auto"),
        # the small plain workload, in a program that tuned its context at start-up
        dict(name="switch_2^15_tuned", op="switch", dnum=2, logn=15, L=10, level=10,
             plan="tuned"),
        # the benchmark's configuration, tuned: the steady state of a server
        dict(name="switch_2^16_tuned", op="switch", dnum=4, logn=16, L=35, level=35,
             plan="tuned"),
        # the largest sweep point (1.5 GB of key), no plan named
        dict(name="switch_2^17", op="switch", dnum=10, logn=17, L=60, level=60, plan="auto"),
        # ciphertext multiplication at the benchmark's configuration
        dict(name="hmul_2^16", op="hmul", dnum=4, logn=16, L=35, level=35, plan="auto"),
        # rotation at the small plain workload: the most frequent call of a
        # matrix-vector product
        dict(name="hrot_2^15", op="hrot", dnum=2, logn=15, L=10, level=10, plan="auto"),
        # multiplication late in a circuit: a level view, two digits (9 and 5 limbs)
        dict(name="hmul_2^16_level13", op="hmul", dnum=4, logn=16, L=35, level=13, plan="auto"),
        # many short digits with a ragged last one (31 limbs in sevens of 5 and one of 1)
        dict(name="switch_2^14_ragged", op="switch", dnum=7, logn=14, L=30, level=30,
             plan="auto"),
        # ciphertexts that live in pinned host memory (a client's or a pipeline's buffers)
        dict(name="host_2^15", op="host", dnum=2, logn=15, L=10, level=10, plan="auto"),
        # a caller that may not allocate: the static scratch, chunked to fit it
        dict(name="noalloc_2^16", op="noalloc", dnum=4, logn=16, L=35, level=35,
             plan="dsoc4"),
        # independent KeySwitches of uneven size issued together (a multi-tenant server)
        dict(name="batch_uneven", op="batch", plan="auto",
             jobs="6,13,44;2,13,11;9,14,52;3,14,27;4,15,19;10,15,33;2,15,8;5,16,24;2,16,47;"
                  "8,16,15"),
    ]


def _cost(case):
    w = work(case)
    return w["bytes"] / 6.8e12 + w["flops"] / 2e12


def draw(rng):
    """One more case of the same ranges: any operation, N = 2^12..2^17, L from 1 to 60
    (spread over its logarithm), dnum 1..10, any level, no plan named."""
    top = max(_cost(c) for c in listed())
    while True:
        op = rng.choice(["switch", "switch", "switch", "hmul", "hmul", "hrot", "hrot", "host",
                         "batch"])
        if op == "batch":
            jobs = []
            for _ in range(rng.randint(2, 8)):
                L = rng.randint(4, 60)
                jobs.append("%d,%d,%d" % (rng.randint(2, min(10, L + 1)), rng.randint(13, 16), L))
            case = dict(op=op, plan="auto", jobs=";".join(jobs))
        else:
            L = min(60, int(round(math.exp(rng.uniform(math.log(1), math.log(60.4))))))
            level = L if op == "host" or rng.random() < 0.6 else rng.randint(L // 3, L)
            case = dict(op=op, dnum=rng.randint(1, min(10, L + 1)), logn=rng.randint(12, 17), L=L,
                        level=level, plan="auto")
        if _cost(case) <= top:
            return case


# -- inputs -------------------------------------------------------------------------
def _limbs(g, mods, shape, n):
    """int64 [*shape, len(mods), n], uniform mod each prime."""
    out = torch.empty((*shape, len(mods), n), dtype=torch.int64, device="cuda")
    for t, m in enumerate(mods):
        out[..., t, :] = torch.randint(0, int(m), (*shape, n), generator=g, device="cuda",
                                       dtype=torch.int64)
    return out


def _one(case, g):
    """Context (at the case's level), input, key and output of one operation."""
    prm = W.make_params(case["dnum"], case["logn"], case["L"])
    top = ks.Context(prm)
    ctx = top if case["level"] == case["L"] else top.at_level(case["level"])
    q = prm.q[:case["level"] + 1]
    evk = _limbs(g, prm.mods, (prm.beta, 2), prm.N)
    return prm, top, ctx, q, evk


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    op = case["op"]
    if op == "batch":
        jobs, keep = [], []
        for j in case["jobs"].split(";"):
            dnum, logn, L = (int(x) for x in j.split(","))
            prm, top, ctx, q, evk = _one(dict(dnum=dnum, logn=logn, L=L, level=L), g)
            d = _limbs(g, q, (), prm.N)
            jobs.append((ctx.h, d, evk, torch.empty((2, *d.shape), dtype=d.dtype, device="cuda")))
            keep.append(ctx)
        return dict(op=op, jobs=jobs, keep=keep)
    prm, top, ctx, q, evk = _one(case, g)
    st = dict(op=op, ctx=ctx, keep=top, evk=evk, variant=ks.KS_AUTO, chunks=0)
    if op in ("hmul", "hrot"):
        st["ct"] = _limbs(g, q, (2,), prm.N)
        st["out"] = torch.empty_like(st["ct"])
        st["k"] = ks.galois_elt(1 + seed % 16, prm.N)
        if op == "hmul":
            st["ct2"] = _limbs(g, q, (2,), prm.N)
        kind = ks.KS_OP_HMUL if op == "hmul" else ks.KS_OP_HROT
        ws = ks.ks_eval_workspace_size(ctx.h, kind)
    else:
        d = _limbs(g, q, (), prm.N)
        out = torch.empty((2, *d.shape), dtype=d.dtype, device="cuda")
        if op == "host":
            d, out = d.cpu().pin_memory(), torch.empty(out.shape, dtype=d.dtype, pin_memory=True)
        st["d"], st["out"] = d, out
        if case["plan"] == "dsoc4":
            st["variant"], st["chunks"] = ks.KS_DSOC, 4
        elif case["plan"] == "tuned":
            st["variant"], st["chunks"] = ks.ks_tune(ctx.h, d, evk, out)
        ws = ks.ks_workspace_size(ctx.h, st["variant"], st["chunks"]) if op == "switch" else 0
    # the scratch that a program keeps beside its context
    st["ws"] = torch.empty(ws // 8, dtype=torch.int64, device="cuda") if ws else None
    return st


# -- the call -----------------------------------------------------------------------
def run(st):
    op = st["op"]
    if op == "batch":
        ks.ks_switch_batch(st["jobs"])
        return [jb[3] for jb in st["jobs"]]
    if op == "switch":
        st["ctx"].switch(st["d"], st["evk"], st["out"], st["variant"], st["chunks"], st["ws"])
    elif op == "hmul":
        st["ctx"].hmul(st["ct"], st["ct2"], st["evk"], st["out"], workspace=st["ws"])
    elif op == "hrot":
        st["ctx"].hrot(st["ct"], st["k"], st["evk"], st["out"], workspace=st["ws"])
    elif op == "host":
        ks.ks_switch_host_async(st["ctx"].h, st["d"], st["evk"], st["out"])
    else:
        ks.ks_switch_noalloc(st["ctx"].h, st["d"], st["evk"], st["out"], st["variant"],
                             st["chunks"])
    return st["out"]


def exact(case, seed):
    """Every output is a residue, a whole number that has to be equal bit for bit; there is
    no rounding whose error could be told in 64 bits."""
    return None


# -- what a pass cannot do without --------------------------------------------------------
def work(case):
    """bytes: each input word (ciphertext limbs and the key rows that the level uses) read
    once and each output word written once. flops: two for each modular multiply-add (NTT
    butterflies, basis-conversion and key-multiply terms, scalings) on 64-bit words."""
    if case["op"] == "batch":
        tot = dict(bytes=0.0, flops=0.0)
        for j in case["jobs"].split(";"):
            dnum, logn, L = (int(x) for x in j.split(","))
            w = work(dict(op="switch", dnum=dnum, logn=logn, L=L, level=L))
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    N, nq = 1 << case["logn"], case["level"] + 1
    alpha = -(-(case["L"] + 1) // case["dnum"])
    beta = -(-nq // alpha)
    qp = nq + alpha
    conv = beta * qp - nq  # (digit, target) pairs of ModUp
    terms = sum(min(alpha, nq - j * alpha) * (qp - min(alpha, nq - j * alpha))
                for j in range(beta))
    butterflies = (nq + conv + 2 * alpha + 2 * nq) * N / 2 * case["logn"]
    macs = (terms + 2 * beta * qp + 2 * alpha * nq + nq + 2 * alpha + 2 * nq) * N
    limbs_io = {"switch": 3, "host": 3, "noalloc": 3, "hmul": 6, "hrot": 4}[case["op"]] * nq
    if case["op"] == "hmul":
        macs += 4 * nq * N
    return dict(bytes=8.0 * N * (limbs_io + 2 * beta * qp), flops=2.0 * (butterflies + macs))
