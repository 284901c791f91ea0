"""KeySwitch and HMUL with moduli at the top of the exact class (62 bits) and next to it ==
oracle: more sources than one exact basis-conversion sum holds (four at 62 bits, eight at 61,
sixteen at 60), sums that are folded on the way, and the largest residues as input, as key and
as the conversion's sources.
"""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch, host

pytestmark = pytest.mark.gpu


def params(dnum, logn, L, qbits, pbits):
    """L+1 + alpha distinct primes, the largest of their bits; limb i takes qbits[i % len]."""
    alpha = -(-(L + 1) // dnum)
    out = []
    for n, bits in ((L + 1, qbits), (alpha, pbits)):
        for i in range(n):
            out.append(next(x for x in W.primes_below(bits[i % len(bits)], logn, L + 2 + alpha)
                            if x not in out))
    return dataclasses.replace(W.make_params(dnum, logn, L), q=tuple(out[:L + 1]),
                               p=tuple(out[L + 1:]))


def inputs(prm, kind):
    g = W.rng(23, 13)
    evk = W.uniform_limbs(g, prm.mods * (2 * prm.beta), prm.N)
    d = W.uniform_limbs(g, prm.q, prm.N)
    if kind == "top":  # every word m - 1
        d[:] = np.array(prm.q, dtype=np.uint64)[:, None] - np.uint64(1)
        evk[:] = np.array(prm.mods * (2 * prm.beta), dtype=np.uint64)[:, None] - np.uint64(1)
    elif kind == "sources":  # every source of the ModUp conversion m - 1
        x = np.empty_like(d)
        for i, m in enumerate(prm.q):
            lo = i // prm.alpha * prm.alpha
            qhat = 1
            for k in range(lo, min(prm.L + 1, lo + prm.alpha)):
                if k != i:
                    qhat = qhat * prm.q[k] % m
            x[i] = m - qhat
        d = O.ntt_fwd(x, prm.q, prm.logn)
    return d, evk.reshape(prm.beta, 2, prm.QP, prm.N)


CASES = [((1, 12, 8), (62,), (62,)), ((1, 13, 9), (62,), (61, 62)), ((4, 12, 7), (62,), (62,)),
         ((2, 14, 19), (61,), (62,)), ((1, 14, 17), (60,), (62, 60)), ((1, 11, 8), (62,), (62,)),
         ((2, 15, 11), (62, 50), (60, 62)), ((1, 16, 5), (62,), (62,)), ((1, 13, 18), (50,), (61,)),
         ((1, 12, 17), (60, 50), (62,)), ((1, 17, 4), (62,), (62,))]


@pytest.mark.parametrize("kind", ["uniform", "top", "sources"])
@pytest.mark.parametrize("case", CASES, ids=str)
def test_switch(case, kind):
    cfg, qbits, pbits = case
    prm = params(*cfg, qbits, pbits)
    d, evk = inputs(prm, kind)
    want = O.keyswitch(prm, d, evk)
    ctx = ks.Context(prm)
    try:
        dd, de = dev(d), dev(evk)
        for v, c in ((ks.KS_AUTO, 0), (ks.KS_DSOB, 0), (ks.KS_DPOC, 3),
                     (ks.KS_DPOB | ks.KS_BCONV_TC, 0), (ks.KS_DPOB | ks.KS_UNFUSED, 0)):
            got = host(ctx.switch(dd, de, variant=v, chunks=c))
            assert np.array_equal(got, want), f"{ks.variant_name(v)}: " + first_mismatch(got, want)
    finally:
        ctx.close()


@pytest.mark.parametrize("bits", [50, 51, 52, 59, 60, 61, 62])
@pytest.mark.parametrize("kind", ["uniform", "top"])
def test_hmul(bits, kind):
    prm = params(2, 13, 3, (bits,), (60 if bits <= 60 else bits,))
    ct1, evk = inputs(prm, kind)
    g = W.rng(29, 13)
    cts = [np.stack([ct1, W.uniform_limbs(g, prm.q, prm.N) if kind == "uniform" else ct1])
           for _ in range(2)]
    want = O.hmul(prm, prm.L, cts[0], cts[1], evk)
    ctx = ks.Context(prm)
    try:
        got = host(ctx.hmul(dev(cts[0]), dev(cts[1]), dev(evk)))
        assert np.array_equal(got, want), first_mismatch(got, want)
    finally:
        ctx.close()
