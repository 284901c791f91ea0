"""KeySwitch with moduli of every butterfly class (below 2^51, 2^60 and 2^62) == oracle.

The primes of the other tests are 50-bit (Q) and 60-bit (P). Here the classes are mixed
between and within Q and P, at the edges of each class, so that every class runs as a
ciphertext limb, as a special limb, and next to another class in one pair of tensor-core
targets. Bit-exact: integer work.
"""
import dataclasses

import numpy as np
import pytest

from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch, host
from oracle import oracle as O

pytestmark = pytest.mark.gpu


def params(dnum, logn, L, qbits, pbits):
    """L+1 + alpha distinct primes; limb i takes qbits[i % len] (pbits alike)."""
    alpha = -(-(L + 1) // dnum)
    used, out = set(), []
    for n, bits in ((L + 1, qbits), (alpha, pbits)):
        for i in range(n):
            b = bits[i % len(bits)]
            m = next(x for x in W.primes_below(b, logn, 3 * (L + 1 + alpha)) if x not in used)
            used.add(m)
            out.append(m)
    return dataclasses.replace(W.make_params(dnum, logn, L), q=tuple(out[:L + 1]),
                               p=tuple(out[L + 1:]))


CASES = [(dnum, logn, L, q, p)
         for dnum, logn, L in [(2, 11, 4), (3, 12, 5), (2, 13, 5), (3, 14, 7), (2, 15, 4),
                               (2, 16, 5), (3, 17, 5)]
         for q, p in [((50,), (61,)), ((51,), (60,)), ((52, 50, 40), (60, 50)),
                      ((60,), (60,)), ((61, 50, 59), (61, 55)), ((30, 45), (51,))]]


@pytest.mark.parametrize("case", CASES, ids=str)
def test_modulus_classes(case):
    prm = params(*case)
    s_from, s_to, a, e = W.gen_keys(prm, 5)
    d = W.gen_input(prm, 5)
    evk_o = O.keygen(prm, s_from, s_to, a, e)
    out_o = O.keyswitch(prm, d, evk_o)
    ctx = ks.Context(prm)
    try:
        evk = ctx.keygen(dev(s_from), dev(s_to), dev(a), dev(e))
        assert np.array_equal(host(evk), evk_o), first_mismatch(host(evk), evk_o)
        for v in (ks.KS_AUTO, ks.KS_DPOB | ks.KS_RADIX4, ks.KS_DPOB | ks.KS_BCONV_TC,
                  ks.KS_DSOB, ks.KS_DPOB | ks.KS_UNFUSED):
            out = host(ctx.switch(dev(d), evk, variant=v))
            assert np.array_equal(out, out_o), f"{ks.variant_name(v)}: " + first_mismatch(
                out, out_o)
    finally:
        ctx.close()
