"""The cluster kernels of N = 2^12 .. 2^14 == oracle, bit for bit, on both sides of their
dispatch rule (eight CTAs per target limb within the 152 SMs; digits within a CTA's shared
memory), with every epilogue that they share with the general kernels.

Cases: one digit (its Q-limb targets transform nothing), one limb per digit, ragged last
digits, the widest launch the rule takes (QP = 19) and the next one (QP = 20, general
kernels), more digits than thread groups, level views (the top level's key rows), HMUL and
HROT additions, host-buffer input, several jobs of one context in a batch, and moduli of
every butterfly class.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch, host, oracle_case

pytestmark = pytest.mark.gpu

CFGS = [(1, 12, 0), (1, 12, 8), (2, 12, 3), (2, 12, 4), (6, 12, 5), (9, 12, 16), (15, 12, 14),
        (4, 12, 15), (1, 13, 5), (2, 13, 7), (5, 13, 6), (8, 13, 15), (4, 13, 14), (4, 13, 15),
        (1, 14, 0), (3, 14, 7)]


@pytest.mark.parametrize("cfg", CFGS, ids=str)
def test_switch(cfg):
    prm, s_from, s_to, a, e, d, evk_o, out_o = oracle_case(cfg, 11)
    ctx = ks.Context(prm)
    try:
        evk = ctx.keygen(dev(s_from), dev(s_to), dev(a), dev(e))
        for v in (ks.KS_AUTO, ks.KS_DPOB):
            for _ in range(2):
                out = host(ctx.switch(dev(d), evk, variant=v))
                assert np.array_equal(out, out_o), first_mismatch(out, out_o)
    finally:
        ctx.close()


@pytest.mark.parametrize("cfg", [(3, 12, 7), (2, 13, 7)], ids=str)
def test_other_entry_points(cfg):
    import torch
    prm, s_from, s_to, a, e, d, evk_o, out_o = oracle_case(cfg, 12)
    ctx = ks.Context(prm)
    try:
        evk = ctx.keygen(dev(s_from), dev(s_to), dev(a), dev(e))
        # host buffers (pinned: read and written by the kernels), queued back to back
        dh = torch.from_numpy(d).pin_memory()
        outs = [torch.empty((2, *d.shape), dtype=dh.dtype).pin_memory() for _ in range(3)]
        for o in outs:
            ks.ks_switch_host_async(ctx.h, dh, evk, o)
        torch.cuda.synchronize()
        for o in outs:
            assert np.array_equal(o.numpy(), out_o)
        # two jobs of one context share every launch
        dd, ob = dev(d), [torch.empty((2, *d.shape), dtype=torch.uint64, device="cuda")
                          for _ in range(2)]
        ks.ks_switch_batch([(ctx.h, dd, evk, o) for o in ob])
        torch.cuda.synchronize()
        for o in ob:
            assert np.array_equal(host(o), out_o)
        # HROT and a level view
        k = ks.galois_elt(3, prm.N)
        rtk = ctx.keygen_galois(dev(s_to), k, dev(a), dev(e))
        ct = np.stack([d, W.gen_input(prm, 77)])
        got = host(ctx.hrot(dev(ct), k, rtk))
        want = O.hrot(prm, prm.L, ct, k, host(rtk))
        assert np.array_equal(got, want), first_mismatch(got, want)
        lvl = prm.L - 2
        view = ctx.at_level(lvl)
        got = host(view.switch(dev(d[:lvl + 1]), evk))
        want = O.keyswitch_level(prm, lvl, d[:lvl + 1], evk_o)
        assert np.array_equal(got, want), first_mismatch(got, want)
        rlk = ctx.keygen_relin(dev(s_to), dev(a), dev(e))
        got = host(ctx.hmul(dev(ct), dev(ct[::-1].copy()), rlk))
        want = O.hmul(prm, prm.L, ct, ct[::-1].copy(), host(rlk))
        assert np.array_equal(got, want), first_mismatch(got, want)
        view.close()
    finally:
        ctx.close()
