"""KS_AUTO with the device's memory taken: the context's arena (and the batch's) that holds the
plan only without the tensor-core conversions that the rule adds is kept and used, call after
call and under stream capture, instead of being given up for an allocation that fails.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch, host

pytestmark = pytest.mark.gpu


def test_arena_is_kept():
    import torch
    prm = W.make_params(4, 16, 35)
    g = W.rng(19, 13)
    d = W.uniform_limbs(g, prm.q, prm.N)
    evk = W.uniform_limbs(g, prm.mods * (2 * prm.beta), prm.N).reshape(
        prm.beta, 2, prm.QP, prm.N)
    want = O.keyswitch(prm, d, evk)
    ctx = ks.Context(prm)
    hog = None
    try:
        dd, de = dev(d), dev(evk)
        out = torch.empty((2, prm.L + 1, prm.N), dtype=torch.uint64, device="cuda")
        calls = [lambda: ks.ks_switch(ctx.h, dd, de, out),
                 lambda: ks.ks_switch_batch([(ctx.h, dd, de, out)])]
        # the arenas at the integer plan's size; every kernel loaded, a first graph made
        ks.ks_switch(ctx.h, dd, de, out, ks.KS_DPOB)
        ks.ks_switch_batch([(ctx.h, dd, de, out, ks.KS_DPOB, 0)])
        grow = ks.ks_workspace_size(ctx.h, ks.KS_AUTO) - ks.ks_workspace_size(ctx.h, ks.KS_DPOB)
        ws = torch.empty(ks.ks_workspace_size(ctx.h, ks.KS_AUTO) // 8, dtype=torch.uint64,
                         device="cuda")
        ks.ks_switch(ctx.h, dd, de, out, workspace=ws)
        gr = torch.cuda.CUDAGraph()
        with torch.cuda.graph(gr):
            ks.ks_switch(ctx.h, dd, de, out, workspace=ws)
        gr.replay()
        out.zero_()
        torch.cuda.synchronize()
        del ws, gr
        torch.cuda.empty_cache()
        # all but what a graph takes, which is less than the arena would grow by
        hog = torch.empty(torch.cuda.mem_get_info()[0] - (36 << 20), dtype=torch.uint8,
                          device="cuda")
        assert torch.cuda.mem_get_info()[0] < grow
        for call in calls:
            for captured in (False, True):
                out.zero_()
                if captured:
                    gr = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(gr):
                        call()
                    gr.replay()
                else:
                    call()
                torch.cuda.synchronize()
                assert np.array_equal(host(out), want), first_mismatch(host(out), want)
    finally:
        del hog
        torch.cuda.empty_cache()
        ctx.close()
