"""Host-buffer KeySwitches whose input is the result of the call queued before them on the
stream, without a synchronization in between: every link of the chain == oracle. The first
kernel of such a call may read its input while the call before runs, unless that call writes
it. Cluster sizes, general kernels of one and of several waves, tensor-core conversions, the
graph-replayed single-pass sizes; results of ks_switch and HROT in pinned memory; a chain
under stream capture.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch

pytestmark = pytest.mark.gpu

LINKS = 5


def chain(cfg):
    """Input, key and the LINKS results, each link taking the second half of the one before."""
    prm = W.make_params(*cfg)
    g = W.rng(17, 13)
    d = W.uniform_limbs(g, prm.q, prm.N)
    evk = W.uniform_limbs(g, prm.mods * (2 * prm.beta), prm.N).reshape(
        prm.beta, 2, prm.QP, prm.N)
    wants = []
    for _ in range(LINKS):
        wants.append(O.keyswitch(prm, wants[-1][1] if wants else d, evk))
    return prm, d, evk, wants


def pinned(shape):
    import torch
    return torch.zeros(shape, dtype=torch.uint64).pin_memory()


def same(outs, wants):
    for k, (o, w) in enumerate(zip(outs, wants)):
        assert np.array_equal(o.numpy(), w), f"link {k}: " + first_mismatch(o.numpy(), w)


@pytest.mark.parametrize("cfg", [(2, 9, 3), (2, 12, 3), (2, 13, 7), (3, 14, 12), (2, 15, 10),
                                 (4, 16, 11), (1, 17, 2)], ids=str)
def test_chained_calls(cfg):
    import torch
    prm, d, evk, wants = chain(cfg)
    shape = (2, prm.L + 1, prm.N)
    ctx = ks.Context(prm)
    try:
        de, dh = dev(evk), torch.from_numpy(d).pin_memory()
        for sync in (False, True):
            outs = [pinned(shape) for _ in range(LINKS)]
            for k, o in enumerate(outs):
                f = ks.ks_switch_host if sync and k == LINKS - 1 else ks.ks_switch_host_async
                f(ctx.h, outs[k - 1][1] if k else dh, de, o)
            torch.cuda.synchronize()
            same(outs, wants)
        # after a call whose result is elsewhere, the chain goes on from an older one
        outs, other = [pinned(shape) for _ in range(2)], pinned(shape)
        ks.ks_switch_host_async(ctx.h, dh, de, outs[0])
        ks.ks_switch_host_async(ctx.h, dh, de, other)
        ks.ks_switch_host_async(ctx.h, outs[0][1], de, outs[1])
        torch.cuda.synchronize()
        same(outs + [other], [wants[0], wants[1], wants[0]])
    finally:
        ctx.close()


@pytest.mark.parametrize("cfg", [(2, 13, 7), (4, 16, 11)], ids=str)
def test_after_other_calls(cfg):
    """ks_switch (caller's scratch, then the context's), a batch and HROT write the input."""
    import torch
    prm, d, evk, wants = chain(cfg)
    shape = (2, prm.L + 1, prm.N)
    ctx = ks.Context(prm)
    try:
        dd, de, dh = dev(d), dev(evk), torch.from_numpy(d).pin_memory()
        ws = torch.empty(ks.ks_workspace_size(ctx.h, ks.KS_AUTO) // 8, dtype=torch.uint64, device="cuda")
        for first in (lambda o: ks.ks_switch(ctx.h, dd, de, o, workspace=ws),
                      lambda o: ks.ks_switch(ctx.h, dd, de, o),
                      lambda o: ks.ks_switch_batch([(ctx.h, dd, de, o)])):
            outs, other = [pinned(shape) for _ in range(2)], pinned(shape)
            ks.ks_switch_host_async(ctx.h, dh, de, other)
            first(outs[0])
            ks.ks_switch_host_async(ctx.h, outs[0][1], de, outs[1])
            torch.cuda.synchronize()
            same(outs, wants)
        ct = np.stack([d, d])
        rot, out = pinned(shape), pinned(shape)
        ctx.hrot(dev(ct), 5, de, rot)
        ks.ks_switch_host_async(ctx.h, rot[0], de, out)
        torch.cuda.synchronize()
        want = O.keyswitch(prm, rot[0].numpy(), evk)
        assert np.array_equal(out.numpy(), want), first_mismatch(out.numpy(), want)
    finally:
        ctx.close()


def test_chain_under_capture():
    import torch
    prm, d, evk, wants = chain((2, 15, 10))
    ctx = ks.Context(prm)
    try:
        de, dh = dev(evk), torch.from_numpy(d).pin_memory()
        outs = [pinned((2, prm.L + 1, prm.N)) for _ in range(LINKS)]

        def links():
            for k, o in enumerate(outs):
                ks.ks_switch_host_async(ctx.h, outs[k - 1][1] if k else dh, de, o)
        links()  # the context's scratch is in place
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            links()
        for o in outs:
            o.zero_()
        g.replay()
        torch.cuda.synchronize()
        same(outs, wants)
    finally:
        ctx.close()
