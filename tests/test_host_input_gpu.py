"""Host-buffer KeySwitches on both sides of the line where the input pass paces its reads
(2^18 words), through the cluster inverse (2^13, 2^14) and the general row pass: == oracle, queued
back to back so that one call's reads overlap the previous one's writes.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch

pytestmark = pytest.mark.gpu


# limbs x N: (2, 13, 31), (2, 14, 15), (2, 15, 7), (1, 17, 1) are 2^18 words, the others past it
@pytest.mark.parametrize("cfg", [(2, 13, 31), (2, 13, 32), (2, 14, 15), (2, 14, 16), (2, 15, 7),
                                 (2, 15, 8), (1, 17, 1), (1, 17, 2)], ids=str)
def test_host_input(cfg):
    import torch
    prm = W.make_params(*cfg)
    g = W.rng(31, 13)
    ds = [W.uniform_limbs(g, prm.q, prm.N) for _ in range(2)]
    evk = W.uniform_limbs(g, prm.mods * (2 * prm.beta), prm.N).reshape(
        prm.beta, 2, prm.QP, prm.N)
    wants = [O.keyswitch(prm, d, evk) for d in ds]
    ctx = ks.Context(prm)
    try:
        de, dh = dev(evk), [torch.from_numpy(d).pin_memory() for d in ds]
        outs = [torch.empty((2, *ds[0].shape), dtype=dh[0].dtype).pin_memory() for _ in range(4)]
        for k, o in enumerate(outs):
            ks.ks_switch_host_async(ctx.h, dh[k % 2], de, o)
        torch.cuda.synchronize()
        for k, o in enumerate(outs):
            assert np.array_equal(o.numpy(), wants[k % 2]), first_mismatch(o.numpy(), wants[k % 2])
    finally:
        ctx.close()
