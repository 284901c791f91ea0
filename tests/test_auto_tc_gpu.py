"""KS_AUTO's choice of the tensor-core basis conversions: on where the work of a conversion
launch reaches the line that ks.h states, the oracle's result on both sides of it, and the
integer plan where the scratch at hand holds only that.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, first_mismatch, host

pytestmark = pytest.mark.gpu


def operands(prm, seed):
    g = W.rng(seed, 13)
    d = W.uniform_limbs(g, prm.q, prm.N)
    evk = W.uniform_limbs(g, prm.mods * (2 * prm.beta), prm.N).reshape(
        prm.beta, 2, prm.QP, prm.N)
    return d, evk


def rule(prm):
    return (prm.beta * prm.QP + prm.L + 1) * prm.alpha * prm.N >= 2 * 7 << 20


# (2, 13, 7), (3, 14, 18): below the line; (3, 14, 26): one past it on 9 sources; (7, 14, 30),
# (10, 13, 60): above on few points; (2, 15, 10), (4, 15, 19): both sides at 2^15; (2, 14, 19):
# above, but 10 sources have no tensor-core form
@pytest.mark.parametrize("cfg", [(2, 13, 7), (3, 14, 18), (3, 14, 26), (7, 14, 30), (10, 13, 60),
                                 (2, 15, 10), (4, 15, 19), (2, 14, 19)], ids=str)
def test_rule(cfg):
    import torch
    prm = W.make_params(*cfg)
    d, evk = operands(prm, 21)
    want = O.keyswitch(prm, d, evk)
    ctx = ks.Context(prm)
    try:
        tc = rule(prm) and bool(ks.ks_context_info(ctx.h)["tc"])
        size = {v: ks.ks_workspace_size(ctx.h, v) for v in
                (ks.KS_AUTO, ks.KS_DPOB, ks.KS_DPOB | ks.KS_BCONV_TC)}
        assert size[ks.KS_AUTO] == size[ks.KS_DPOB | (ks.KS_BCONV_TC if tc else 0)]
        dd, de = dev(d), dev(evk)
        # scratch for the plan, and for the integer plan alone
        for n in (size[ks.KS_AUTO], size[ks.KS_DPOB]):
            ws = torch.empty(n // 8, dtype=torch.uint64, device="cuda")
            got = host(ctx.switch(dd, de, workspace=ws))
            assert np.array_equal(got, want), first_mismatch(got, want)
        with pytest.raises(ks.KSError):
            ctx.switch(dd, de, workspace=ws[:-1])
    finally:
        ctx.close()


def test_static_scratch():
    """(5, 2^15, 40): the integer plan fits the static scratch, the tensor-core one does not."""
    import torch
    prm = W.make_params(5, 15, 40)
    d, evk = operands(prm, 22)
    ctx = ks.Context(prm)
    try:
        room = ks.ks_noalloc_scratch_bytes()
        assert ks.ks_workspace_size(ctx.h, ks.KS_DPOB) <= room < \
            ks.ks_workspace_size(ctx.h, ks.KS_AUTO)
        out = torch.empty((2, prm.L + 1, prm.N), dtype=torch.uint64, device="cuda")
        ks.ks_switch_noalloc(ctx.h, dev(d), dev(evk), out)
        got, want = host(out), O.keyswitch(prm, d, evk)
        assert np.array_equal(got, want), first_mismatch(got, want)
    finally:
        ctx.close()
