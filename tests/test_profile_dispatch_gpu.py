"""The per-kernel profile times the kernels that the call launches: the cluster kernels where
they serve the plan, the general ones elsewhere.
"""
import pytest

from oracle import oracle as O
from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W
from tests.gpu_util import dev, host

pytestmark = pytest.mark.gpu

FUSED = {"fused_intt(d)": 1, "fused_modup_keymult": 1, "fused_intt(accP)": 1, "fused_moddown": 1}
MIXED = {"fused_intt(d)": 1, "modup_col": 1, "modup_row_keymult": 1, "fused_intt(accP)": 1,
         "moddown_col": 1, "moddown_row": 1}


# (2, 2^12, 3), (2, 2^13, 7): cluster kernels throughout; (4, 2^13, 15), (3, 2^14, 8): the
# inverse transforms only; with chunks and with the tensor-core conversions
@pytest.mark.parametrize("cfg,variant,chunks,want", [
    ((2, 12, 3), ks.KS_DPOB, 0, FUSED),
    ((2, 13, 7), ks.KS_DPOB, 0, FUSED),
    ((4, 13, 15), ks.KS_DPOB, 0, MIXED),
    ((3, 14, 8), ks.KS_DPOB, 0, MIXED),
    ((2, 13, 7), ks.KS_DPOC, 2,
     {k: n * (1 if k.startswith("fused") else 2) for k, n in MIXED.items()}),
    ((2, 13, 7), ks.KS_DPOB | ks.KS_BCONV_TC, 0,
     {"intt_row(d)": 1, "intt_col(d)": 1, "modup_col": 1, "modup_row_keymult": 1,
      "intt_row(accP)": 1, "intt_col(accP)": 1, "moddown_col": 1, "moddown_row": 1}),
], ids=str)
def test_profiled_launches(cfg, variant, chunks, want):
    import torch
    prm = W.make_params(*cfg)
    g = W.rng(3, 13)
    d = W.uniform_limbs(g, prm.q, prm.N)
    evk = W.uniform_limbs(g, prm.mods * (2 * prm.beta), prm.N).reshape(
        prm.beta, 2, prm.QP, prm.N)
    ctx = ks.Context(prm)
    try:
        dd, de = dev(d), dev(evk)
        out = ctx.switch(dd, de, variant=variant, chunks=chunks)
        torch.cuda.synchronize()
        ks.ks_profile_begin()
        got = ctx.switch(dd, de, variant=variant, chunks=chunks)
        stats = ks.ks_profile_end()
    finally:
        ctx.close()
    assert (host(got) == host(out)).all() and (host(out) == O.keyswitch(prm, d, evk)).all()
    assert {s["name"]: s["launches"] for s in stats} == want
    # each stage's terms and the traffic are counted whichever kernels run it
    macs = sum(s["macs"] for s in stats)
    ds = [min(prm.L + 1, (j + 1) * prm.alpha) - j * prm.alpha for j in range(prm.beta)]
    if not variant & ks.KS_BCONV_TC:
        assert macs == prm.N * (sum((prm.QP - n) * (n + 1) for n in ds) +
                                2 * prm.beta * prm.QP + prm.L + 1 +
                                2 * (prm.L + 1) * (prm.alpha + 1))
    assert all(s["bytes"] > 0 and s["ops"] >= s["macs"] and s["ms"] > 0 for s in stats)
