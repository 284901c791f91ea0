"""KS_AUTO's choice of the tensor-core conversions counts the limbs that a level's last digit
has: at levels where that digit is short, the integer conversions are the faster ones.
"""
import pytest

from paper_2603_16692_gb300 import ks
from paper_2603_16692_gb300 import workload as W

pytestmark = pytest.mark.gpu


# ((dnum, log N, L), level, tensor cores): a short last digit and a short only digit, full
# digits, both sides of the line
@pytest.mark.parametrize("cfg,level,tc", [
    ((4, 14, 35), 19, False), ((4, 16, 21), 8, False), ((4, 16, 35), 7, False),
    ((4, 17, 12), 6, False), ((7, 14, 36), 24, True), ((4, 16, 35), 11, True),
    ((7, 14, 30), 30, True), ((4, 15, 19), 19, True), ((2, 15, 10), 10, False)], ids=str)
def test_rule_at_level(cfg, level, tc):
    prm = W.make_params(*cfg)
    top = ks.Context(prm)
    ctx = top if level == prm.L else top.at_level(level)
    try:
        words = (level + 1) * (level + 1 + 2 * prm.alpha) * prm.N
        assert (words >= 2 * 7 << 20) == tc
        want = ks.KS_DPOB | (ks.KS_BCONV_TC if tc else 0)
        assert ks.ks_workspace_size(ctx.h, ks.KS_AUTO) == ks.ks_workspace_size(ctx.h, want)
    finally:
        if ctx is not top:
            ctx.close()
        top.close()
