"""The arithmetic of the tensor-core basis conversion's eight-slot form, on the CPU.

The kernel (paper_2603_16692_gb300/csrc/ks_tc.cu) multiplies the bytes of the sources with
the bytes of c_i 2^(8a) mod m, so that S = sum_b v_b 2^(8b) is below 2^15 m, and reduces S
with one 32-bit Montgomery step. This emulates it from the fp32 bit patterns on, in wrapped
32/64-bit integers, for moduli of every size the library takes (up to just below 2^62),
up to the largest source count (16) and with all-ones bytes, against exact integers. The
bound: the result is S 2^-32 mod m, in (0, m + 2^-17 m].
"""
import numpy as np
import pytest

from paper_2603_16692_gb300 import workload as W

M32, M64 = (1 << 32) - 1, (1 << 64) - 1
E = 0x4B000000


def reduce_word(r, m):
    """tc_reduce on eight fp32 bit patterns, in wrapped machine words."""
    inv = pow(m, -1, 1 << 32)
    mc = (m - E * 65537) & M64
    p = [(r[2 * k] + ((r[2 * k + 1] << 8) & M32)) & M32 for k in range(4)]
    q0 = (p[0] + (p[1] << 16) - E * 65537) & M64
    q1 = (p[2] + (p[3] << 16) + mc) & M64
    u = (q0 * inv) & M32
    e = (((u * (m & M32)) >> 32) + u * (m >> 32)) & M64
    return (q1 + (q0 >> 32) - e) & M64


@pytest.mark.parametrize("bits", [20, 30, 45, 50, 51, 60, 61])
@pytest.mark.parametrize("ns", [1, 2, 9, 15, 16])
@pytest.mark.parametrize("kind", ["random", "max"])
def test_eight_slots(bits, ns, kind):
    rng = np.random.default_rng(bits * 100 + ns)
    m = W.primes_below(bits, 13, 1)[0]
    for _ in range(20):
        if kind == "max":
            xs, cs = [(1 << 64) - 1] * ns, [m - 1] * ns
        else:
            xs = [int(v) for v in rng.integers(0, 1 << 62, size=ns, dtype=np.uint64)]
            cs = [int(v) % m for v in rng.integers(0, 1 << 62, size=ns, dtype=np.uint64)]
        v = [0] * 8
        for x, c in zip(xs, cs):
            for a in range(8):
                ca = (c << (8 * a)) % m
                for b in range(8):
                    v[b] += ((x >> (8 * a)) & 255) * ((ca >> (8 * b)) & 255)
        assert max(v) < 1 << 23
        # the fp32 accumulators hold 2^23 + v exactly (any order: every partial sum is an
        # integer below 2^24)
        r = [int(np.float32(2 ** 23 + s).view(np.uint32)) for s in v]
        assert r == [E + s for s in v]
        S = sum(s << (8 * b) for b, s in enumerate(v))
        assert S < m << 15 and S % m == sum(x * c for x, c in zip(xs, cs)) % m
        z = reduce_word(r, m)
        assert z % m == S * pow(2, -32, m) % m
        assert 0 < z <= m + (m >> 17) + 1
