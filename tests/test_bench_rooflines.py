"""bench.py's bytes of the covering-subset build: digits of at most 10 bits, so one pass up to 1,024
vertices, two up to 2^20 and three beyond; no keys are written by the last (CPU)."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("n,per_member", [(1, 12), (1024, 12), (1025, 32), (1 << 20, 32), ((1 << 20) + 1, 52)])
def test_bytes_of_the_radix_build(n, per_member):
    sys.path.insert(0, ROOT)
    import bench
    T, theta = 10**8, 10**6
    cs = {"T": T, "n": n, "theta": theta, "k": 1, "s_seed": 0, "covered": 0, "r_covered": 0, "rg_eval": 0, "rg_cover": 0}
    out = bench.kernel_rooflines(None, cs, {"index_radix": (2, 2.0)}, 1000.0)
    assert out["index_radix"]["alg_bytes"] == per_member * T + 8 * theta
    assert out["index_radix"]["gbs"] == round((per_member * T + 8 * theta) / 2e-3 / 1e9, 1)
