"""LT spread of runs that activate enough of the graph to be finished by pulling:
the same activated counts and root hits as the oracle, run by run."""
import numpy as np
import pytest

import oracle as O
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def check(im, g, seeds, seed, first, runs):
    G = im.Graph(g)
    act = np.zeros(runs, np.int64)
    hit = np.zeros(runs, np.uint8)
    total = im.im_spread(G.handle, im.IM_LT, seeds, seed, first, runs, act, hit)
    ref = O.spread(O.LT, g, seed, first, runs, np.asarray(seeds, np.int32))
    assert np.array_equal(act, ref[0])
    assert np.array_equal(hit, ref[1])
    assert total == int(ref[0].sum())
    G.close()


# 2^15 to 2^17 vertices of 16 out-edges: the largest vertices activate far more
# than 65,536 out-edges in some runs and not in others
@pytest.mark.parametrize("n,m,k,runs", [(1 << 15, 1 << 19, 300, 7), (100_003, 1_600_000, 50, 33), (1 << 17, 1 << 21, 1, 40)])
@pytest.mark.parametrize("weights", ["lt", "lt-u0.1"])
def test_rmat(im, n, m, k, runs, weights):
    g = inputs.rmat_graph(n, m, 4, weights)
    top = np.argsort(-np.bincount(g.in_src, minlength=g.n), kind="stable")[:k].astype(np.int32)
    check(im, g, np.concatenate([top, top[:1]]), 6, 3, runs)


# a closed line behind a hub of 70,000 out-edges: chains of 20,000 pointers, some
# of which end at the seed and some of which run round the cycle
@pytest.mark.parametrize("cut", [True, False])
def test_long_chains(im, cut):
    c, h = 20_000, 70_000
    n = c + h
    src = [np.arange(c), np.zeros(h)]                  # i -> i + 1 on the line; 0 -> every leaf
    dst = [(np.arange(c) + 1) % c, np.arange(c, n)]
    w = 2**32 - 1
    in_off, in_src = inputs.in_csr(n, np.concatenate(src).astype(np.int64), np.concatenate(dst).astype(np.int64))
    wts = np.full(n, w, np.uint32)
    if cut:
        wts[1:c] = int(0.9999 * 2**32)                 # a line that breaks here and there
    check(im, inputs.Graph(n, in_off, in_src, wts), [0], 2, 0, 9)
    check(im, inputs.Graph(n, in_off, in_src, wts), [c // 2, n - 1], 2, 9, 9)
