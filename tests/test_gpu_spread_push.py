"""LT spread on graphs where a run's out-edges are few against its vertices: such runs are
pushed to their end, at the rate of an IC spread over the same edges; and runs that stop, are
pulled, or are gone on with equal the oracle."""
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


def kernel_ms(im, G, model, seeds, runs):
    best = 1e9
    for _ in range(4):                                  # (the first makes the indexes)
        im.im_profile_enable(True)
        im.im_profile_reset()
        im.im_spread(G.handle, model, seeds, 6, 0, runs)
        ms = im.im_profile_read()
        im.im_profile_enable(False)
        best = min(best, sum(t for name, (_, t) in ms.items() if name.startswith("spread")))
    return best


def star(n, k, leaves):
    """k seeds with leaves of their own, each reached with probability 1/2 under either model."""
    src, dst = np.repeat(np.arange(k), leaves), np.arange(k * leaves) + k
    in_off, in_src = inputs.in_csr(n, src.astype(np.int64), dst.astype(np.int64))
    return inputs.Graph(n, in_off, in_src, np.full(k * leaves, 1 << 31, np.uint32)), np.arange(k, dtype=np.int32)


def test_few_out_edges_cost_what_ic_costs(im):
    """1,000 seeds with 200 leaves each in a graph of 2^20 vertices: the same out-edges under
    IC and LT, and as many vertices activated.  (A draw for every vertex of the graph
    takes more than twice as long.)"""
    g, seeds = star(1 << 20, 1000, 200)
    G = im.Graph(g)
    ic, lt = kernel_ms(im, G, im.IM_IC, seeds, 3000), kernel_ms(im, G, im.IM_LT, seeds, 3000)
    G.close()
    assert lt < 1.5 * ic


def top(g, k):
    return np.argsort(-np.bincount(g.in_src, minlength=g.n), kind="stable")[:k].astype(np.int32)


# runs of which all stop; first those of which a sample says that they are pushed to their
# end, then those that are pulled; more of them than one round of groups takes, and more
# than the lot of stopped runs holds
@pytest.mark.parametrize("runs", [400, 4200])
@pytest.mark.parametrize("pushed", [True, False])
def test_many_stopped_runs(im, pushed, runs):
    g, seeds = star(1 << 18, 1000, 100) if pushed else (inputs.rmat_graph(1 << 17, 1 << 21, 4, "lt"), None)
    seeds = top(g, 100) if seeds is None else seeds
    G = im.Graph(g)
    act, hit = np.zeros(runs, np.int64), np.zeros(runs, np.uint8)
    assert im.im_spread(G.handle, im.IM_LT, seeds, 6, 5, runs, act, hit) == int(act.sum())
    for at in [0, runs // 2, runs - 12]:
        ref = O.spread(O.LT, g, 6, 5 + at, 12, seeds)
        assert np.array_equal(act[at:at + 12], ref[0]) and np.array_equal(hit[at:at + 12], ref[1])
    few = np.zeros(1, np.int64)                          # (a call of one run stops it alone)
    for at in range(0, runs, 37):
        im.im_spread(G.handle, im.IM_LT, seeds, 6, 5 + at, 1, few)
        assert act[at] == few[0]
    G.close()


@pytest.mark.parametrize("n,m,k,runs", [(1 << 13, 1 << 17, 100, 300), (9000, 40_000, 300, 100), (20_000, 36_000, 2000, 40)])
@pytest.mark.parametrize("weights", ["lt", "lt-u0.1"])
def test_equals_the_oracle(im, n, m, k, runs, weights):
    g = inputs.rmat_graph(n, m, 4, weights)
    seeds = top(g, k)
    G = im.Graph(g)
    act, hit = np.zeros(runs, np.int64), np.zeros(runs, np.uint8)
    total = im.im_spread(G.handle, im.IM_LT, seeds, 6, 3, runs, act, hit)
    ref = O.spread(O.LT, g, 6, 3, runs, seeds)
    G.close()
    assert np.array_equal(act, ref[0]) and np.array_equal(hit, ref[1]) and total == int(ref[0].sum())
