"""The one-walk-per-thread LT sampler where its buffers, filter and checks are at
their limits: walks around the lane buffer's 1,024 entries, cycles (every walk
ends by a revisit, through a saturated filter), roots without in-edges, graphs
of a few vertices, and unequal weights whose draws pass their cut point."""
import numpy as np
import pytest

import oracle as O
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu
MAX = 2**32 - 1


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def line(n, closed, w=MAX):
    src = np.arange(n if closed else n - 1, dtype=np.int64)
    in_off, in_src = inputs.in_csr(n, src, (src + 1) % n)
    return inputs.Graph(n, in_off, in_src, np.full(in_src.shape[0], w, np.uint32))


def check(im, g, seed, theta, first=0):
    G = im.Graph(g)
    P = im.Pool(G, theta, theta * min(g.n, 4096) + 8)
    P.sample(im.IM_LT, seed, first, theta)
    set_off, members = P.export()
    ref = O.sample(O.LT, g, seed, first, theta)
    assert np.array_equal(set_off, ref.set_off)
    assert np.array_equal(members, ref.members)
    assert P.info()[2] == ref.examined
    P.close()
    G.close()


# every walk of a closed line visits all n vertices and then its root again
@pytest.mark.parametrize("n", [2, 3, 31, 500, 509, 1019, 1020, 1021, 1022, 1023, 1024, 1025, 1500])
@pytest.mark.parametrize("closed", [True, False])
def test_lines(im, n, closed):
    check(im, line(n, closed), 3, 700)


# walks of geometric length on a long cycle: many ends by no pick, few revisits
@pytest.mark.parametrize("p", [0.9, 0.99, 0.999])
def test_broken_cycle(im, p):
    check(im, line(3001, True, int(p * 2**32)), 8, 5000, first=77)


def test_one_vertex_and_none_with_in_edges(im):
    check(im, inputs.Graph(1, np.zeros(2, np.int64), np.zeros(0, np.int32), np.zeros(0, np.uint32)), 1, 65)
    check(im, inputs.Graph(40, np.zeros(41, np.int64), np.zeros(0, np.int32), np.zeros(0, np.uint32)), 1, 1000)


# heavily unequal weights: most of a vertex's draws fall on a few edges, some
# behind thousands of others
@pytest.mark.parametrize("seed", [1, 2])
def test_unequal_weights_past_the_cut_point(im, seed):
    rng = np.random.default_rng(seed)
    n, d = 300, 299
    src = np.concatenate([np.delete(np.arange(n), v) for v in range(n)]).astype(np.int64)
    in_off, in_src = inputs.in_csr(n, src, np.repeat(np.arange(n), d))
    w = rng.pareto(0.6, size=(n, d)) + 1e-9
    w = np.floor(w / w.sum(1, keepdims=True) * MAX * rng.uniform(0.5, 1.0, (n, 1))).astype(np.uint32)
    check(im, inputs.Graph(n, in_off, in_src, w.reshape(-1)), 5, 4000)
