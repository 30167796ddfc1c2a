"""The standard greedy where newly covered sets are shared out over the grid in
pieces of 1,024 members: sets of every length (chains) and percolating ones."""
import pytest

import numpy as np
import oracle as O
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def chain(n):
    src = np.arange(n - 1, dtype=np.int64)
    in_off, in_src = inputs.in_csr(n, src, src + 1)
    return inputs.Graph(n, in_off, in_src, np.full(n - 1, 2**32 - 1, np.uint32))


@pytest.mark.parametrize("graph,theta,k", [
    (lambda: chain(4100), 700, 5), (lambda: chain(1025), 300, 3), (lambda: chain(2048), 33, 8),
    (lambda: inputs.rmat_graph(20_011, 400_000, 9, "ic0.2"), 64, 40),
    (lambda: inputs.rmat_graph(9000, 150_000, 2, "u0.1"), 900, 25)])
def test_greedy_long_sets(im, graph, theta, k):
    g = graph()
    G = im.Graph(g)
    P = im.Pool(G, theta, theta * g.n)
    P.sample(im.IM_IC, 5, 0, theta)
    ref = O.sample(O.IC, g, 5, 0, theta)
    assert np.diff(ref.set_off).max() > 1000
    c = P.cover(k)
    r = O.greedy(g.n, ref, O.invert(g.n, ref), k)
    assert c.seeds.tolist() == r.seeds.tolist()
    assert c.gains.tolist() == r.gains.tolist()
    assert c.coverage == r.coverage
    P.close()
    G.close()
