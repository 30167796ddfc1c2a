"""A batch's plain queries in one greedy launch: one query, more queries than
blocks, sizes from a handful of sets to most of the batch, sets long enough to be
shared in pieces -- every query equal to the oracle's."""
import pytest

import oracle as O
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def check(im, specs, kmax):
    """specs: (graph, model, k, theta, seed)"""
    graphs = {}
    for g, *_ in specs:
        graphs.setdefault(id(g), im.Graph(g))
    b = im.im_batch_create()
    out = im.im_solve_batch(b, [(graphs[id(g)].handle, m, k, th, sd) for g, m, k, th, sd in specs], kmax)
    im.im_batch_destroy(b)
    for (g, m, k, th, sd), (seeds, gains, cov, entries) in zip(specs, out):
        ref = O.sample(O.LT if m else O.IC, g, sd, 0, th)
        r = O.greedy(g.n, ref, O.invert(g.n, ref), k)
        assert entries == ref.members.size
        assert seeds.tolist() == r.seeds.tolist()
        assert gains.tolist() == r.gains.tolist()
        assert cov == r.coverage
    for G in graphs.values():
        G.close()


def test_one_query(im):
    check(im, [(inputs.rmat_graph(1 << 12, 1 << 16, 3, "lt"), 1, 40, 5000, 9)], 40)


def test_more_queries_than_blocks(im):
    g = inputs.rmat_graph(200, 1500, 3, "lt")
    check(im, [(g, q % 2, 1 + q % 9, 1 + (q * 37) % 120, q) for q in range(700)], 10)


def test_uneven_queries(im):
    a, b = inputs.rmat_graph(1 << 13, 1 << 17, 3, "lt"), inputs.rmat_graph(33, 200, 4, "lt")
    check(im, [(a, 1, 60, 40_000, 1), (b, 0, 5, 3, 2), (a, 0, 7, 100, 3), (b, 1, 20, 2000, 4), (a, 0, 30, 9000, 5)], 64)


def test_long_sets(im):
    g = inputs.rmat_graph(9000, 150_000, 2, "u0.1")
    check(im, [(g, 0, 25, 300, 1), (g, 0, 3, 40, 2)], 25)
