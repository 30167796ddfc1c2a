"""The radix build of the covering subsets at every number of passes and ballots
(vertex ids of 0 to 21 bits), at pool sizes around a tile of 8,192 pairs, and
with sets that span many tiles: equal to the oracle's, as stored."""
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


def check(im, g, model, theta):
    G = im.Graph(g)
    P = im.Pool(G, theta, theta * min(g.n, 60_000) + 8)
    P.sample(model, 9, 0, theta)
    ref = O.sample(model, g, 9, 0, theta)
    vtx_off, set_ids = P.index()
    ref_off, ref_ids = O.invert(g.n, ref)
    assert np.array_equal(vtx_off, ref_off)
    assert np.array_equal(set_ids, ref_ids)
    P.close()
    G.close()
    return ref.members.size


# one pass up to 1,024 vertices, two up to 1,048,576, then three; 8 or 10 ballots
@pytest.mark.parametrize("n,theta", [(1, 3), (2, 9000), (33, 8193), (256, 3000), (257, 3000), (1024, 4000),
                                     (1025, 4000), (65_536, 3000), (65_537, 3000), (262_144, 2000),
                                     (1 << 20, 2000), ((1 << 20) + 1, 2000)])
def test_digits(im, n, theta):
    m = 0 if n == 1 else min(4 * n, n * (n - 1) // 2)
    if m == 0:
        g = inputs.Graph(1, np.zeros(2, np.int64), np.zeros(0, np.int32), np.zeros(0, np.uint32))
    else:
        g = inputs.rmat_graph(n, m, 5, "lt")
    check(im, g, O.LT, theta)


# singletons: as many pairs as sets, around one and two tiles
@pytest.mark.parametrize("theta", [1, 8191, 8192, 8193, 16384, 16385])
def test_tile_edges(im, theta):
    n = 700
    g = inputs.Graph(n, np.zeros(n + 1, np.int64), np.zeros(0, np.int32), np.zeros(0, np.uint32))
    assert check(im, g, O.IC, theta) == theta


# sets longer than a tile
def test_sets_over_tiles(im):
    assert check(im, inputs.rmat_graph(50_021, 900_001, 9, "ic0.2"), O.IC, 40) > 20 * 8192
