"""IC sampling where the kernels change their way of working: lists of in-edges
around the lengths at which a vertex gets a whole warp (or block), first and
last edge groups cut at every offset, equal and unequal in-weights, the visited
set as bitmap, hash set and spilled, and sets handed to the second pass."""
import numpy as np
import pytest

import oracle
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu

# in-degrees around the group (4), warp (96, 128, 256) and block (2048) limits
DEGREES = [0, 1, 2, 3, 4, 5, 31, 63, 64, 65, 92, 93, 95, 96, 97, 127, 128, 129, 255, 256, 257, 259, 260,
           2043, 2044, 2047, 2048, 2049, 2052]


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def degree_graph(n, seed, weights):
    """n vertices; the first take the in-degrees above in turn, the others 0 to 8."""
    rng = np.random.default_rng(seed)
    deg = np.array([DEGREES[v % len(DEGREES)] if v < 4 * len(DEGREES) else int(rng.integers(0, 9))
                    for v in range(n)])
    src = np.concatenate([rng.choice(n, size=d, replace=False) for d in deg if d])
    dst = np.repeat(np.arange(n), deg)
    keep = src != dst
    in_off, in_src = inputs.in_csr(n, src[keep].astype(np.int64), dst[keep])
    m = in_src.shape[0]
    d = np.diff(in_off)
    if weights == "wc":
        w = inputs.weights_inverse_indegree(in_off)
    elif weights == "mixed":                   # per vertex: equal, unequal, all zero, all live
        kind = np.repeat(np.arange(n) % 4, d)
        w = rng.integers(0, 1 << 30, size=m).astype(np.uint32)
        w[kind == 0] = np.uint32(0.05 * 2**32)
        w[kind == 2] = 0
        w[kind == 3] = np.uint32(2**32 - 1)
    else:
        w = inputs.weights_uniform(m, float(weights))
    return inputs.Graph(n, in_off, in_src, w)


def check(im, g, seed, theta):
    G = im.Graph(g)
    P = im.Pool(G, theta, theta * g.n)
    P.sample(im.IM_IC, seed, 5, theta)
    set_off, members = P.export()
    ref = oracle.sample(oracle.IC, g, seed, 5, theta)
    assert np.array_equal(set_off, ref.set_off)
    assert np.array_equal(members, ref.members)
    assert P.info()[2] == ref.examined
    P.close()
    G.close()


# 4,096 and 32,768 vertices: bitmap in shared memory; 32,769: hash set
@pytest.mark.parametrize("n", [4096, 32768, 32769])
@pytest.mark.parametrize("weights", ["wc", "0.02", "mixed"])
def test_ic_list_lengths(im, n, weights):
    check(im, degree_graph(n, n % 1000 + 7, weights), 11, 257)


# sets of a few hundred members, around the hash set's limit of 384
@pytest.mark.parametrize("weights", ["0.2", "0.25"])
def test_ic_hash_set_spills(im, weights):
    check(im, inputs.rmat_graph(40_001, 120_000, 5, "ic" + weights), 3, 400)


# sets that reach the second pass: by their frontier (percolating), from both
# kinds of visited set, and with every edge live
@pytest.mark.parametrize("n,m,weights", [(20_011, 400_000, "ic0.2"), (50_021, 900_001, "ic0.1"),
                                         (50_021, 900_001, "trivalency"), (33_000, 300_000, "ic0.9999")])
def test_ic_handed_over(im, n, m, weights):
    check(im, inputs.rmat_graph(n, m, 9, weights), 21, 96)


# chains: sets of every length up to n = 20,011, one member a level -- past a
# warp's sort (1,024), its queue (16,384) and a block's sort (16,384)
@pytest.mark.parametrize("model", [0, 1])
def test_long_chains(im, model):
    n = 20_011
    src = np.arange(n - 1, dtype=np.int64)
    in_off, in_src = inputs.in_csr(n, src, src + 1)
    g = inputs.Graph(n, in_off, in_src, np.full(n - 1, 2**32 - 1, np.uint32))
    G = im.Graph(g)
    P = im.Pool(G, 40, 40 * n)
    P.sample(model, 17, 0, 40)
    set_off, members = P.export()
    ref = oracle.sample(oracle.LT if model else oracle.IC, g, 17, 0, 40)
    assert np.array_equal(set_off, ref.set_off)
    assert np.array_equal(members, ref.members)
    assert np.diff(ref.set_off).max() > 16384
    P.close()
    G.close()
