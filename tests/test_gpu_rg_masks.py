"""The mask stage of RandGreedi (k_rg_stream_masks) on pools of just over 2^20 members -- shorter
ones go to a block per bucket -- with streams around the sizes of its groups (64 slots) and of
the window it reads ahead (512); and the cluster stage, more than 64 buckets and sets
beyond a block's bitmap."""
import pytest

import oracle as O
from paper_2408_10982_gb300 import inputs

from test_gpu_parity import _rg_compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    O.build()
    return m


@pytest.fixture(scope="module")
def pool(im):
    g, theta = inputs.rmat_graph(1 << 12, 1 << 16, 5, "lt"), 70_000
    assert 1 << 20 < O.sample(O.LT, g, 42, 0, theta).members.size < 1 << 21
    return g, theta


# slots = parts x k (alpha = 1)
@pytest.mark.parametrize("parts,k", [(1, 1), (7, 1), (63, 1), (16, 4), (13, 5), (64, 7), (449, 1), (128, 4), (27, 19), (54, 19)])
def test_stream_lengths(im, pool, parts, k):
    g, theta = pool
    _rg_compare(im, g, im.IM_LT, theta, k, parts, (1, 1), 0.077, False)


def test_the_most_buckets(im, pool):
    g, theta = pool
    _rg_compare(im, g, im.IM_LT, theta, 100, 148, (1, 4), 0.077, False)


def test_cluster_beyond_64_buckets(im):
    g = inputs.rmat_graph(1 << 10, 1 << 13, 5, "lt-u0.1")
    _rg_compare(im, g, im.IM_LT, 1_700_000, 150, 16, (1, 8), 0.077, False)
