"""The bucket stage with a block per bucket (short streams, more than 64
buckets): every bucket equal to the oracle's, at stream lengths around a window
of 512 slots, set counts around a bitmap word, and subsets around a piece of
256 entries."""
import pytest

import oracle as O
from paper_2408_10982_gb300 import inputs
from test_gpu_parity import _rg_compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


# parts x streamed seeds = 511, 512, 513, 1,026 slots; the last two cases have
# 73 and 90 buckets
@pytest.mark.parametrize("Pn,k,alpha", [(73, 7, (1, 1)), (64, 8, (1, 1)), (27, 19, (1, 1)),
                                        (54, 19, (1, 1)), (33, 220, (1, 4)), (40, 800, (1, 8))])
def test_stream_lengths(im, Pn, k, alpha):
    g = inputs.rmat_graph(1 << 13, 1 << 17, 3, "lt")
    _rg_compare(im, g, im.IM_LT, 9001, k, Pn, alpha, 0.077, False)


@pytest.mark.parametrize("theta", [1, 31, 32, 33, 255, 257, 513])
def test_set_counts(im, theta):
    g = inputs.graph_small_ic()
    _rg_compare(im, g, im.IM_IC, theta, 12, 9, (1, 1), 0.2, False)


def test_many_buckets_percolating(im):
    """Subsets of hundreds to thousands of entries against 0.01-spaced thresholds (B = 231)."""
    g = inputs.rmat_graph(3000, 40000, 8, "ic0.1")
    assert O.num_buckets(10, 0.01) > 128
    _rg_compare(im, g, im.IM_IC, 4000, 10, 16, (1, 1), 0.01, False)
