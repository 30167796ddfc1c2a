"""Set offsets and subset offsets where the scan of counts changes its form: one
tile of 4,096 counts, eight, 8,192, and one count more than each."""
import pytest

import numpy as np
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 4096, 4097, 32768, 32769, 100_003])
@pytest.mark.parametrize("theta,more", [(1, 0), (4096, 1), (4097, 4096), (32768, 32768), (32769, 5), (300_001, 70_000)])
def test_offsets(n, theta, more):
    _check(n, theta, more)


@pytest.mark.parametrize("theta,more", [(1 << 25, 4097), ((1 << 25) + 1, 0)])
def test_offsets_of_many_sets(theta, more):
    _check(70_001, theta, more)


def _check(n, theta, more):
    from paper_2408_10982_gb300 import im

    # every other vertex has the vertex before it as a certain in-neighbour of no
    # further ones: sets of one or two members
    dst = np.arange(1, n, 2, dtype=np.int64)
    in_off, in_src = inputs.in_csr(n, dst - 1, dst)
    G = im.Graph(inputs.Graph(n, in_off, in_src, np.full(dst.size, 2**32 - 1, np.uint32)))
    P = im.Pool(G, theta + more, 2 * (theta + more))
    P.sample(im.IM_IC, 3, 0, theta)
    if more:
        P.sample(im.IM_IC, 3, theta, more)      # appended: the scan goes on from the total
    off, mem = P.export()
    size = np.diff(off)
    assert off[0] == 0 and off[-1] == mem.size and off.size == theta + more + 1
    assert ((size == 1) | (size == 2)).all()
    last = mem[off[1:] - 1]                     # the root: the larger id
    assert (size == 1 + (last & 1)).all()
    two = size == 2
    assert (mem[off[:-1][two]] == last[two] - 1).all()
    voff, ids = P.index()
    assert (np.diff(voff) == np.bincount(mem, minlength=n)).all() and voff[0] == 0
    assert ids.size == mem.size
    P.close()
    G.close()
