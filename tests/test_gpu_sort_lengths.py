"""RRR sets come out ascending at every length that the sort treats apart (a lane's
sixteen keys, a warp's powers of two, two runs of 512, a block's)."""
import pytest

import numpy as np
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,n,theta", [
    ("IC", 20, 40), ("IC", 70, 1_000_003), ("IC", 300, 1_500_000), ("IC", 1100, 9000), ("IC", 2500, 4000),
    ("LT", 1030, 9000), ("LT", 2060, 9000), ("LT", 4200, 30_000), ("LT", 17_000, 2500)])
def test_sorted_at_every_length(model, n, theta):
    from paper_2408_10982_gb300 import im

    # a certain chain over shuffled names: the set of place p holds places 0 .. p
    rng = np.random.default_rng(n)
    name = rng.permutation(n).astype(np.int64)
    in_off, in_src = inputs.in_csr(n, name[:-1], name[1:])
    G = im.Graph(inputs.Graph(n, in_off, in_src, np.full(n - 1, 2**32 - 1, np.uint32)))
    P = im.Pool(G, theta, theta * n)
    P.sample(getattr(im, "IM_" + model), 17, 0, theta)
    off, mem = P.export()
    size = np.diff(off)
    assert size.min() >= 1 and size.max() <= n
    if theta > 20 * n:
        assert np.unique(size).size == n
    place = np.empty(n, np.int64)
    place[name] = np.arange(n)
    assert (place[mem] < np.repeat(size, size)).all()      # only members of the set ...
    up = mem[1:] > mem[:-1]
    up[off[1:-1] - 1] = True
    assert up.all()                                        # ... ascending, so each of them once
    P.close()
    G.close()
