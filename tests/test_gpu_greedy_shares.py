"""The standard greedy where the list of a step's vertex is a share of one entry
per warp, of a whole chunk per warp, and one entry more than either."""
import pytest

import numpy as np
import oracle as O
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_warp,more", [(0, 1), (1, 0), (1, 1), (2, 1), (16, 0), (16, 1), (33, 7)])
def test_greedy_list_shares(per_warp, more):
    import torch
    from paper_2408_10982_gb300 import im

    n = 5000
    dst = np.arange(1, n, dtype=np.int64)
    in_off, in_src = inputs.in_csr(n, np.zeros(n - 1, np.int64), dst)
    g = inputs.Graph(n, in_off, in_src, np.full(n - 1, 2**32 - 1, np.uint32))   # every set holds vertex 0
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 2 * 16
    theta = per_warp * warps + more
    G = im.Graph(g)
    P = im.Pool(G, theta, 2 * theta)
    P.sample(im.IM_IC, 11, 0, theta)
    ref = O.sample(O.IC, g, 11, 0, theta)
    c = P.cover(4)
    r = O.greedy(n, ref, O.invert(n, ref), 4)
    assert c.seeds.tolist() == r.seeds.tolist()
    assert c.gains.tolist() == r.gains.tolist()
    assert c.coverage == r.coverage == theta
    P.close()
    G.close()
