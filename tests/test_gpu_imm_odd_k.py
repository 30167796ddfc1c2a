"""im_solve with an odd number of seeds: its 8-byte results lie behind k 4-byte
seeds and k 8-byte gains, at an aligned address for every k."""
import pytest

import oracle as O
from oracle import imm as oimm
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 3, 7, 10, 89])
def test_imm_any_k(k):
    from paper_2408_10982_gb300 import im
    im.lib()
    g = inputs.rmat_graph(4096, 40000, 3, "lt")
    ref = oimm.imm(g, O.LT, k, 0.5, 1.0, 11)
    G = im.Graph(g)
    seeds, cov, theta, info = im.im_solve(G.handle, im.IM_LT, k, 0.5, 1.0, 11)
    assert theta == ref.theta
    assert seeds.tolist() == ref.seeds.tolist()
    assert cov == ref.coverage
    G.close()
