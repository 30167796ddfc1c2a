"""Scratch of an IC sampling call: per sample what its result and its sort need, and nothing for the
state of samples that are handed over, of which there are few."""
import pytest

from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_ic_scratch_per_sample():
    import torch
    from paper_2408_10982_gb300 import im
    theta = 1 << 24
    G = im.Graph(inputs.rmat_graph(64, 200, 3, "ic0.1"))
    warm = im.Pool(G, 64, 4096)                          # the graph's records, the library's own memory
    warm.sample(im.IM_IC, 1, 0, 64)
    warm.close()
    P = im.Pool(G, theta, 8 * theta)
    im.im_trim_memory()
    before = torch.cuda.mem_get_info()[0]
    P.sample(im.IM_IC, 1, 0, theta)
    used = before - torch.cuda.mem_get_info()[0]
    assert P.info()[0] == theta
    P.close()
    G.close()
    # 8 + 4 bytes of place and size, 8 of the list of left samples, 16 of the sort's lists, a quarter
    # of room to grow, and about 50 MB whatever the number of samples; 24 bytes of state a sample more are 30
    assert used < 36 * 1.25 * theta + (160 << 20)
