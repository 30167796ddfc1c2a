"""A batch refuses a graph of more than 26,214,400 vertices before it does any work, and takes one of
as many."""
import numpy as np
import pytest

from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu

LIMIT = 26_214_400


def graph(n):
    src = np.arange(1, 2001, dtype=np.int64)
    in_off, in_src = inputs.in_csr(n, src, src - 1)
    return inputs.Graph(n, in_off, in_src, np.full(2000, 1 << 31, np.uint32))


def test_the_limit():
    from paper_2408_10982_gb300 import im
    b = im.im_batch_create()
    G = im.Graph(graph(LIMIT + 1))
    im.im_profile_enable(True)
    im.im_profile_reset()
    for opts in (None, im.cover_opts(im.IM_RANDGREEDI, 4096)):
        with pytest.raises(im.ImError) as e:
            im.im_solve_batch(b, [(G.handle, im.IM_IC, 2, 50, 1) + ((opts,) if opts else ())], 2)
        assert im.status_str(e.value.status) == "unsupported"
    kernels = im.im_profile_read()
    im.im_profile_enable(False)
    assert not [k for k in kernels if k.startswith(("sample", "sort", "index_radix"))]
    G.close()
    G = im.Graph(graph(LIMIT))
    (seeds, gains, cov, entries), = im.im_solve_batch(b, [(G.handle, im.IM_IC, 2, 50, 1)], 2)
    P = im.Pool(G, 50, 5000)
    P.sample(im.IM_IC, 1, 0, 50)
    c = P.cover(2)
    assert seeds.tolist() == c.seeds.tolist() and cov == c.coverage and entries == P.info()[1]
    P.close()
    im.im_batch_destroy(b)
    G.close()
