"""Device memory of a batch of many small queries, and what the server takes a request to need."""
import time

import pytest

from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def test_small_queries_take_rows_for_their_vertices(im):
    """700 queries of 200 vertices and a handful of sets: 33 words for every vertex that may be
    a hub, 0.03 MB a query and not 0.13 (and 0.01 MB of everything else)."""
    import torch
    G = im.Graph(inputs.rmat_graph(200, 1500, 3, "lt"))
    nq = 700
    b = im.im_batch_create()
    im.im_solve_batch(b, [(G.handle, 1, 1, 1, 1)], 10)   # the graph's tables, the library's own memory
    im.im_trim_memory()
    before = torch.cuda.mem_get_info()[0]
    im.im_solve_batch(b, [(G.handle, 1, 1 + q % 9, 1 + q % 120, q) for q in range(nq)], 10)
    used = before - torch.cuda.mem_get_info()[0]
    im.im_batch_destroy(b)
    G.close()
    assert used < nq * (80 << 10)


def test_the_server_counts_the_rows(im):
    """Requests of 200 vertices and one set behind a long one, under a budget of 1 MB: a
    batch takes as many as their rows of 26 KB allow."""
    big, small = inputs.rmat_graph(1 << 17, 1 << 21, 3, "lt"), inputs.rmat_graph(200, 1500, 3, "lt")
    L, S = im.Graph(big), im.Graph(small)
    srv = im.im_server_create(workers=1, max_batch=256, mem_budget=1 << 20)
    try:
        tickets = [im.im_server_submit(srv, L.handle, im.IM_IC, 50, 1 << 22, 2)]
        time.sleep(0.02)
        tickets += [im.im_server_submit(srv, S.handle, im.IM_LT, 3, 1, q) for q in range(200)]
        for t in tickets:
            im.im_server_wait(srv, t, 50, 60)
        batches = im.im_server_stats(srv)[0]
    finally:
        im.im_server_destroy(srv)
    L.close()
    S.close()
    assert batches >= 1 + 200 * 26_000 // (1 << 20)
