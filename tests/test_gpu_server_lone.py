"""A request that finds an idle worker is taken at once: while a long batch runs, pairs of small
requests 1.5 ms apart do not wait to share a batch.  (There is no heavy lane; with one, a request
may wait behind the lane's sampling kernels.)"""
import time

import pytest

import oracle as O
from paper_2408_10982_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def im():
    from paper_2408_10982_gb300 import im as m
    m.lib()
    return m


def test_small_requests_do_not_wait(im):
    gl, gs = inputs.rmat_graph(1 << 17, 1 << 21, 3, "lt"), inputs.rmat_graph(1 << 10, 1 << 13, 3, "lt")
    L, S = im.Graph(gl), im.Graph(gs)
    pairs, theta, k = 7, 500, 4
    srv = im.im_server_create(workers=16, max_batch=64, mem_budget=200 << 30)
    try:
        warm = [im.im_server_submit(srv, g.handle, m, k, theta, 1) for g, m in ((L, im.IM_IC), (S, im.IM_LT))]
        for t in warm:
            im.im_server_wait(srv, t, k, 60)
        before = im.im_server_stats(srv)[0]
        long = im.im_server_submit(srv, L.handle, im.IM_IC, 50, 1 << 23, 2)
        time.sleep(0.02)                                 # it runs
        small = []
        for q in range(pairs):
            for _ in range(2):
                small.append((im.im_server_submit(srv, S.handle, im.IM_LT, k, theta, 100 + len(small)), 100 + len(small)))
                time.sleep(0.0015)
            time.sleep(0.004)
        got = [(im.im_server_wait(srv, t, k, 60), seed) for t, seed in small]
        im.im_server_wait(srv, long, 50, 60)
        batches = im.im_server_stats(srv)[0] - before
    finally:
        im.im_server_destroy(srv)
    for (seeds, cov, _), seed in got:
        ref = O.sample(O.LT, gs, seed, 0, theta)
        r = O.greedy(gs.n, ref, O.invert(gs.n, ref), k)
        assert seeds.tolist() == r.seeds.tolist() and cov == r.coverage
    L.close()
    S.close()
    assert batches > 1 + pairs + pairs // 2              # 1 + 2 pairs; 1 + pairs if they wait for company
