"""The server's pool and streams: what a large request takes of the pool, and
which poll launches a request."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCoreServer  # noqa: E402


def test_two_large_requests_fit():
    """A pool with room for two requests' graphs, results and peel state (16
    bytes per vertex and 8 per 64 arcs) admits both at once."""
    n = 200_000
    s, d = gg.er(n, 20 * n, seed=3)
    off, adj = oracle.build_csr(n, s, d)
    want = oracle.bz(n, off, adj)
    m = len(adj)
    rounds = 512 * (2 * int(m ** 0.5) + 8)
    pool = 2 * (8 * n + 4 * m + 4 * n + 20 * n + m // 8 + rounds + (1 << 18))
    outs = [np.full(n, -9, np.int32) for _ in range(2)]
    with KCoreServer(0, pool_bytes=pool, large_vertices=1000) as srv:
        t = [srv.submit(off, adj, c) for c in outs]
        assert None not in t
        res, stop = {}, time.time() + 30
        while len(res) < 2 and time.time() < stop:
            res.update({x: (km, st) for x, km, st in srv.poll()})
    for x, c in zip(t, outs):
        assert res[x] == (int(want.max()), 0)
        np.testing.assert_array_equal(c, want)


def test_a_poll_launches_on_the_stream_it_finds_finished():
    """One launch stream: the poll that finds its launch finished also launches
    the request that became ready meanwhile."""
    n, s, d = gg.complete(50)
    off, adj = oracle.build_csr(n, s, d)
    outs = [np.full(n, -9, np.int32) for _ in range(2)]

    with KCoreServer(0, pool_bytes=1 << 26, streams=1) as srv:
        got = []

        def poll():
            got.extend(t for t, _, _ in srv.poll())
            torch.cuda.synchronize()

        a = srv.submit(off, adj, outs[0])
        torch.cuda.synchronize()
        poll()  # launches a
        b = srv.submit(off, adj, outs[1])
        torch.cuda.synchronize()
        poll()  # finds a finished; launches b
        poll()  # finds b finished: its results are copied back
        np.testing.assert_array_equal(outs[1], 49)
        poll()
        assert sorted(got) == [a, b]
    np.testing.assert_array_equal(outs[0], 49)
