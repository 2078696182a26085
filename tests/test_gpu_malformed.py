"""Malformed graphs through the batched peel's kernels (batches, mode 4, the
server): the offsets and lists that reach a kernel's own checks are reported,
and the sound graphs beside them are peeled."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore, KCoreError, KCoreServer  # noqa: E402
from tests.batch_util import oracle_segmented  # noqa: E402
from tests.gpu_util import assert_parity, to_dev  # noqa: E402


def run_batch(k, gv, off, adj):
    core = torch.full((len(off) - 1,), -9, dtype=torch.int32, device="cuda")
    km = torch.full((len(gv) - 1,), -9, dtype=torch.int32, device="cuda")
    err = None
    try:
        k.decompose_batched(torch.from_numpy(gv).cuda(), *to_dev(off, adj), coreness=core, kmax=km)
    except KCoreError as e:
        err = e.code
    return core.cpu().numpy(), km.cpu().numpy(), err


FORMS = [dict(), dict(batch_block=512), dict(batch_block=256), dict(batch_cluster=4, batch_big_arcs=1),
         dict(batch_cluster=2, batch_block=512)]


@pytest.mark.parametrize("opts", FORMS, ids=str)
@pytest.mark.parametrize("sound", [0, 1, 700])
def test_last_offset_below_the_first(opts, sound):
    """The last graph's arcs number less than none; the others are sound, up to
    more than the kernel has teams."""
    parts = [gg.complete(20 + i % 5) for i in range(sound)] + [gg.path(30)]
    gv, off, adj = oracle_segmented([p[0] for p in parts], [(p[1], p[2]) for p in parts])
    want_core, want_km = oracle.bz_batch(gv, off, adj)
    bad = off.copy()
    bad[-1] = bad[gv[-2]] - 1
    with KCore(0, **opts) as k:
        core, km, err = run_batch(k, gv, bad, adj)
        assert err == "NOT_SIMPLE"
        assert km[-1] == -1
        np.testing.assert_array_equal(km[:-1], want_km[:-1])
        np.testing.assert_array_equal(core[:gv[-2]], want_core[:gv[-2]])
        core, km, err = run_batch(k, gv, off, adj)
        assert err is None
        np.testing.assert_array_equal(core, want_core)


@pytest.mark.parametrize("cluster", [0, 2, 8])
def test_last_offset_below_the_first_mode4(cluster):
    n, s, d = gg.complete(50)
    off, adj = oracle.build_csr(n, s, d)
    bad = off.copy()
    bad[-1] = -1
    with KCore(0, sync_mode=4, batch_cluster=cluster) as k:
        with pytest.raises(KCoreError) as e:
            k.decompose(*to_dev(bad, adj))
        assert e.value.code == "NOT_SIMPLE"
        assert_parity(k, n, off, adj)


@pytest.mark.parametrize("cluster", [1, 4])
def test_last_offset_below_the_first_served(cluster):
    n, s, d = gg.complete(50)
    off, adj = oracle.build_csr(n, s, d)
    want = oracle.bz(n, off, adj)
    bad = off.copy()
    bad[-1] = -1
    outs = [np.full(n, -9, np.int32) for _ in range(4)]
    with KCoreServer(0, pool_bytes=1 << 26, batch_cluster=cluster) as srv:
        t = [srv.submit(o, adj, c) for o, c in zip((off, bad, off, off), outs)]
        res, stop = {}, time.time() + 30
        while len(res) < 4 and time.time() < stop:
            res.update({x: (km, st) for x, km, st in srv.poll()})
    assert res[t[1]][1] != 0
    for i in (0, 2, 3):
        assert res[t[i]][0] == 49  # (a launch's requests share its status)
        np.testing.assert_array_equal(outs[i], want)


@pytest.mark.parametrize("opts", FORMS, ids=str)
@pytest.mark.parametrize("per", [1, 4])
def test_arcs_into_a_vertex_without_arcs(opts, per):
    """Not symmetric: more than 2^16 arcs into the last vertex, which has none
    of its own. Its 16-bit d~ comes round and lands on the level that many
    others land on at once; its empty list is reported, and no arc is read for
    it (its list starts where the arcs end)."""
    a = 70_000 // per  # vertices of `per` arcs to the last vertex and one to a vertex of a K4, which it lands on level per + 1
    x = 4 * ((a + 3) // 4)
    n = a + x + 1
    block = np.arange(x) // 4 * 4
    others = np.stack([(np.arange(x) + 1 + j) % 4 for j in range(3)], 1) + block[:, None]
    pad = np.zeros((x, per - 1), np.int64)  # degree per + 2 = level + 1: arcs to the first vertex, repeated
    lists = np.concatenate([np.concatenate([np.full((a, per), n - 1), a + np.arange(a)[:, None]], 1).ravel(),
                            np.concatenate([pad, a + others], 1).ravel()])
    deg = np.concatenate([np.full(a, per + 1), np.full(x, per + 2), [0]])
    off = np.concatenate([[0], np.cumsum(deg)])
    assert off[-1] == len(lists) and off[-2] == off[-1]
    gv = np.array([0, n], np.int64)
    with KCore(0, **opts) as k:
        _, _, err = run_batch(k, gv, off, lists)
        assert err == "NOT_SIMPLE"
        nn, s, d = gg.complete(60)
        assert_parity(k, nn, *oracle.build_csr(nn, s, d))
