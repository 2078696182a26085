"""The CSR check over rows of 32 arcs: runs of vertices without arcs longer
than a row's 32 list starts, lists longer than a warp's share, and an arc
without its reverse in either direction (towards the longer and the shorter
list)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore, KCoreError  # noqa: E402
from tests.gpu_util import to_dev  # noqa: E402


def sparse_ids(gap, hub):
    """A random graph on every gap-th id, with a hub of `hub` neighbours."""
    r = np.random.default_rng(gap * 1000 + hub)
    k = max(hub + 2, 300)
    s, d = r.integers(0, k, 3 * k), r.integers(0, k, 3 * k)
    s = np.concatenate([s, np.zeros(hub, np.int64)])
    d = np.concatenate([d, np.arange(1, hub + 1)])
    n = k * gap + 70
    return (n, *oracle.build_csr(n, (s * gap + 40).astype(np.int32), (d * gap + 40).astype(np.int32)))


@pytest.mark.parametrize("gap", [1, 2, 31, 33, 65, 200])
@pytest.mark.parametrize("hub", [0, 5, 513, 5000])
def test_rows(gap, hub):
    n, off, adj = sparse_ids(gap, hub)
    with KCore(0) as k:
        o, a = to_dev(off, adj)
        k.validate_csr(o, a)
        src = np.repeat(np.arange(n), np.diff(off))
        deg = np.diff(off)
        up = deg[adj] > deg[src]
        for pick in (np.flatnonzero(up)[:1], np.flatnonzero(deg[adj] < deg[src])[-1:]):
            for j in pick:  # drop arc j, keep its reverse
                v = src[j]
                off2 = off.copy()
                off2[v + 1:] -= 1
                o2, a2 = to_dev(off2, np.delete(adj, j))
                with pytest.raises(KCoreError) as e:
                    k.validate_csr(o2, a2)
                assert e.value.code == "NOT_SIMPLE"
                st = k.stats()
                assert (st["invalid_check"], st["invalid_vertex"]) == (6, int(adj[j]))


def test_hub_of_more_than_2_to_30_arcs():
    """A star of 2^30 + 1,000 leaves, its hub without the arc to the last leaf:
    the third launch searches every leaf's arc in the hub's list."""
    leaves = (1 << 30) + 1000
    adj = torch.zeros(2 * leaves - 1, dtype=torch.int32, device="cuda")
    adj[:leaves - 1] = torch.arange(1, leaves, dtype=torch.int32, device="cuda")
    off = torch.arange(leaves - 2, 2 * leaves, dtype=torch.int64, device="cuda")
    off[0] = 0
    with KCore(0) as k:
        with pytest.raises(KCoreError) as e:
            k.validate_csr(off, adj)
        assert e.value.code == "NOT_SIMPLE"
        s = k.stats()
        assert (s["invalid_check"], s["invalid_vertex"], s["invalid_arc"]) == (6, leaves, 2 * leaves - 2)
