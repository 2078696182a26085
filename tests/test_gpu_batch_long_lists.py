"""The batched peel on a frontier of 1,024 lists that hold more than 2^31 arcs
together: 1,024 hubs joined to every vertex of a clique and to every leaf."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.slow]

from paper_2502_08042_gb300 import KCore  # noqa: E402

HUBS, CLIQUE, LEAVES = 1024, 2000, 2_100_000


def graph():
    dev = "cuda:0"
    i32 = dict(dtype=torch.int32, device=dev)
    hub = torch.arange(HUBS, HUBS + CLIQUE + LEAVES, **i32)  # a hub's list: the clique, the leaves
    to_hubs = torch.arange(HUBS, **i32)                      # a leaf's list
    c = torch.arange(CLIQUE - 1, **i32)[None, :].expand(CLIQUE, -1)
    c = HUBS + c + (c >= torch.arange(CLIQUE, **i32)[:, None]).to(torch.int32)  # the other vertices of the clique
    clique = torch.cat([to_hubs.expand(CLIQUE, -1), c], 1)
    deg = torch.cat([torch.full((HUBS,), CLIQUE + LEAVES), torch.full((CLIQUE,), HUBS + CLIQUE - 1),
                     torch.full((LEAVES,), HUBS)]).to(dev)
    off = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), deg.cumsum(0)])
    adj = torch.empty(int(off[-1]), **i32)
    a, b = HUBS * hub.numel(), HUBS * hub.numel() + clique.numel()
    adj[:a].view(HUBS, -1).copy_(hub)
    adj[a:b] = clique.reshape(-1)
    adj[b:].view(LEAVES, HUBS).copy_(to_hubs)
    return off, adj


@pytest.mark.parametrize("cluster", [0, 8])
def test_frontier_of_more_than_2_to_31_arcs(cluster):
    off, adj = graph()
    assert HUBS * (CLIQUE + LEAVES) > 1 << 31
    gv = torch.tensor([0, off.numel() - 1], dtype=torch.int64, device="cuda:0")
    with KCore(0, batch_cluster=cluster, batch_big_arcs=1) as k:
        core, km = k.decompose_batched(gv, off, adj)
        # the leaves have HUBS neighbours; without them a hub has the clique's
        # CLIQUE, and a clique vertex the hubs and CLIQUE - 1
        assert int(km) == CLIQUE
        assert bool((core[:HUBS + CLIQUE] == CLIQUE).all())
        assert bool((core[HUBS + CLIQUE:] == HUBS).all())
