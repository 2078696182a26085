"""The batched peel's forms: induced degrees wholly, partly or not in shared
memory (16 and 32 bits), whole CTAs and teams, chunks whose arcs start many
short lists or few long ones. Exact against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore  # noqa: E402
from tests.test_gpu_push import cliques_on_peelers  # noqa: E402


def segmented(graphs):
    offs, adjs, gv, at = [np.zeros(1, np.int64)], [], [0], 0
    wants = []
    for n, s, d in graphs:
        off, adj = oracle.build_csr(n, s, d)
        offs.append(off[1:] + at)
        adjs.append(adj)
        at += len(adj)
        gv.append(gv[-1] + n)
        wants.append(oracle.bz(n, off, adj) if n else np.zeros(0, np.int32))
    dev = "cuda:0"
    return (torch.tensor(gv, dtype=torch.int64, device=dev), torch.from_numpy(np.concatenate(offs)).to(dev),
            torch.from_numpy(np.concatenate(adjs).astype(np.int32)).to(dev), wants)


def check(k, batch):
    gv, off, adj, wants = batch
    core, km = k.decompose_batched(gv, off, adj)
    np.testing.assert_array_equal(core.cpu().numpy(), np.concatenate(wants))
    np.testing.assert_array_equal(km.cpu().numpy(), [int(w.max()) if len(w) else 0 for w in wants])


def mixed():
    gs = [cliques_on_peelers(k, f) for k, f in ((1, 300), (3, 90), (8, 700), (33, 40), (65, 70))]
    gs += [(n, *gg.er(n, 8 * n, seed=n)) for n in (999, 1000, 1001, 5000)]
    gs += [gg.staircase(120), gg.path(3000), gg.star(2500), gg.complete(1), gg.complete(90)]
    return gs


@pytest.mark.parametrize("opts", [dict(batch_smem_vertices=v) for v in (0, 1, 499, 500, 501, 4000)] + [
    dict(batch_block=512, batch_smem_vertices=300), dict(batch_block=256, batch_smem_vertices=300),
    dict(batch_cluster=2, batch_big_arcs=4000, batch_smem_vertices=300)],
    ids=lambda o: ",".join(f"{a[6:]}={b}" for a, b in o.items()))
def test_split_and_teams(opts):
    batch = segmented(mixed())
    with KCore(0, **opts) as k:
        check(k, batch)


@pytest.mark.parametrize("copies", [1, 2, 303, 305])
def test_team_boundaries(copies):
    """One large graph and many small ones: the CTAs leave whole-graph work at
    different draws; counts on both sides of two teams per SM."""
    small = [(60 + i % 7, *gg.er(60 + i % 7, 300, seed=i)) for i in range(copies)]
    batch = segmented([(4000, *gg.er(4000, 40000, seed=1))] + small)
    with KCore(0) as k:
        check(k, batch)


@pytest.mark.parametrize("sv", [0, 65536, 70000 - 1, 70001])
def test_wide_degrees(sv):
    """A hub of 70,000 arcs: 32-bit induced degrees, split at sv vertices."""
    n, s, d = gg.star(70001)
    e = gg.er(n, 100000, seed=5)
    batch = segmented([(n, np.concatenate([s, e[0]]), np.concatenate([d, e[1]]))])
    with KCore(0, batch_smem_vertices=min(sv, 50000)) as k:
        check(k, batch)


@pytest.mark.parametrize("sv", [0, 1, 30_001, 50_000])
def test_wide_degrees_split(sv):
    """The same hub with the first sv vertices' 32-bit degrees in shared memory.
    (No graph with a degree of 2^16 fits there as a whole.)"""
    n, s, d = gg.star(70001)
    e = gg.er(n, 100000, seed=6)
    batch = segmented([(n, np.concatenate([s, e[0]]), np.concatenate([d, e[1]]))])
    with KCore(0, batch_smem_vertices=sv) as k:
        check(k, batch)
