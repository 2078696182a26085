"""The CSR build's two routes for a batch (one key per edge, two arcs per edge)
and its tiles: edge counts around a sort tile and a warp's chunk, repeats and
self-loops, unaligned edge arrays. Exact against the oracle's builder."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore  # noqa: E402
from tests.batch_util import oracle_segmented  # noqa: E402


def edges(n, m, seed):
    r = np.random.default_rng(seed)
    s, d = r.integers(0, n, m, dtype=np.int32), r.integers(0, n, m, dtype=np.int32)
    if m > 10:
        s[m // 2:], d[m // 2:] = d[:m - m // 2].copy(), s[:m - m // 2].copy()  # repeats, the other way round
    return s, d


@pytest.mark.parametrize("m", [0, 1, 31, 32, 33, 255, 256, 257, 4095, 4096, 4097, 8193, 100_003])
@pytest.mark.parametrize("n,shift", [(1, 0), (3, 1), (700, 3), (70_001, 2)])
def test_single(n, m, shift):
    s, d = edges(n, m, 7 * m + n)
    want_off, want_adj = oracle.build_csr(n, s, d)
    pad = np.zeros(shift, np.int32)
    S = torch.from_numpy(np.concatenate([pad, s])).to("cuda:0")[shift:]
    D = torch.from_numpy(np.concatenate([pad, d])).to("cuda:0")[shift:]
    with KCore(0) as k:
        off, adj = k.build_csr(n, S, D)
    np.testing.assert_array_equal(off.cpu().numpy(), want_off)
    np.testing.assert_array_equal(adj.cpu().numpy(), want_adj)


def batch(ns, ms, seed):
    lists = [edges(n, m, seed + i) if n else (np.zeros(0, np.int32),) * 2 for i, (n, m) in enumerate(zip(ns, ms))]
    eo = np.cumsum([0] + [len(s) for s, _ in lists])
    dev = "cuda:0"
    args = (torch.tensor(np.cumsum([0] + list(ns)), device=dev), torch.tensor(eo, device=dev),
            torch.from_numpy(np.concatenate([s for s, _ in lists])).to(dev),
            torch.from_numpy(np.concatenate([d for _, d in lists])).to(dev), max(ns))
    return args, oracle_segmented(ns, lists)


# few graphs of many vertices (edge keys), many of few (arc keys), empty graphs at both ends
BATCHES = [([40_000, 60_000, 0, 50_000], [90_000, 4096, 0, 70_001]), ([20] * 300, [40] * 300),
           ([0, 0, 5, 100_000, 1, 0], [0, 0, 9, 200_003, 3, 0]), ([9], [0])]


@pytest.mark.parametrize("b", range(len(BATCHES)))
@pytest.mark.parametrize("small_ws", [False, True])
def test_batch_routes(b, small_ws):
    ns, ms = BATCHES[b]
    args, (gv, want_off, want_adj) = batch(ns, ms, 11)
    N, E = sum(ns), args[2].numel()
    with KCore(0) as k:
        if small_ws:
            # room for the arc route only: 8 bytes per vertex less than the single-graph build
            k.set_workspace(torch.empty(k.build_csr_workspace_size(N, E) - 8 * N + 512, dtype=torch.uint8, device="cuda:0"))
        off, adj = k.build_csr_batched(*args)
    np.testing.assert_array_equal(off.cpu().numpy(), want_off)
    np.testing.assert_array_equal(adj.cpu().numpy(), want_adj)


def test_batch_bad_id():
    ns, ms = BATCHES[0]
    args, _ = batch(ns, ms, 3)
    args[2][5] = 40_000  # the first graph's ids end at 39,999
    with KCore(0) as k:
        with pytest.raises(Exception, match="outside"):
            k.build_csr_batched(*args)
