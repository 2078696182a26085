"""The batched CSR build's edge route (one key per edge, global ids), which
starts at three sort tiles per SM: empty and tiny graphs at the ends and between
large ones, unaligned edge arrays, ids outside their graph, a workspace with
room for the arc route only. Exact against the oracle's builder."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2502_08042_gb300 import KCore, KCoreError, _native  # noqa: E402
from tests.batch_util import oracle_segmented  # noqa: E402

TINY = ([0, 1, 2, 5, 0, 9], [0, 2, 1, 7, 0, 20])  # vertices, edges
BATCHES = {
    "large": ([0, 0, 40_000, 0, 60_001, 1, 50_000, 0], [0, 0, 900_000, 0, 700_003, 3, 800_000, 0]),
    "tiny_between": (TINY[0] * 150 + [70_000] + TINY[0] * 150 + [50_000, 30_011] + TINY[0],
                     TINY[1] * 150 + [900_001] + TINY[1] * 150 + [600_000, 700_000] + TINY[1]),
    "forty": ([10_000 + i for i in range(40)], [50_000 + 37 * i for i in range(40)]),
    "one": ([0, 90_000, 0], [0, 1_900_001, 0]),
}


def takes_edge_route(n, E, top):
    """The builder's rule, and that it is still the rule."""
    with open(os.path.join(_native.CSRC, "csr_build.cu")) as f:
        assert "E > (long long)sms * 3 * kSortTile && edge_passes < 2 * arc_passes" in f.read()
    bits = lambda x: max(1, (x - 1).bit_length())  # noqa: E731
    up = lambda x: (x + 7) // 8  # noqa: E731
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return E > sms * 3 * 4096 and up(2 * bits(n)) + up(bits(n)) < 2 * up(bits(n) + bits(top + 1))


def batch(name, shift=0):
    ns, ms = BATCHES[name]
    r = np.random.default_rng(len(ns))
    lists = []
    for n, m in zip(ns, ms):
        s, d = (r.integers(0, max(n, 1), m, dtype=np.int32) for _ in range(2))
        if m > 1:  # repeats, the other way round
            s[m // 2:], d[m // 2:] = d[:m - m // 2].copy(), s[:m - m // 2].copy()
        lists.append((s, d))
    dev, pad = "cuda:0", np.zeros(shift, np.int32)
    args = [torch.tensor(np.cumsum([0] + list(ns)), device=dev), torch.tensor(np.cumsum([0] + list(ms)), device=dev)]
    args += [torch.from_numpy(np.concatenate([pad] + [x[i] for x in lists])).to(dev)[shift:] for i in range(2)]
    args.append(max(ns))
    assert takes_edge_route(sum(ns), sum(ms), max(ns))
    return args, ns, ms, lists


@pytest.mark.parametrize("name", list(BATCHES))
@pytest.mark.parametrize("small_ws,shift", [(False, 0), (False, 1), (True, 3)])
def test_edge_route(name, small_ws, shift):
    args, ns, ms, lists = batch(name, shift)
    _, want_off, want_adj = oracle_segmented(ns, lists)
    with KCore(0) as k:
        if small_ws:
            size = k.build_csr_workspace_size(sum(ns), sum(ms)) - 8 * sum(ns) + 256
            k.set_workspace(torch.empty(size, dtype=torch.uint8, device="cuda:0"))
        for _ in range(2):
            off, adj = k.build_csr_batched(*args)
            np.testing.assert_array_equal(off.cpu().numpy(), want_off)
            np.testing.assert_array_equal(adj.cpu().numpy(), want_adj)


@pytest.mark.parametrize("side", [2, 3])
@pytest.mark.parametrize("where,value", [("first", 40_000), ("first", -1), ("last", 50_000), ("middle", 2**31 - 1),
                                         ("tiny", 1)])
def test_id_outside_its_graph(side, where, value):
    args, ns, ms, _ = batch("large")
    ends = np.cumsum(ms)
    at = {"first": 0, "last": ends[-1] - 1, "middle": ends[4] - 1, "tiny": ends[4] + 1}[where]
    args[side][int(at)] = value
    with KCore(0) as k:
        with pytest.raises(KCoreError, match="outside"):
            k.build_csr_batched(*args)
