"""Short CSR builds captured in a CUDA graph (their early starts become the
graph's edges) and run one after another on the same buffers: every replay
builds the CSR of the inputs at hand."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore  # noqa: E402
from tests.batch_util import oracle_segmented  # noqa: E402


def lists(n, m, i):
    r = np.random.default_rng(1000 * i + m)
    hi = max(1, n // (1 + i % 3))  # sparse and dense ids: other counts of repeats and empty lists
    return r.integers(0, hi, m, dtype=np.int32), r.integers(0, hi, m, dtype=np.int32)


@pytest.mark.parametrize("n,m", [(50, 300), (3_000, 4_097), (99_991, 400_003), (70_000, 1_500_000)])
def test_single(n, m):
    dev = "cuda:0"
    S, D = (torch.zeros(m, dtype=torch.int32, device=dev) for _ in range(2))
    with KCore(0) as k:
        k.build_csr(n, S, D)  # the workspace exists before the capture
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            off, adj, cnt = k.build_csr(n, S, D, sync=False)
        for i in range(6):
            s, d = lists(n, m, i)
            S.copy_(torch.from_numpy(s))
            D.copy_(torch.from_numpy(d))
            for _ in range(3):
                graph.replay()
            torch.cuda.synchronize()
            want_off, want_adj = oracle.build_csr(n, s, d)
            np.testing.assert_array_equal(off.cpu().numpy(), want_off)
            np.testing.assert_array_equal(adj.cpu().numpy()[:int(cnt)], want_adj)


def test_batch():
    dev = "cuda:0"
    ns, ms = [0, 900, 40_000, 7, 0], [0, 4_096, 150_001, 30, 0]
    E = sum(ms)
    gv = torch.tensor(np.cumsum([0] + ns), device=dev)
    eo = torch.tensor(np.cumsum([0] + ms), device=dev)
    S, D = (torch.zeros(E, dtype=torch.int32, device=dev) for _ in range(2))
    with KCore(0) as k:
        k.build_csr_batched(gv, eo, S, D, max(ns))
        N, G = sum(ns), len(ns)
        off = torch.empty(N + 1, dtype=torch.int64, device=dev)
        adj = torch.empty(2 * E, dtype=torch.int32, device=dev)
        cnt = torch.zeros(1, dtype=torch.int64, device=dev)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):  # (the Python call reads gv on the host: the C entry point)
            st = k._L.kcore_build_csr_batched(k._h, G, N, E, max(ns), gv.data_ptr(), eo.data_ptr(), S.data_ptr(),
                                              D.data_ptr(), off.data_ptr(), adj.data_ptr(), cnt.data_ptr(),
                                              torch.cuda.current_stream().cuda_stream)
            assert st == 0
        for i in range(4):
            edge_lists = [lists(n, m, i) if n else (np.zeros(0, np.int32),) * 2 for n, m in zip(ns, ms)]
            S.copy_(torch.from_numpy(np.concatenate([s for s, _ in edge_lists])))
            D.copy_(torch.from_numpy(np.concatenate([d for _, d in edge_lists])))
            graph.replay()
            torch.cuda.synchronize()
            _, want_off, want_adj = oracle_segmented(ns, edge_lists)
            np.testing.assert_array_equal(off.cpu().numpy(), want_off)
            np.testing.assert_array_equal(adj.cpu().numpy()[:int(cnt)], want_adj)
