"""The k'-core query's batch update counts in the query's output array: exact
against the oracle and against returning atomics, in a workspace without room
for counts, and a fresh handle allocates no more for it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import graphgen as gg  # noqa: E402
import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore  # noqa: E402
from tests.gpu_util import to_dev  # noqa: E402

N, SCALE = 1 << 22, 18  # the R-MAT graph's vertices lead a long tail of isolated ones


@pytest.fixture(scope="module")
def graph():
    s, d = gg.rmat(SCALE, 24, seed=5, perm_seed=6)
    off, adj = oracle.build_csr(N, s, d)
    assert len(adj) >= 1 << 22
    return off, adj, to_dev(off, adj)


@pytest.mark.parametrize("kprime", [15, 16, 17, 64, 130, 300, 5000])
def test_mask(graph, kprime):
    off, adj, (o, a) = graph
    want, size = oracle.kcore_mask(N, off, adj, kprime)
    with KCore(0) as k, KCore(0, batch_update=0) as plain:
        ws = torch.empty(plain.workspace_size(N, len(adj)), dtype=torch.uint8, device="cuda")
        for h in (k, plain):
            h.set_workspace(ws)
            for _ in range(2):
                mask, cnt = h.core_mask(o, a, kprime)
                np.testing.assert_array_equal(mask.cpu().numpy(), want)
                assert int(cnt) == size


def test_fresh_handle_allocates_no_more(graph):
    _, _, (o, a) = graph
    mask = torch.empty(N, dtype=torch.int32, device="cuda")
    used = []
    for opt in (0, 1):
        with KCore(0, batch_update=opt) as k:
            torch.cuda.synchronize()
            before = torch.cuda.mem_get_info()[0]
            k.core_mask(o, a, 64, mask=mask)
            used.append(before - torch.cuda.mem_get_info()[0])
    assert used[0] > 4 * N and used[1] == used[0]
