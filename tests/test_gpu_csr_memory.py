"""The batched CSR build on a device with less memory left than the edge route's
list starts take: it goes by arcs, as in a caller's workspace of that size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore  # noqa: E402


def test_batch_with_little_memory_left():
    dev = "cuda:0"
    ids, n, E = 5000, 1 << 28, 3_000_000  # list starts: 2 GB; everything else of either route: 0.1 GB
    r = np.random.default_rng(1)
    s, d = (r.integers(0, ids, E, dtype=np.int32) for _ in range(2))
    want_off, want_adj = oracle.build_csr(ids, s, d)
    S, D = torch.from_numpy(s).to(dev), torch.from_numpy(d).to(dev)
    gv = torch.tensor([0, n], dtype=torch.int64, device=dev)
    eo = torch.tensor([0, E], dtype=torch.int64, device=dev)
    off = torch.empty(n + 1, dtype=torch.int64, device=dev)
    adj = torch.empty(2 * E, dtype=torch.int32, device=dev)
    cnt = torch.zeros(1, dtype=torch.int64, device=dev)
    with KCore(0) as k:
        def build():
            st = k._L.kcore_build_csr_batched(k._h, 1, n, E, n, gv.data_ptr(), eo.data_ptr(), S.data_ptr(),
                                              D.data_ptr(), off.data_ptr(), adj.data_ptr(), cnt.data_ptr(), None)
            assert st == 0
            k.sync()
            m = int(cnt)
            assert m == len(want_adj)
            np.testing.assert_array_equal(off[:ids + 1].cpu().numpy(), want_off)
            assert bool((off[ids:] == m).all())
            np.testing.assert_array_equal(adj[:m].cpu().numpy(), want_adj)

        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        filler = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device=dev)
        try:
            build()
        finally:
            del filler
            torch.cuda.empty_cache()
        k.set_workspace(None)  # the next call allocates anew: with room, the edge route
        build()
