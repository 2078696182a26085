"""Crossing vertices staged by a warp and pushed together, and the arc map of a
batch of items: whole iterations of crossings, lists on both sides of a slice
and of a 32-arc window, against the oracle (exact)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2502_08042_gb300 import KCore  # noqa: E402
from tests.gpu_util import assert_parity, to_dev  # noqa: E402


def cliques_on_peelers(k, f):
    """f vertices of degree k whose neighbours are the members of (k+1)-cliques,
    each member with one such neighbour: at level k the f vertices are the whole
    frontier and every arc they hold makes its target cross."""
    groups = -(-f * k // (k + 1))  # the last clique may have members without a peeler
    base = f
    i, j = np.triu_indices(k + 1, 1)
    s = [base + g * (k + 1) + i for g in range(groups)]
    d = [base + g * (k + 1) + j for g in range(groups)]
    arc = np.arange(f * k)
    s.append(arc // k)
    d.append(base + arc)
    return base + groups * (k + 1), np.concatenate(s).astype(np.int32), np.concatenate(d).astype(np.int32)


@pytest.mark.parametrize("mode", [dict(), dict(local_queue=0), dict(slice_arcs=16), dict(sampling=1, sample_threshold=8),
                                  dict(level_window=4), dict(sync_mode=3), dict(min_ctas=1, vertices_per_cta=1 << 30)],
                         ids=lambda m: ",".join(f"{a}={b}" for a, b in m.items()) or "default")
@pytest.mark.parametrize("k,f", [(1, 5), (7, 33), (8, 36), (31, 40), (32, 40), (33, 40), (64, 9), (65, 70)])
def test_all_arcs_cross(mode, k, f):
    n, s, d = cliques_on_peelers(k, f)
    off, adj = oracle.build_csr(n, s, d)
    with KCore(0, **mode) as h:
        assert_parity(h, n, off, adj)
        want = oracle.bz(n, off, adj)
        o, a = to_dev(off, adj)
        for kp in (k, k + 1):
            mask, size = h.core_mask(o, a, kp)
            np.testing.assert_array_equal(mask.cpu().numpy(), (want >= kp).astype(np.int32))
            assert int(size.cpu()[0]) == int((want >= kp).sum())
