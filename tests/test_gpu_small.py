"""Roots of the warp-register path at k >= 7: dense ones are counted on their complement, the others
enumerated (sizes around 16 and 32, sides of the line, DAGs that keep ids, no re-encoding), against
the CPU oracle."""
import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def _sets(size, copies, p, seed):
    """`copies` roots whose `size` out-neighbours form G(size, p)."""
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(size, 1)
    shift = np.arange(copies)[:, None] * (size + 1)
    keep = rng.random((copies, i.size)) < p
    hub = np.repeat(np.arange(copies) * (size + 1) + size, size)
    return gg.csr_from_edges(copies * (size + 1), np.concatenate([(i + shift)[keep], hub]),
                             np.concatenate([(j + shift)[keep], (np.arange(size) + shift).ravel()]))


@pytest.mark.parametrize("size", [15, 16, 17, 24, 31, 32])
@pytest.mark.parametrize("p", [0.4, 0.69, 0.9, 1.0])
@pytest.mark.parametrize("k", [7, 8, 10, 12])
def test_small_roots_of_deep_counts(gpu, oracle_lib, size, p, k):
    import torch

    g = _sets(size, 9, p, size * 100 + k)
    for relabel in (True, False):
        G = gpu.DeviceGraph(g, relabel=relabel)
        off, cols = G.dag_numpy()
        want = oracle_lib.count(off, cols, g.n, k)
        per_root = torch.zeros(g.n, dtype=torch.int64, device="cuda")
        assert G.count(k, per_root=per_root) == want
        assert int(per_root.sum().item()) == want
        assert G.count(k, compact_max=1) == want
        assert G.count(k, small_max=16) == want
