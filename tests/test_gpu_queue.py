"""The bitmap path's queue in one launch and in two (few or many roots up to the line between them, DAGs
that keep ids, no re-encoding, capped launches), from single counts and from batches, against the
CPU oracle."""
import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def _copies(size, copies, p, seed, wide=170, q=0.5):
    """`copies` disjoint random graphs of `size` vertices and one of `wide` beside them."""
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(size, 1)
    shift = np.arange(copies)[:, None] * size
    keep = rng.random((copies, i.size)) < p
    base = size * copies
    bi, bj = np.triu_indices(wide, 1)
    big = rng.random(bi.size) < q
    src = np.concatenate([(i + shift)[keep], bi[big] + base])
    dst = np.concatenate([(j + shift)[keep], bj[big] + base])
    return gg.csr_from_edges(base + wide, src, dst)


# about 35 roots a copy on the bitmap path: 70, 2,450 (around four per 8-warp block of 152 SMs) and 6,000
@pytest.mark.parametrize("copies", [2, 70, 72, 170])
@pytest.mark.parametrize("k", [3, 5, 6])
@pytest.mark.parametrize("relabel", [True, False])
def test_one_launch_or_two(gpu, oracle_lib, copies, k, relabel):
    import torch

    g = _copies(72, copies, 0.93, copies)
    G = gpu.DeviceGraph(g, relabel=relabel)
    off, cols = G.dag_numpy()
    want = oracle_lib.count(off, cols, g.n, k)
    assert G.count(k) == want
    assert G.count(k, compact_max=1) == want
    assert G.count(k, max_blocks=5) == want
    zeros = torch.zeros(g.n, dtype=torch.int32, device="cuda")
    ks = torch.tensor([k], dtype=torch.int32, device="cuda")
    counts = torch.zeros(1, dtype=torch.int64, device="cuda")
    for opts in (None, gpu.CountOpts(0, 0, 0, 0, 1, 0, None, 0), gpu.CountOpts(0, 0, 0, 0, 0, 7, None, 0)):
        gpu.citron_count_batch(g.n, G.dag_off, G.dag_cols, G.rank, zeros, ks, 1, 1 << k, G.max_outdeg, counts,
                               G.ws, None, opts)
        gpu.citron_workspace_status(G.ws)
        assert int(counts.item()) == want


def test_busy_time_covers_both_launches(gpu):
    """busy_ms spans the launch of large blocks (few roots here) and the one of small blocks (12,000 roots)."""
    g = _copies(72, 340, 0.93, 5, wide=260, q=0.7)
    G = gpu.DeviceGraph(g)
    for _ in range(2):  # (the first call pays for loading the kernels)
        _, o = gpu.citron_count_ex(G.n, G.dag_off, G.dag_cols, 5, G.ws, G.max_outdeg, time_kernels=True, balance=True)
    assert G.max_outdeg > 128 and o.kernel_ms[1] > 0.1
    assert 0.7 * o.kernel_ms[1] < o.busy_ms[0] <= 1.05 * o.kernel_ms[1] + 0.02
    assert 0 <= o.busy_ms[1] <= o.busy_ms[0]
