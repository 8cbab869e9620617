"""The local subgraph's rows (k_count_mid, k_count_small): ids inside and below the membership
window of a root, lists longer than one step of the scan, and root sizes at the edges of the paths
and of the two launches, against the CPU oracle."""
import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def spread(n, core, span, seed):
    """A random graph on `core` vertices whose ids lie `span` apart on average (some neighbours of a
    root are then far below its largest one), with a tail of filler edges up to n."""
    rng = np.random.default_rng(seed)
    ids = np.sort(rng.choice(min(n, core * span), core, replace=False))
    i, j = np.triu_indices(core, 1)
    keep = rng.random(i.size) < 0.5
    fill = rng.integers(0, n, (2, 4 * n // 10))
    return gg.csr_from_edges(n, np.concatenate([ids[i[keep]], fill[0]]), np.concatenate([ids[j[keep]], fill[1]]))


@pytest.mark.parametrize("core", [20, 32, 33, 64, 127, 128, 129, 160, 300])
@pytest.mark.parametrize("span", [1, 100, 400])
def test_rows_inside_and_below_the_window(gpu, oracle_lib, core, span):
    import paper_2112_10913_gb300 as cg

    g = spread(150_000, core, span, core * 1000 + span)
    rank = np.arange(g.n, dtype=np.uint32)  # ids are ranks: the window sees the spread as it is
    off, cols = oracle_lib.dag_by_rank(g.off, g.cols, g.n, rank, relabel=True)
    G = cg.DeviceGraph(g, rank=rank)
    for k in (3, 4, 5):
        want = oracle_lib.count(off, cols, g.n, k)
        assert G.count(k) == want
        assert G.count(k, small_max=1) == want
        assert G.count(k, warps_per_cta=1) == want
    H = cg.DeviceGraph(g, relabel=False)  # rows that are not upper-triangular
    assert H.count(4) == oracle_lib.count(off, cols, g.n, 4)
