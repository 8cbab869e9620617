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


@pytest.mark.parametrize("arcs", [2, 64, 510, 512, 514, 1024, 1536, 4094])
@pytest.mark.parametrize("width", [1, 31, 32, 33, 255, 600])
def test_relabelled_dag_at_chunk_edges(gpu, oracle_lib, arcs, width):
    """Rows of about `width` arcs beside empty rows, with the arcs ending at and around the 512-arc chunks."""
    import paper_2112_10913_gb300 as cg

    rng = np.random.default_rng(arcs * 7 + width)
    m = arcs // 2
    hubs = -(-m // width)
    src = np.repeat(np.arange(hubs) * 3, width)[:m]  # two empty rows between the hubs
    dst = 3 * hubs + np.concatenate([rng.permutation(max(width, 8))[:width] for _ in range(hubs)])[:m]
    g = gg.csr_from_edges(3 * hubs + max(width, 8) + 5, src, dst)
    for rank in (oracle_lib.degree_rank(g.off, g.n), rng.permutation(g.n).astype(np.uint32)):
        off, cols = oracle_lib.dag_by_rank(g.off, g.cols, g.n, rank, relabel=True)
        goff, gcols = cg.DeviceGraph(g, rank=rank).dag_numpy()
        assert np.array_equal(goff, off) and np.array_equal(gcols, cols)
