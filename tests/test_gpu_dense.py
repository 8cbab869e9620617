"""Dense candidate sets counted on their complement (csrc/dense.cuh): one edge task whose set has
exactly s members, at the sizes where the layout changes (words of 32, the 128 members of one warp,
the chunks of wide sets), from sparse to complete, against the CPU oracle."""
import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def one_set(s, p, seed, hubs=0):
    """Vertices 0 and 1 adjacent to every vertex; the others form G(s, p), the first `hubs` of them
    with a third of those edges only (a skewed complement)."""
    rng = np.random.default_rng(seed)
    i, j = np.triu_indices(s, 1)
    keep = rng.random(i.size) < np.where((i < hubs) | (j < hubs), p / 3, p)
    src = np.concatenate([[0], np.zeros(s, int), np.ones(s, int), i[keep] + 2])
    dst = np.concatenate([[1], np.arange(s) + 2, np.arange(s) + 2, j[keep] + 2])
    return gg.csr_from_edges(s + 2, src, dst, name=f"set{s}-{p}-{hubs}")


CASES = [(s, p, 0, k) for s in (31, 32, 33, 64, 65, 96, 127, 128) for p in (0.3, 0.6, 0.93) for k in (5, 6)]
CASES += [(s, p, 0, k) for s in (129, 160, 193) for p in (0.3, 0.55, 0.8) for k in (5, 6)]
CASES += [(40, 0.9, 0, 7), (96, 0.7, 0, 7), (128, 0.6, 0, 7), (129, 0.7, 0, 7), (150, 0.6, 0, 7)]
CASES += [(s, 0.95, 24, k) for s in (33, 64, 128) for k in (5, 6)]
CASES += [(140, 0.9, 24, 6), (256, 0.8, 24, 5), (257, 0.75, 40, 6), (50, 0.95, 10, 8), (140, 0.6, 10, 8)]
# subsets packed again on the way down
CASES += [(45, 0.9, 0, 8), (64, 0.85, 6, 8), (65, 0.8, 0, 8), (100, 0.75, 10, 8), (128, 0.62, 0, 8), (66, 0.75, 0, 9)]
CASES += [(40, 1.0, 0, 9), (100, 1.0, 0, 6), (140, 1.0, 0, 5)]
# a third and more chunks, members of more than 255 missing neighbours, more than 128 of them
CASES += [(300, 0.7, 40, 6), (385, 0.52, 0, 6), (530, 0.5, 0, 6), (520, 0.55, 0, 5)]


@pytest.mark.parametrize("s,p,hubs,k", CASES)
def test_one_dense_set(gpu, oracle_lib, s, p, hubs, k):
    import paper_2112_10913_gb300 as cg

    g = one_set(s, p, s * 7 + k, hubs)
    rank = np.arange(g.n, dtype=np.uint32)
    off, cols = oracle_lib.dag_by_rank(g.off, g.cols, g.n, rank, relabel=True)
    want = oracle_lib.count(off, cols, g.n, k)
    G = cg.DeviceGraph(g, rank=rank)
    assert G.count(k) == want
    # few warps per block (groups of warps at the block's edge) and every root split
    assert G.count(k, warps_per_cta=3) == want
    assert G.count(k, split_min=33, small_max=1) == want
    if k <= 6 and s <= 200:
        total, per_arc = G.count_per_arc(k)
        assert total == want and int(per_arc.sum()) == want


@pytest.mark.parametrize("s,p", [(140, 0.6), (260, 0.4), (700, 0.15)])
@pytest.mark.parametrize("k", [6, 7])
@pytest.mark.parametrize("plan", [dict(relabel=False), dict(compact_max=1), dict(warps_per_cta=2)])
def test_heavy_roots_cut_by_member(gpu, oracle_lib, s, p, k, plan):
    """Heavy roots whose rows of more than 128 members are not re-encoded: a DAG that keeps ids, no
    re-encoding, and rows too wide for the buffers of a block of two warps; split and whole."""
    import paper_2112_10913_gb300 as cg

    if k == 7 and s == 140:
        s = 132  # (a shorter oracle run)
    g = one_set(s, p, s + k)
    relabel = plan.get("relabel", True)
    tuned = {a: b for a, b in plan.items() if a != "relabel"}
    rank = np.arange(g.n, dtype=np.uint32)
    G = cg.DeviceGraph(g, rank=rank) if relabel else cg.DeviceGraph(g, relabel=False)
    off, cols = G.dag_numpy()
    want = oracle_lib.count(off, cols, g.n, k)
    for split in (33, 129, 0, 1):
        assert G.count(k, split_min=split, **tuned) == want
    total, per_arc = G.count_per_arc(k, split_min=33, **tuned)
    assert total == want and int(per_arc.sum()) == want


# Sets around the line between the two sides: one warp's (k = 5, 6, 8), small ones of deep walks, wide
# ones on packed rows of 5 and 6 words, on the root-wide bitmap and by groups
LINE = [(s, p, k) for s in (31, 32, 33, 96, 97, 128) for p, k in ((0.56, 5), (0.56, 6), (0.56, 8), (0.69, 8))]
LINE += [(s, p, 5) for s in (129, 160, 161, 192) for p in (0.45, 0.78)]
LINE += [(s, p, 5) for s in (193, 400) for p in (0.5, 0.66)]
LINE += [(s, p, 6) for s in (129, 300) for p in (0.4, 0.57)]
LINE += [(s, p, 7) for s in (129, 170) for p in (0.5, 0.73)]


@pytest.mark.parametrize("s,p,k", LINE)
def test_sets_around_the_line(gpu, oracle_lib, s, p, k):
    import paper_2112_10913_gb300 as cg

    g = one_set(s, p, s * 11 + k)
    rank = np.arange(g.n, dtype=np.uint32)
    off, cols = oracle_lib.dag_by_rank(g.off, g.cols, g.n, rank, relabel=True)
    want = oracle_lib.count(off, cols, g.n, k)
    G = cg.DeviceGraph(g, rank=rank)
    assert G.count(k) == want
    assert G.count(k, warps_per_cta=3) == want
    assert G.count(k, split_min=33) == want
    if k <= 6:
        total, per_arc = G.count_per_arc(k)
        assert total == want and int(per_arc.sum()) == want


def test_nested_wide_set_beyond_the_planes(gpu):
    """k = 7: subsets of a wide set with more than 128 members of complement degree above 128 (an
    independent part of 135 at the end of the order), counted one level further down."""
    from math import comb

    import paper_2112_10913_gb300 as cg

    clique, part = 137, 135
    i, j = np.triu_indices(clique, 1)
    src = np.concatenate([i, np.repeat(np.arange(clique), part)])
    dst = np.concatenate([j, np.tile(np.arange(part) + clique, clique)])
    g = gg.csr_from_edges(clique + part, src, dst)
    G = cg.DeviceGraph(g, rank=np.arange(g.n, dtype=np.uint32))
    want = comb(clique, 7) + part * comb(clique, 6)
    assert G.count(7) == want
    assert G.count(7, split_min=129) == want


@pytest.mark.parametrize("parts,k", [([7] * 10, 10), ([6] * 11, 11), ([16] * 4 + [1] * 8, 12)])
def test_deep_walks_pack_their_subsets(gpu, parts, k):
    """Two vertices joined to a complete multipartite graph of 66 to 72: sets of four words whose subsets
    are packed to two and to one on the way down."""
    import paper_2112_10913_gb300 as cg

    n = sum(parts)
    part = np.repeat(np.arange(len(parts)), parts)
    i, j = np.triu_indices(n, 1)
    keep = part[i] != part[j]
    src = np.concatenate([[0], np.zeros(n, int), np.ones(n, int), i[keep] + 2])
    dst = np.concatenate([[1], np.arange(n) + 2, np.arange(n) + 2, j[keep] + 2])
    g = gg.csr_from_edges(n + 2, src, dst)
    G = cg.DeviceGraph(g, rank=np.arange(g.n, dtype=np.uint32))
    e = [1] + [0] * k  # elementary symmetric polynomials of the part sizes
    for q in parts:
        for m in range(k, 0, -1):
            e[m] += e[m - 1] * q
    assert G.count(k) == e[k] + 2 * e[k - 1] + e[k - 2]
