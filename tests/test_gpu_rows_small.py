"""Rows of warp-register roots by scanning the members' lists and by looking up pairs: lists shorter and
longer than one load, few and many members, DAGs that keep ids, against the CPU oracle."""
import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members", [2, 3, 8, 11, 12, 31, 32])
@pytest.mark.parametrize("tail", [0, 20, 33, 70, 200])
def test_lists_and_pairs(gpu, oracle_lib, members, tail):
    """Roots whose `members` out-neighbours form G(members, 0.6) and have `tail` more neighbours each,
    above or below the members' ids."""
    rng = np.random.default_rng(members * 1000 + tail)
    copies = 40
    i, j = np.triu_indices(members, 1)
    shift = np.arange(copies)[:, None] * (members + 1)
    keep = rng.random((copies, i.size)) < 0.6
    base = copies * (members + 1)
    n = base + 600
    hub = np.repeat(np.arange(copies) * (members + 1) + members, members)
    mem = (np.arange(members) + shift).ravel()
    ends = base + rng.integers(0, 600, (mem.size, tail))
    src = np.concatenate([(i + shift)[keep], hub, np.repeat(mem, tail)])
    dst = np.concatenate([(j + shift)[keep], mem, ends.ravel()])
    for perm in (np.arange(n), np.arange(n)[::-1].copy(), rng.permutation(n)):
        g = gg.csr_from_edges(n, perm[src], perm[dst])
        for relabel in (True, False):
            G = gpu.DeviceGraph(g, relabel=relabel)
            off, cols = G.dag_numpy()
            for k in (3, 4, 6):
                assert G.count(k) == oracle_lib.count(off, cols, g.n, k)
