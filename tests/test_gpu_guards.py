"""Inputs that break a counting call's contract in ways a kernel can see: the call reports an error
instead of a count, and the next call on the same workspace is exact."""
import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


def _dag(size, hubs, seed, n=50_000):
    """A DAG with `hubs` roots (lowest ids) that all have the same `size` out-neighbours, spread over
    the ids (some below a root's membership window), which form G(size, 0.4) among themselves."""
    rng = np.random.default_rng(seed)
    ids = np.sort(rng.choice(np.arange(hubs, n), size, replace=False))
    keep = np.triu(rng.random((size, size)) < 0.4, 1)
    rows = [ids] * hubs + [np.empty(0, ids.dtype)] * (n - hubs)
    for i in range(size):
        rows[ids[i]] = ids[keep[i]]
    return rows


def _count(gpu, rows, k, **tuned):
    import torch

    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    cols = np.concatenate(rows).astype(np.int32)
    d_off, d_cols = torch.from_numpy(off).cuda(), torch.from_numpy(cols).cuda()
    n, widest = len(rows), max(len(r) for r in rows)
    ws = gpu.alloc_workspace(n, 2 * len(cols), widest)
    return lambda: gpu.citron_count_ex(n, d_off, d_cols, k, ws, widest, **tuned)[0], d_cols


@pytest.mark.parametrize("k", [3, 4, 5, 6, 7])
@pytest.mark.parametrize("size", [33, 64, 129, 400])
@pytest.mark.parametrize("order", ["reversed", "first above the last", "two swapped"])
def test_unsorted_rows_are_refused(gpu, oracle_lib, size, k, order):
    """Rows of a bitmap-path root that are not ascending: their ids would fall outside the window of
    the ids below the last one."""
    import torch

    rows = _dag(size, 3, size)
    run, d_cols = _count(gpu, rows, k)
    good = d_cols.clone()
    row = rows[0].copy()
    if order == "reversed":
        row = row[::-1]
    elif order == "first above the last":
        row[0], row[-1] = row[-1], row[0]
    else:
        row[size // 2], row[size // 2 + 1] = row[size // 2 + 1], row[size // 2]
    d_cols[:size] = torch.from_numpy(row.astype(np.int32)).cuda()  # the first root's row
    with pytest.raises(gpu.CitronError) as e:
        run()
    assert e.value.name == "CITRON_E_INVALID"
    d_cols.copy_(good)
    off = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.uint64)
    assert run() == oracle_lib.count(off, np.concatenate(rows).astype(np.uint32), len(rows), k)


@pytest.mark.parametrize("k", [3, 5, 7])
@pytest.mark.parametrize("bound", [12, 16, 17, 31, 32, 33, 64, 96, 127, 128, 129, 160, 192, 193, 200, 300])
def test_understated_bound_of_a_batch(gpu, bound, k):
    """citron_count_batch sizes its launches by the caller's largest row (here 200): a bound whose
    launches leave a root out is reported, one that only rounds up to the row's capacity is not."""
    import torch
    from math import comb

    G = gpu.DeviceGraph(gg.complete(201))  # a relabelled DAG with rows of 200, 199, .., 0
    zeros = torch.zeros(G.n, dtype=torch.int32, device="cuda")
    ks = torch.tensor([k], dtype=torch.int32, device="cuda")
    counts = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = gpu.alloc_workspace(G.n, G.arcs, 300)

    def run(widest):
        gpu.citron_count_batch(G.n, G.dag_off, G.dag_cols, G.rank, zeros, ks, 1, 1 << k, widest, counts, ws)
        gpu.citron_workspace_status(ws)
        return int(counts.item())

    if bound >= 193:
        assert run(bound) == comb(201, k)
    else:
        with pytest.raises(gpu.CitronError) as e:
            run(bound)
        assert e.value.name == "CITRON_E_INVALID"
    assert run(200) == comb(201, k)
