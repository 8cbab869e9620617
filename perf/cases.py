"""What a program does with this framework, as cases that can be timed: `listed()` names them,
`prepare` makes a case's inputs on the GPU from a seed, `run` is one pass through the public entry
points, `work` is what that pass cannot do without.

The graphs are the ones of the repository's own workloads (Erdos-Renyi with a planted clique, R-MAT
with edge factor 16, Chung-Lu with exponent 2.1, batches of small graphs with 50 to 50,000 vertices),
drawn on the GPU so that a new input costs little.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2112_10913_gb300 as cg
from paper_2112_10913_gb300 import batch as cb
from paper_2112_10913_gb300.graphgen import Csr

DEV = "cuda"
RMAT = (0.57, 0.19, 0.19)  # quadrant probabilities a, b, c (d is the rest)


def listed():
    return [
        # one small graph from host memory, counted for three k: the shortest whole call a user
        # makes, where copies, launches and synchronisations are most of the time
        dict(name="host-er2000-k345", do="host", graph="er", n=2000, degree=20.0, ks="3,4,5"),
        # a mid-size graph from host memory, small k: upload, ordering, DAG and two counts
        dict(name="host-rmat18-k34", do="host", graph="rmat", scale=18, factor=16, ks="3,4"),
        # the ordering phase (degree ordering and the DAG relabelled by it) on the headline graph ...
        dict(name="order-rmat20", do="order", graph="rmat", scale=20, factor=16, layout="rank"),
        # ... and on the largest graph of the repository's configurations
        dict(name="order-chunglu4m", do="order", graph="chunglu", n=4_000_000, degree=30.0, layout="rank"),
        # the alternative ordering (core ordering) and its DAG
        dict(name="core-rmat20", do="core", graph="rmat", scale=20, factor=16),
        # the counting phase on the headline graph, DAG resident: k = 4, 5 and 6
        dict(name="count4-rmat20", do="count", graph="rmat", scale=20, factor=16, k=4, per_root=False),
        dict(name="count5-rmat20", do="count", graph="rmat", scale=20, factor=16, k=5, per_root=False),
        dict(name="count6-rmat20", do="count", graph="rmat", scale=20, factor=16, k=6, per_root=False),
        # a deep count on a smaller graph, with the count of every vertex asked for too
        dict(name="count8-rmat15", do="count", graph="rmat", scale=15, factor=16, k=8, per_root=True),
        # counting on the large skewed graph
        dict(name="count5-chunglu4m", do="count", graph="chunglu", n=4_000_000, degree=30.0, k=5, per_root=False),
        # a batch of many graphs of uneven sizes, each with its own k, replayed as one CUDA graph
        dict(name="batch-256", do="batch", graphs=256, n_min=50, n_max=50_000, deg_min=8.0, deg_max=64.0,
             k_min=3, k_max=7),
        # a serving loop's micro-batch: graphs that were not seen before are ordered, built and counted
        dict(name="micro-64", do="micro", graphs=64, n_min=50, n_max=50_000, deg_min=8.0, deg_max=64.0,
             k_min=3, k_max=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["host", "order", "core", "count", "count", "count", "batch", "micro"])
    if do == "host":
        if rng.random() < 0.5:
            return dict(do=do, graph="er", n=_log_int(rng, 60, 20_000), degree=round(rng.uniform(6, 40), 2),
                        ks=rng.choice(["3", "4", "3,4,5", "5,6"]))
        return dict(do=do, graph="rmat", scale=rng.randint(10, 18), factor=rng.randint(4, 16),
                    ks=rng.choice(["3", "4", "3,4", "4,5"]))
    if do == "order":
        layout = rng.choice(["rank", "rank", "ids"])
        if rng.random() < 0.5:
            return dict(do=do, graph="chunglu", n=_log_int(rng, 2000, 3_500_000), degree=round(rng.uniform(6, 30), 2),
                        layout=layout)
        return dict(do=do, graph="rmat", scale=rng.randint(11, 20), factor=rng.randint(4, 15), layout=layout)
    if do == "core":
        return dict(do=do, graph="rmat", scale=rng.randint(11, 19), factor=rng.randint(4, 16))
    if do == "count":
        per_root = rng.random() < 0.25
        if rng.random() < 0.3:
            n = _log_int(rng, 3000, 3_500_000)
            return dict(do=do, graph="chunglu", n=n, degree=round(rng.uniform(8, 30), 2),
                        k=rng.randint(3, 5) if n > 1_000_000 else rng.randint(3, 6), per_root=per_root)
        scale = rng.randint(12, 20)
        top = 5 if scale == 20 else 6 if scale >= 18 else 7 if scale >= 16 else 8 if scale >= 14 else 9
        return dict(do=do, graph="rmat", scale=scale, factor=rng.randint(4, 15), k=rng.randint(3, top),
                    per_root=per_root)
    top = rng.randint(4, 7) if do == "batch" else rng.randint(4, 6)
    return dict(do=do, graphs=_log_int(rng, 2, 200 if do == "batch" else 80), n_min=50,
                n_max=_log_int(rng, 500, 50_000), deg_min=8.0, deg_max=round(rng.uniform(12, 64), 1), k_min=3,
                k_max=top)


# ---------------------------------------------------------------------------------------------
# Inputs, drawn on the GPU


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _uniform(gen, count):
    return torch.rand(count, generator=gen, device=DEV)


def _rmat_pairs(gen, scale, count):
    a, b, c = RMAT
    src = torch.zeros(count, dtype=torch.int64, device=DEV)
    dst = torch.zeros(count, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        x = _uniform(gen, count)
        down = x >= a + b
        right = ((x >= a) & (x < a + b)) | (x >= a + b + c)
        src = 2 * src + down
        dst = 2 * dst + right
    return src, dst


def _csr(n, src, dst):
    """(off, cols) of the undirected graph of the pairs: loops and repeats dropped, both arcs of
    every edge, rows ascending; int64 and int32 tensors on the GPU."""
    keep = src != dst
    src, dst = src[keep], dst[keep]
    keys = torch.cat([src * n + dst, dst * n + src])
    keys = torch.unique_consecutive(torch.sort(keys).values)
    rows = torch.div(keys, n, rounding_mode="floor")
    cols = (keys - rows * n).to(torch.int32)
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return off, cols


def _planted(gen, n, size):
    v = torch.randperm(n, generator=gen, device=DEV)[:size]
    i, j = torch.triu_indices(size, size, 1, device=DEV)
    return v[i], v[j]


def _pairs(case):
    """Endpoint pairs that the case's graph is drawn from: its edges before repeats are dropped."""
    if case["graph"] == "rmat":
        return case["factor"] << case["scale"]
    return int(case["n"] * case["degree"] / 2) + 50 * 40 * 40


def _graph(case, seed):
    """(n, off, cols) of the case's graph."""
    gen = _gen(seed)
    if case["graph"] == "er":
        n = case["n"]
        count = int(n * case["degree"] / 2)
        src = torch.randint(n, (count,), generator=gen, device=DEV)
        dst = torch.randint(n, (count,), generator=gen, device=DEV)
        u, v = _planted(gen, n, 12)
        src, dst = torch.cat([src, u]), torch.cat([dst, v])
    elif case["graph"] == "rmat":
        n = 1 << case["scale"]
        src, dst = _rmat_pairs(gen, case["scale"], case["factor"] * n)
        perm = torch.randperm(n, generator=gen, device=DEV)
        src, dst = perm[src], perm[dst]
    else:  # Chung-Lu, exponent 2.1, expected degrees capped at n / 200, planted cliques of 20 to 40
        n = case["n"]
        w = torch.arange(1, n + 1, dtype=torch.float64, device=DEV) ** (-1.0 / 1.1)
        cap = max(50.0, n / 200)
        lo, hi = 0.0, 1.0
        while float(torch.clamp(w * hi, max=cap).mean()) < case["degree"]:
            hi *= 2
        for _ in range(40):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if float(torch.clamp(w * mid, max=cap).mean()) < case["degree"] else (lo, mid)
        # weights as whole numbers: a prefix sum of doubles on the GPU does not add in a fixed order,
        # and the same seed has to give the same graph
        cum = torch.cumsum((torch.clamp(w * hi, max=cap) * (1 << 20)).to(torch.int64), 0)
        count = int(n * case["degree"] / 2)
        ends = []
        for _ in range(2):
            x = torch.rand(count, generator=gen, device=DEV, dtype=torch.float64) * cum[-1].double()
            x = x.to(torch.int64)
            ends.append(torch.clamp(torch.searchsorted(cum, x, right=True), max=n - 1))
        perm = torch.randperm(n, generator=gen, device=DEV)
        src, dst = perm[ends[0]], perm[ends[1]]
        for i in range(max(1, min(50, n // 80_000))):
            u, v = _planted(gen, n, 20 + (7 * i + seed) % 21)
            src, dst = torch.cat([src, u]), torch.cat([dst, v])
    off, cols = _csr(n, src, dst)
    return n, off, cols


def _host(off, cols):
    return off.cpu().numpy().view(np.uint64), cols.cpu().numpy().view(np.uint32)


def _many(case, seed):
    """(graphs, ks): small graphs, half Erdos-Renyi and half R-MAT, sizes log-uniform.  The sizes are
    spread evenly over their range and the seed draws the edges, so that one seed's batch is about
    as much work as another's."""
    gen = _gen(seed)
    count, lo, hi = case["graphs"], math.log(case["n_min"]), math.log(case["n_max"])
    graphs, ks = [], []
    for i in range(count):
        at = (i + 0.5) / count
        n = int(round(math.exp(lo + at * (hi - lo))))
        part = (i * 0.6180339887498949) % 1.0
        degree = min(case["deg_min"] + part * (case["deg_max"] - case["deg_min"]), n - 1)
        ks.append(case["k_min"] + (i * 7 + 3) % (case["k_max"] - case["k_min"] + 1))
        pairs = int(round(n * degree / 2))
        if i % 2 == 0:
            src = torch.randint(n, (pairs,), generator=gen, device=DEV)
            dst = torch.randint(n, (pairs,), generator=gen, device=DEV)
        else:
            scale = max(1, math.ceil(math.log2(n)))
            src, dst = _rmat_pairs(gen, scale, int(pairs * 1.5))
            inside = (src < n) & (dst < n)
            src, dst = src[inside][:pairs], dst[inside][:pairs]
            perm = torch.randperm(n, generator=gen, device=DEV)
            src, dst = perm[src], perm[dst]
        off, cols = _host(*_csr(n, src, dst))
        graphs.append(Csr(n=n, off=off, cols=cols))
    return graphs, ks


# ---------------------------------------------------------------------------------------------
# States and passes


def prepare(case, seed):
    do = case["do"]
    if do == "batch":
        graphs, ks = _many(case, seed)
        counter = cb.BatchCounter(graphs, ks, device=DEV)
        counter.capture()
        return dict(case=case, counter=counter)
    if do == "micro":
        graphs, ks = _many(case, seed)
        union, group = cb.union_csr(graphs)
        n, arcs = union.n, union.arcs
        kmask = 0
        for k in ks:
            kmask |= 1 << k
        # a serving slot's buffers are sized once, for its largest micro-batch
        return dict(case=case, n=n, ngroups=len(ks), kmask=kmask,
                    off=torch.from_numpy(union.off.view(np.int64)).to(DEV),
                    cols=torch.from_numpy(union.cols.view(np.int32)).to(DEV),
                    group=torch.from_numpy(group.view(np.int32)).to(DEV),
                    group_k=torch.tensor(ks, dtype=torch.int32, device=DEV),
                    rank=torch.empty(n, dtype=torch.int32, device=DEV),
                    dag_off=torch.empty(n + 1, dtype=torch.int64, device=DEV),
                    dag_cols=torch.empty(max(1, arcs // 2), dtype=torch.int32, device=DEV),
                    counts=torch.zeros(len(ks), dtype=torch.int64, device=DEV),
                    ws=cg.alloc_workspace(n, arcs, 4096, device=DEV))
    n, off, cols = _graph(case, seed)
    arcs = int(cols.numel())
    if do == "host":
        h_off, h_cols = off.cpu().pin_memory(), cols.cpu().pin_memory()
        return dict(case=case, n=n, off=h_off, cols=h_cols, ks=[int(k) for k in case["ks"].split(",")],
                    buf=torch.empty(cg.citron_host_buffer_bytes(n, arcs), dtype=torch.uint8, device=DEV),
                    ws=cg.alloc_workspace(n, arcs, 4096, device=DEV))
    if do == "count":
        h_off, h_cols = _host(off, cols)
        graph = cg.DeviceGraph(Csr(n=n, off=h_off, cols=h_cols), device=DEV)
        per_root = torch.zeros(n, dtype=torch.int64, device=DEV) if case["per_root"] else None
        return dict(case=case, graph=graph, per_root=per_root)
    # room for every drawn pair, so that the buffer does not depend on how many of them repeat
    return dict(case=case, n=n, off=off, cols=cols, rank=torch.empty(n, dtype=torch.int32, device=DEV),
                dag_off=torch.empty(n + 1, dtype=torch.int64, device=DEV),
                dag_cols=torch.zeros(_pairs(case), dtype=torch.int32, device=DEV),
                ws=cg.alloc_workspace(n, arcs, 1, device=DEV))


def run(s):
    case = s["case"]
    do = case["do"]
    if do == "host":
        return cg.citron_count_host(s["n"], s["off"], s["cols"], s["ks"], s["buf"], s["ws"])
    if do == "count":
        total = s["graph"].count(case["k"], per_root=s["per_root"])
        return [total] if s["per_root"] is None else [total, s["per_root"]]
    if do == "batch":
        s["counter"].replay()
        return s["counter"].counts
    if do == "micro":
        cg.citron_order_grouped(s["n"], s["off"], s["group"], s["ngroups"], s["rank"], None, s["ws"])
        widest = cg.citron_build_dag(s["n"], s["off"], s["cols"], s["rank"], s["dag_off"], s["dag_cols"], s["ws"])
        cg.citron_count_batch(s["n"], s["dag_off"], s["dag_cols"], s["rank"], s["group"], s["group_k"],
                              s["ngroups"], s["kmask"], widest, s["counts"], s["ws"])
        cg.citron_workspace_status(s["ws"])
        return s["counts"]
    rank = s["rank"]
    extra = []
    if do == "core":
        extra = list(cg.citron_core_order(s["n"], s["off"], s["cols"], rank, None, s["ws"]))
    elif case["layout"] == "rank":
        cg.citron_order(s["n"], s["off"], rank, None, s["ws"])
    else:
        rank = None  # the paper's own layout: vertex ids kept
    widest = cg.citron_build_dag(s["n"], s["off"], s["cols"], rank, s["dag_off"], s["dag_cols"], s["ws"])
    return [widest, s["dag_off"], s["dag_cols"]] + ([] if rank is None else [rank]) + extra


def work(case):
    """Bytes: the input read once and the output written once.  The intersections of a count have no
    lower bound that is known in advance, so a count's work is the reading of its DAG."""
    do = case["do"]
    if do in ("batch", "micro"):
        lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
        n = arcs = 0.0
        for i in range(case["graphs"]):
            size = math.exp(lo + (i + 0.5) / case["graphs"] * (hi - lo))
            part = (i * 0.6180339887498949) % 1.0
            n += size
            arcs += size * min(case["deg_min"] + part * (case["deg_max"] - case["deg_min"]), size - 1)
    else:
        n = float(1 << case["scale"]) if case["graph"] == "rmat" else float(case["n"])
        arcs = 2.0 * n * case["factor"] if case["graph"] == "rmat" else n * case["degree"]
    graph, dag = 8 * (n + 1) + 4 * arcs, 8 * (n + 1) + 2 * arcs
    if do == "host":  # read once by the copy; the DAG need not exist
        nbytes = graph
    elif do == "batch":
        nbytes = dag + 8 * case["graphs"]
    elif do == "micro":
        nbytes = graph + 8 * case["graphs"]
    elif do == "count":
        nbytes = dag + (8 * n if case["per_root"] else 8)
    else:
        nbytes = graph + dag + (0 if case.get("layout") == "ids" else 4 * n)
    return {"bytes": nbytes, "flops": 0.0}


def exact(case, seed):
    """The degree ordering and its DAG in plain torch integers; every output here is a whole number,
    and counts and the core ordering have no short plain form."""
    if case["do"] != "order":
        return None
    n, off, cols = _graph(case, seed)
    degree = off[1:] - off[:-1]
    ids = torch.arange(n, device=DEV)
    rank = torch.empty(n, dtype=torch.int64, device=DEV)
    rank[torch.argsort(degree, stable=True)] = ids
    src, dst = torch.repeat_interleave(ids, degree), cols.long()
    keep = rank[src] < rank[dst]
    src, dst = src[keep], dst[keep]
    if case["layout"] == "rank":
        keys = torch.sort(rank[src] * n + rank[dst]).values
        src, dst = torch.div(keys, n, rounding_mode="floor"), keys % n
    count = torch.bincount(src, minlength=n)
    dag_off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    dag_off[1:] = torch.cumsum(count, 0)
    dag_cols = torch.zeros(_pairs(case), dtype=torch.int32, device=DEV)
    dag_cols[: dst.numel()] = dst.to(torch.int32)
    out = [int(count.max()), dag_off, dag_cols]
    return out + ([rank.to(torch.int32)] if case["layout"] == "rank" else [])
