"""max_blocks leaves SMs to other streams: while a capped count runs, a count on another stream that
needs whole SMs (blocks of 32 warps) starts and ends."""
import time

import numpy as np
import pytest

from paper_2112_10913_gb300 import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warps", [32, 16])
def test_a_capped_count_leaves_whole_sms(gpu, warps):
    import torch

    rng = np.random.default_rng(7)
    size, copies, k = 120, 1500, 6
    i, j = np.triu_indices(size, 1)
    shift = np.arange(copies)[:, None] * size
    keep = rng.random((copies, i.size)) < 0.85  # every root of at most 119 out-neighbours
    heavy = gpu.DeviceGraph(gg.csr_from_edges(size * copies, (i + shift)[keep], (j + shift)[keep]))
    light = gpu.DeviceGraph(gg.complete(200))
    want_light, want_heavy = light.count(4), heavy.count(k)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    opts = gpu.CountOpts(0, 0, warps, 0, 0, sms * 3 // 4, None, 0)
    group = torch.zeros(heavy.n, dtype=torch.int32, device="cuda")
    ks = torch.tensor([k], dtype=torch.int32, device="cuda")
    counts = torch.zeros(1, dtype=torch.int64, device="cuda")
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    started, ended = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    started.record(a)
    gpu.citron_count_batch(heavy.n, heavy.dag_off, heavy.dag_cols, heavy.rank, group, ks, 1, 1 << k,
                           heavy.max_outdeg, counts, heavy.ws, a, opts)
    ended.record(a)
    waits = []
    time.sleep(0.002)
    while not ended.query():
        t = time.perf_counter()
        assert light.count(4, stream=b) == want_light
        waits.append(time.perf_counter() - t)
    torch.cuda.synchronize()
    gpu.citron_workspace_status(heavy.ws, a)
    assert int(counts.item()) == want_heavy
    whole = started.elapsed_time(ended) * 1e-3
    assert whole > 0.01, "the capped count is too short to tell"
    # about 0.15 ms each; one that waits for a block of the capped count to leave its SM takes most of that
    # count's time (the last one may meet the end of it)
    assert max(waits[:-1], default=whole) < whole / 4, waits
