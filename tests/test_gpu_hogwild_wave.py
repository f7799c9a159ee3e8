"""The number of samples that the Hogwild schedule has in flight by default, and
at most, at every row width and type: it is part of the schedule's results, so
it is stated and not left to a kernel's registers.  Read from the launches."""
import json

import numpy as np
import pytest

from paper_2604_09419_gb300 import inputs as I
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def blocks_launched(run, tmp_path):
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):  # (the first session of a process may record no kernels)
        torch.cuda.synchronize()
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
            run()
            torch.cuda.synchronize()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        events = json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
        found = {(tuple(e["args"]["grid"]), tuple(e["args"]["block"])) for e in events
                 if e.get("cat") == "kernel" and "k_hogwild" in e["name"]}
        if found:
            break
    else:
        pytest.skip("the profiler records no kernels here")
    (grid, block), = found
    assert block == (128, 1, 1)
    return grid[0]


# K = 5 leaves shared memory for every wave; tables of 32 MB and more take the
# copying form at dim 64 and 128; K = 32 at dim 128 leaves room for three
# blocks of 70,720 bytes
@pytest.mark.parametrize("dim,dtype,nodes,K,per_sm", [
    (16, 0, 100, 5, 8), (32, 1, 100, 5, 8), (64, 0, 131071, 5, 8), (64, 0, 131072, 5, 8), (64, 1, 131072, 5, 8),
    (128, 0, 65535, 5, 8), (128, 0, 65536, 5, 8), (128, 1, 65536, 5, 8), (128, 0, 65536, 32, 3),
    (256, 0, 32768, 5, 5), (256, 1, 65536, 5, 4),
])
def test_samples_in_flight(dim, dtype, nodes, K, per_sm, tmp_path):
    import torch

    from paper_2604_09419_gb300 import line as L
    g = I.canonicalize(nodes, np.zeros(40, np.int64), nodes - 1 - np.arange(40), None, symmetrize=True)
    ctx = G.context()
    G.upload(ctx, g)
    ctx.init_embeddings(2, dim, dtype, seed=1)
    n, sms = 1 << 17, torch.cuda.get_device_properties(0).multi_processor_count
    for workers in (0, 100_000):
        got = blocks_launched(lambda: ctx.train_steps(2, dim, K, n, 5, batch=64, mode=L.MODE_HOGWILD,
                                                      hogwild_workers=workers), tmp_path)
        assert got == per_sm * sms, (got, per_sm * sms)
    ctx.close()
