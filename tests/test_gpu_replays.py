"""Training calls of few chunks, repeated: when their launches are captured into
a graph, and that a replay gives what direct launches give, bit for bit, with
everything changed that a captured graph does not hold."""
import json

import numpy as np
import pytest

from paper_2604_09419_gb300 import inputs as I
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

DIM, K, BATCH = 16, 5, 256


def captures(run, tmp_path):
    """The graphs instantiated and launched by run()."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(3):  # (the first session of a process may record nothing)
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
            run()
            torch.cuda.synchronize()
        p.export_chrome_trace(str(tmp_path / "trace.json"))
        names = [e["name"] for e in json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
                 if e.get("cat") == "cuda_runtime"]
        if names:
            return sum("GraphInstantiate" in n for n in names), sum("GraphLaunch" in n for n in names)
    pytest.skip("the profiler records no calls here")


def test_short_runs_of_equal_calls_are_not_captured(tmp_path):
    from paper_2604_09419_gb300 import line as L
    g = G.graph("tiny")
    ctx = G.context()
    G.upload(ctx, g)
    ctx.init_embeddings(2, DIM, L.DTYPE_F32, seed=1)

    def call(lam):
        ctx.train_steps(2, DIM, K, 20_000, 7, batch=BATCH, lam=lam)

    def pairs():
        for lam in (0.0, 0.0, 1e-3, 1e-3) * 3:
            call(lam)

    # two calls of one kind after two of another: each capture would be
    # thrown away before it is replayed
    assert captures(pairs, tmp_path) == (0, 0)

    def many():
        for _ in range(12):
            call(1e-2)

    # the same call again and again is captured once, and replayed
    made, launched = captures(many, tmp_path)
    assert made <= 1 and launched >= 3, (made, launched)
    ctx.close()


# one ragged chunk; one full chunk; a full chunk and a ragged one (chunks of 40 batches)
@pytest.mark.parametrize("samples", [39 * BATCH + 77, 40 * BATCH, 40 * BATCH + 1000])
@pytest.mark.parametrize("both", [False, True])
def test_replays_equal_direct_launches(samples, both):
    from paper_2604_09419_gb300 import line as L
    g = G.graph("tiny")
    other = I.Graph(g.n_nodes, g.src, np.roll(g.dst, 1), g.w[::-1].copy(), False)  # the same sizes
    ctxs = [G.context(), G.context()]
    orders = (1, 2) if both else (2,)

    def each(f):
        for c, graph in zip(ctxs, (1, 0)):
            f(c, graph)

    def tables(c):
        return [t for o in orders for t in G.tables(c, g, o, DIM) if t is not None]

    def start(dtype):
        each(lambda c, _: [c.init_embeddings(o, DIM, dtype, seed=3) for o in orders])

    each(lambda c, _: G.upload(c, g))
    start(L.DTYPE_F32)
    offset = 0
    for k in range(30):
        if k == 13:
            each(lambda c, _: G.upload(c, other))
        if k == 18:  # tables of another type, in the same memory
            start(L.DTYPE_BF16)

        def call(c, graph):
            kw = dict(lr0=0.01 + 0.001 * k, batch=BATCH, sample_offset=offset, chunk_batches=40, graph=graph)
            if both:
                c.train_orders(DIM, K, samples, 5 + k, **kw)
            else:
                c.train_steps(2, DIM, K, samples, 5 + k, **kw)

        each(call)
        offset += -(-samples // BATCH) * BATCH
        for a, b in zip(*(tables(c) for c in ctxs)):
            assert np.array_equal(a, b), k
    each(lambda c, _: c.close())
