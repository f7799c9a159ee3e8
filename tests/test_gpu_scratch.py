"""Scratch that the evaluation calls keep is given back when a later call of the
context needs the memory: training on a device that is all but full."""
import numpy as np
import pytest

from tests import gpu_util as G

pytestmark = pytest.mark.gpu

MB = 1 << 20
DIM, K, BATCH, SAMPLES = 256, 5, 8192, 1 << 18


def free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def prepared():
    from paper_2604_09419_gb300 import line as L
    ctx = G.context()
    G.upload(ctx, G.graph("rmat14"))
    ctx.init_embeddings(2, DIM, L.DTYPE_F32, seed=1)
    return ctx


def train(ctx):
    ctx.train_steps(2, DIM, K, SAMPLES, 5, batch=BATCH, graph=0)


def evaluate(ctx, m):
    import torch
    rng = np.random.default_rng(1)
    a, b = (torch.from_numpy(rng.integers(0, 1 << 14, m).astype(np.int32)).cuda() for _ in range(2))
    return ctx.eval_auc(2, a, b, b, a)


def test_training_takes_back_the_scratch_of_an_evaluation():
    import torch

    ctx = prepared()
    evaluate(ctx, 1000)  # (module loading)
    before = free()
    train(ctx)
    need = before - free()
    U, C = G.tables(ctx, G.graph("rmat14"), 2, DIM)
    ctx.close()
    ctx = prepared()
    torch.cuda.empty_cache()
    before = free()
    want = evaluate(ctx, 6 << 20)
    torch.cuda.empty_cache()
    kept = before - free()
    assert need > 64 * MB and kept > 64 * MB, (need, kept)
    # room for the training call's buffers only with half of the scratch
    filler = torch.empty(free() - need + kept // 2, dtype=torch.uint8, device="cuda")
    try:
        train(ctx)
        del filler
        got = G.tables(ctx, G.graph("rmat14"), 2, DIM)
        assert np.array_equal(got[0], U) and np.array_equal(got[1], C)
        # and an evaluation afterwards takes scratch again
        ctx.eval_loss(2, K, 3, 1000)
        assert want[0] > 0.0
    finally:
        filler = None
        torch.cuda.empty_cache()
        ctx.close()
