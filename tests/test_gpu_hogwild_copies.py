"""Hogwild on both sides of the size from which the context rows of a sample
are copied asynchronously (FP32 tables of 32 MB), and over batches of rows
that pass through registers: one worker, which is the sequential per-pair SGD,
against the FP64 oracle.  The nodes beyond the star are isolated, so a sample
meets the same row in several slots, in order 1 its own source row too."""
import numpy as np
import pytest

import oracle as O
from paper_2604_09419_gb300 import inputs as I
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

TOL = 1e-5  # the bound of the one-worker runs: FP32 updates of at most 1e4 samples, values below 1


@pytest.mark.parametrize("dim,nodes,order,K", [
    (128, 65535, 2, 5), (128, 65536, 2, 5), (128, 65536, 1, 5), (128, 65536, 2, 0), (128, 65536, 1, 32),
    (64, 131071, 1, 10), (64, 131072, 1, 10), (64, 131072, 2, 17), (256, 32768, 2, 6),
])
def test_rows_copied_or_through_registers(dim, nodes, order, K):
    from paper_2604_09419_gb300 import line as L
    g = I.canonicalize(nodes, np.zeros(40, np.int64), nodes - 1 - np.arange(40), None, symmetrize=True)
    ctx = G.context()
    G.upload(ctx, g)
    ctx.init_embeddings(order, dim, L.DTYPE_F32, seed=1)
    n = 1501
    ctx.train_steps(order, dim, K, n, 5, batch=64, lam=1e-3, mode=L.MODE_HOGWILD, hogwild_workers=1)
    U, C = G.tables(ctx, g, order, dim)
    ctx.close()
    Uo = O.init_uniform(nodes, dim, 1)
    Co = np.zeros_like(Uo) if order == 2 else None
    O.train_pairwise(O.Tables(g), Uo, Co, order=order, K=K, n_samples=n, seed=5, batch=64, lam=1e-3)
    assert np.abs(U - Uo).max() <= TOL
    if order == 2:
        assert np.abs(C - Co).max() <= TOL
