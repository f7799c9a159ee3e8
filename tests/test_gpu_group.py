"""Grouping of a batch's items by row, against the FP64 oracle at the sizes
where its split into parts changes: one part up to 16,384 items, then 2, 4, 8
and 16 parts, then the path through global memory; parts whose keys exceed a
CTA's shared memory; rows with thousands of entries (a warp sorts them)."""
import numpy as np
import pytest

from tests import gpu_util as G

pytestmark = pytest.mark.gpu

# The learning rate is scaled so that a batch changes no value by more than
# about 1: a row's n entries are summed in chunks of 8, then chunk by chunk,
# each addition off by at most 2^-24 of a partial sum of at most 1, so two
# batches of n = 2^15 entries stay within sqrt(2 n / 8) 2^-24 = 6e-6 unless
# the roundings conspire; the library's stated bound is 1e-5.
TOL = 1e-5


@pytest.mark.parametrize("name,order,K,B", [
    ("tiny", 2, 5, 2340),     # 16,380 items, nearly all in shared rows: one part, keys in the scratch array
    ("tiny", 1, 5, 2341),     # 16,387: two parts
    ("two", 2, 5, 4096),      # four rows of thousands of entries
    ("two", 1, 2, 4096),      # 16,384 items on two rows, source and context entries mixed
    ("isolated", 1, 0, 8192),  # a hub of a star: half of all entries
    ("rmat14", 2, 5, 4682),   # 32,774: four parts
    ("rmat14", 1, 32, 1928),  # 65,552 at the widest record: eight parts
    ("rmat14", 2, 5, 37449),  # 262,143: sixteen parts
    ("rmat14", 1, 5, 37450),  # 262,150: through global memory
])
def test_group_sizes(name, order, K, B):
    from paper_2604_09419_gb300 import line as L
    g = G.graph(name)
    ctx = G.context()
    G.upload(ctx, g)
    ctx.init_embeddings(order, 16, L.DTYPE_F32, seed=1)
    n, lr = 2 * B + 17, 0.025 * min(1.0, 256.0 / B)
    ctx.train_steps(order, 16, K, n, 5, lr0=lr, batch=B, lam=1e-3)
    U, C = G.tables(ctx, g, order, 16)
    Uo, Co = G.oracle_run(name, order, 16, K, n, 5, B, 1, lam=1e-3, lr0=lr)
    err = np.abs(U - Uo).max()
    if order == 2:
        err = max(err, np.abs(C - Co).max())
    ctx.close()
    assert err <= TOL, err
