"""The loss' dots over values that stress integer sums, against the FP64
oracle: widely spread exponents, subnormals and zeros, products that cancel,
rows of infinities and NaNs, at every row width and type and at the numbers of
scores that fill a warp's lanes to the last, by one over and by halves."""
import math

import numpy as np
import pytest

import oracle as O
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def _values(kind, n, dim, rng):
    x = rng.normal(size=(n, dim))
    if kind == "wide":
        x *= 2.0 ** rng.integers(-30, 3, (n, dim))
    elif kind == "tiny":  # subnormals, zeros and rows of zeros among them
        x *= 2.0 ** -128.0
        x[:, ::3] = 0.0
        x[::5] = 0.0
    elif kind == "cancel":
        x[:, 1::2] = -x[:, ::2]
        x[:, 0] *= 1 + 2.0 ** -20
    return x.astype(np.float32)


@pytest.mark.parametrize("dim,dtype", [(d, t) for d in (16, 32, 64, 128, 256) for t in ("f32", "bf16")])
@pytest.mark.parametrize("kind", ["wide", "tiny", "cancel"])
def test_loss_of_difficult_values(dim, dtype, kind):
    from paper_2604_09419_gb300 import line as L
    g = G.graph("tiny")
    ctx = G.context()
    G.upload(ctx, g)
    rng = np.random.default_rng(dim)
    U, C = _values(kind, g.n_nodes, dim, rng), np.abs(_values(kind, g.n_nodes, dim, rng))
    if kind == "tiny":
        C = np.abs(_values("wide", g.n_nodes, dim, rng)) * np.float32(2.0 ** 100)
    if dtype == "bf16":
        U, C = [(a.view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32) for a in (U, C)]
    ctx.init_embeddings(2, dim, L.DTYPE_BF16 if dtype == "bf16" else L.DTYPE_F32, seed=1)
    ctx.set_embeddings(2, L.WHICH_U, U)
    ctx.set_embeddings(2, L.WHICH_C, C)
    T = G.oracle_tables("tiny")
    for K, m in ((0, 70), (5, 301), (15, 33), (31, 9), (32, 9)):
        rec = G.gpu_samples(ctx, K, 9, 0, m, domain=3)
        size = sum(float(np.abs(U[r[0]].astype(np.float64)) @ np.abs(C[r[1:]].astype(np.float64)).sum(0)) for r in rec)
        got = ctx.eval_loss(2, K, 9, m)
        want = O.eval_loss(T, U, C, order=2, K=K, seed=9, m=m)
        # a chain of dim FP64 additions (the oracle's) and one of m (K + 1)
        # terms of a few roundings each, per unit of the sums' magnitudes
        assert abs(got - want) <= (dim + m * (K + 1) + 16) * 2.0 ** -53 * (size + abs(want)), (K, got, want)
    ctx.close()


def test_loss_of_infinities_and_nans():
    from paper_2604_09419_gb300 import line as L
    g = G.graph("two")
    ctx = G.context()
    G.upload(ctx, g)
    for bad in (np.inf, -np.inf, np.nan):
        U = np.full((2, 128), 0.125, np.float32)
        C = U.copy()
        U[0, 77] = bad
        ctx.init_embeddings(2, 128, L.DTYPE_F32, seed=1)
        ctx.set_embeddings(2, L.WHICH_U, U)
        ctx.set_embeddings(2, L.WHICH_C, C)
        got = ctx.eval_loss(2, 5, 9, 200)
        # of a score of +inf the positive term is 0 and a negative one
        # infinite, of -inf the other way round; NaN spreads
        assert math.isnan(got) if math.isnan(bad) else got == math.inf, (bad, got)
    ctx.close()
