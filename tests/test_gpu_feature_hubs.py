"""The MLP's inputs where the search for a chunk's hub changes its depth (1,
32, 33, 1,024 and 1,025 hubs, and hubs of two chunks), at every row width and
type, against the FP64 oracle.  H nodes are each joined to all of a number of
leaves, so the leaves take the path of short nodes up to 256 such nodes and
are hubs themselves beyond."""
import numpy as np
import pytest

from oracle import mlp as OM
from paper_2604_09419_gb300 import inputs as I
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hubs,leaves,dim,dtype", [
    (1, 300, 16, 0), (32, 300, 32, 1), (33, 300, 64, 0), (33, 300, 128, 1), (256, 257, 256, 1),
    (724, 300, 16, 1), (725, 300, 32, 0), (725, 300, 64, 1), (40, 2100, 128, 0), (40, 2049, 256, 0),
])
def test_inputs_of_hub_lists(hubs, leaves, dim, dtype):
    from paper_2604_09419_gb300 import line as L
    n = hubs + leaves + 5  # five nodes without arcs
    g = I.canonicalize(n, np.repeat(np.arange(hubs), leaves), hubs + np.tile(np.arange(leaves), hubs), None, symmetrize=True)
    rng = np.random.default_rng(hubs)
    ctx = G.context()
    G.upload(ctx, g)
    U, _ = G.upload_tables(ctx, 2, rng.normal(size=(n, dim)), rng.normal(size=(n, dim)), dtype=dtype)
    known = (rng.random(n) < 0.7).astype(np.uint8)
    ctx.mlp_create(2, hidden=32, act_dtype=L.DTYPE_F32, seed=1)
    X = OM.features(n, g.src, g.dst, g.w, U, known.astype(bool))
    got = np.empty(X.shape, np.float32)
    ctx.mlp_features(known)
    ctx.mlp_get_features(got)
    cnt = np.bincount(g.src[known.astype(bool)[g.dst]], minlength=n).astype(np.float64)
    # an FP32 sum of cnt rows and its division: (cnt + 2) 2^-24 max |U|
    bound = (cnt[:, None] + 2) * 2.0 ** -24 * np.abs(U).max() + 2.0 ** -23 * np.abs(X)
    assert (np.abs(got - X) <= bound).all()
    ctx.close()
