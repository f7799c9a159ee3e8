"""Dots of one large product and many tiny ones: every FP64 sum of them is the
large product, so the loss has to be, bit for bit, that of rows without the
tiny values - also where a factor of the large product is subnormal."""
import numpy as np
import pytest

from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [16, 32, 64, 128, 256])
@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("u,c", [(2.0, 4.0), (2.0 ** -3, 2.0 ** -3), (2.0 ** -133, 2.0 ** 127)])
@pytest.mark.parametrize("tiny", [-(2.0 ** -60), 2.0 ** -60])
def test_tiny_products_do_not_count(dim, dtype, u, c, tiny):
    from paper_2604_09419_gb300 import line as L
    g = G.graph("two")
    ctx = G.context()
    G.upload(ctx, g)
    ctx.init_embeddings(2, dim, dtype, seed=1)

    def loss(u, c, tiny):
        U, C = np.full((2, dim), tiny, np.float32), np.full((2, dim), 2.0 ** -80 if tiny else 0.0, np.float32)
        U[:, dim // 3], C[:, dim // 3] = u, c
        ctx.set_embeddings(2, L.WHICH_U, U)
        ctx.set_embeddings(2, L.WHICH_C, C)
        return ctx.eval_loss(2, 0, 9, 1)

    # the same product from two normal factors
    e = int(round(np.log2(u * c)))
    assert loss(u, c, tiny) == loss(2.0 ** (e // 2), 2.0 ** (e - e // 2), 0.0)
    ctx.close()
