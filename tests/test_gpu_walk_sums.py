"""Walks over the running weight sums of long nodes, bit for bit against the
oracle: stars at the numbers of arcs where a warp takes over from a thread and
around its blocks of 32, with whole weights, fractions from the first arc or
from the middle on, and weights beyond 2^24."""
import numpy as np
import pytest

import oracle as O
from paper_2604_09419_gb300 import inputs as I
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

LEAVES = (1, 2, 31, 33, 63, 64, 65, 66, 95, 96, 97, 127, 128, 129, 1000, 4096, 20001)


@pytest.mark.parametrize("kind", ["none", "whole", "fractions", "middle", "large"])
def test_walks_of_stars(kind):
    rng = np.random.default_rng(7)
    src, dst, w, n = [], [], [], 0
    for d in LEAVES:
        src.append(np.full(d, n))
        dst.append(n + 1 + np.arange(d))
        x = rng.integers(1, 9, d).astype(np.float64)
        if kind == "fractions":
            x = rng.lognormal(0, 1, d)
        elif kind == "middle":
            x[d // 2:] += 0.3
        elif kind == "large":
            x = np.where(rng.random(d) < 0.01, 2.0 ** 25 + 4, x * 2.0 ** 21)
        # the short stars' arcs weigh more, so that walks visit all stars alike
        w.append(x * max(1, 20001 // d))
        n += d + 1
    g = I.canonicalize(n, np.concatenate(src), np.concatenate(dst),
                       None if kind == "none" else np.concatenate(w).astype(np.float32), symmetrize=True)
    ctx = G.context()
    G.upload(ctx, g)
    m = 60_000
    out = np.empty((m, 2), np.int32)
    ctx.sample_walk_debug(0, 5, 21, 1, 0, m, out)
    assert np.array_equal(out, O.sample_walk(O.Tables(g), O.walk_cumw(g), 5, 0, m, 0, 21, 1))
    ctx.close()
