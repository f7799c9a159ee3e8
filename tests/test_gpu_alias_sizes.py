"""Alias tables, bit-exact against the oracle, where the parallel pairing
changes form: tiles of 4,096 items, groups of 1,024 lights, windows of heavies
above and below what fits shared memory, no light or heavy items, weights whose
masses come from the small-integer table, from larger integers, or from FP64."""
import numpy as np
import pytest

import oracle as O
from paper_2604_09419_gb300 import inputs as I
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


def ring(n, w):
    """One arc per node, of the given weights."""
    i = np.arange(n, dtype=np.int32)
    return I.Graph(n, i, np.roll(i, -1), np.asarray(w, np.float32), True)


def weights(kind, n):
    rng = np.random.default_rng(n)
    if kind == "equal":
        return np.full(n, 3.0)
    if kind == "ints":
        return rng.integers(1, 40, n)
    if kind == "large ints":
        return rng.integers(1, 1 << 24, n)
    if kind == "reals":
        return rng.lognormal(size=n)
    if kind == "one light":  # all other items are heavy: one light's window holds them all
        return np.where(np.arange(n) == n // 2, 1.0, 1000.0)
    if kind == "one heavy":
        return np.where(np.arange(n) == n // 3, 1000.0, 1.0)
    raise KeyError(kind)


@pytest.mark.parametrize("kind,n", [("equal", 4097), ("ints", 1), ("ints", 1023), ("ints", 4095), ("ints", 4096),
                                    ("ints", 70001), ("large ints", 8193), ("reals", 1025), ("reals", 50021),
                                    ("one light", 30011), ("one heavy", 12289)])
def test_alias_sizes(kind, n):
    from paper_2604_09419_gb300 import line as L
    g = ring(n, weights(kind, n))
    T = O.Tables(g)
    ctx = G.context()
    G.upload(ctx, g)
    for which, (thr, alias) in ((L.TABLE_EDGE, (T.thr_e, T.alias_e)), (L.TABLE_NEG, (T.thr_n, T.alias_n))):
        got = G.gpu_alias(ctx, g, which)
        assert np.array_equal(got[0], thr) and np.array_equal(got[1], alias), which
    ctx.close()
