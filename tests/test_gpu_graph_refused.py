"""Large invalid graphs are refused at once: arcs out of order, whose row offsets
would be n_nodes writes for every ascent, and a single bad arc at the end."""
import time

import numpy as np
import pytest

import oracle as O
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

N, M = 1 << 20, 1 << 22


def arcs(kind):
    rng = np.random.default_rng(11)
    src = np.sort(rng.integers(0, N, M)).astype(np.int32)
    dst = rng.integers(0, N, M).astype(np.int32)
    w = np.ones(M, np.float32)
    if kind == "random":
        rng.shuffle(src)
    elif kind == "first and last by turns":
        src[::2], src[1::2] = 0, N - 1
    elif kind == "runs of sixteen":  # each in order, up to the last node
        src = np.tile(np.linspace(0, N - 1, 16).astype(np.int32), M // 16)
    elif kind == "descent at the end":
        src[-1] = 0
    elif kind == "negative source":
        src[M // 2] = -1
    elif kind == "target beyond the nodes":
        dst[-1] = N
    elif kind == "weight of zero":
        w[-1] = 0.0
    return src, dst, w


@pytest.mark.parametrize("kind", ["random", "first and last by turns", "runs of sixteen", "descent at the end",
                                  "negative source", "target beyond the nodes", "weight of zero"])
def test_refused_at_once(kind):
    import torch

    from paper_2604_09419_gb300 import line as L
    ctx = G.context()
    good = [torch.from_numpy(a).cuda() for a in arcs("")]
    ctx.build_alias(N, *good)  # (allocations, module loading)
    bad = [torch.from_numpy(a).cuda() for a in arcs(kind)]
    torch.cuda.synchronize()
    t = time.perf_counter()
    with pytest.raises(L.LineError) as e:
        ctx.build_alias(N, *bad)
    t = time.perf_counter() - t
    assert e.value.status == L.LINE_ERR_VALIDATE
    # at most 32 offsets an arc, and a piece of 1,024 per resident thread:
    # 4e8 writes, a few ms
    assert t < 0.25, t
    # and the context takes a valid graph afterwards
    g = G.graph("isolated")
    G.upload(ctx, g)
    T = O.Tables(g)
    got = G.gpu_alias(ctx, g, L.TABLE_NEG)
    assert np.array_equal(got[0], T.thr_n) and np.array_equal(got[1], T.alias_n)
    ctx.close()
