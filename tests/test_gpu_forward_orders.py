"""The forward over several tiles per warp, in both tile orders (by bag; table by table for arrays of
2^24 elements and more), with tables that the warps' stride does not divide: every warp crosses
table boundaries.  One id, several ids per bag, ids outside their table, the variant for many
one-id bags, and the pinned host output that is computed in chunks of rows.  Weights are multiples
of 1/256, so every sum is exact and the rows equal w[locations] summed in fp64."""
import numpy as np
import pytest

from paper_2207_10731_gb300 import binding
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

BY_TABLE, BY_BAG = 1 << 24, 1 << 20      # array lengths on either side of the rule


def _batch(t, T, B, several, bad):
    g = t.Generator(device="cuda")
    g.manual_seed(5)
    lens = t.randint(0, 10, (T * B,), device="cuda", generator=g) if several else \
        t.ones(T * B, dtype=t.int64, device="cuda")
    off = t.zeros(T * B + 1, dtype=t.int64, device="cuda")
    t.cumsum(lens, 0, out=off[1:])
    idx = t.randint(0, 5000, (int(off[-1]),), device="cuda", generator=g)
    if bad:
        idx[3::17] = 5000
        idx[-1] = -1
    return idx, off, lens


@pytest.mark.parametrize("M", [BY_TABLE, BY_BAG], ids=["by-table", "by-bag"])
@pytest.mark.parametrize("T,B,d,Z,several,bad,host", [
    (7, 30011, 32, 32, False, False, False),
    (7, 30011, 32, 32, True, True, False),
    (26, 13001, 128, 32, False, False, False),     # 338,026 bags: the variant for many of them
    (26, 13001, 128, 32, False, True, False),
    (3, 60007, 64, 16, True, False, False),
    (11, 20021, 16, 16, True, True, False),
    (5, 40003, 128, 32, False, False, True),       # 102 MB of rows to the host, in four chunks
    (5, 40003, 128, 32, True, True, True)])
def test_rows_are_the_weights_at_the_locations(M, T, B, d, Z, several, bad, host):
    t = gu.torch()
    h = binding.PSS(np.full(T, 5000, np.int64), dim=d, M=M, Z=Z, G=4, seed=9, optimizer="sgd")
    w = t.randint(-512, 513, (M,), device="cuda").float() / 256
    h.set_weights(w)
    idx, off, lens = _batch(t, T, B, several, bad)
    out = t.empty((B, T, d), pin_memory=True) if host else None
    out = h.forward(idx, off, B, out=out)
    t.cuda.synchronize()
    locs = h.compute_locations(idx, off, B).view(-1, h.J)
    ok = (idx >= 0) & (idx < 5000)
    assert bool((locs[~ok] == -1).all())
    slot = t.arange(T * B, device="cuda").repeat_interleave(lens)[ok]
    col = t.arange(d, device="cuda")
    want = t.zeros((T * B, d), dtype=t.float64, device="cuda")
    locs = locs[ok]
    for a in range(0, locs.shape[0], 1 << 18):
        at = locs[a:a + (1 << 18), col // Z] + col % Z
        want.index_add_(0, slot[a:a + (1 << 18)], w[at].double())
    want = want.float().view(T, B, d).transpose(0, 1)
    assert t.equal(out.cuda(), want)
    status, first = h.get_error()
    assert first == (int((~ok).nonzero()[0, 0]) if bad else -1)
    h.close()
