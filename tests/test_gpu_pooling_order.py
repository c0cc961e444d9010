"""A bag that the whole warp pools: lane group g of ng adds ids g, g + ng, .. in rounds of four (a
tree, then a compensated addition), and the groups' sums meet in pairs, each sum and each
compensation added with compensation.  Restated in numpy, one fp32 rounding per operation: the rows
are the same bits."""
import numpy as np
import pytest

import oracle
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu
F = np.float32


def _kahan(s, c, x):
    y = x - c
    t = s + y
    return t, (t - s) - y


def _pool(v, ng):
    """v: [ids, d] fp32 -> [d]."""
    n, d = v.shape
    rounds = -(-n // (4 * ng))
    v = np.concatenate([v, np.zeros((rounds * 4 * ng - n, d), F)]).reshape(rounds, 4, ng, d)
    s, c = np.zeros((ng, d), F), np.zeros((ng, d), F)
    for r in v:
        s, c = _kahan(s, c, (r[0] + r[1]) + (r[2] + r[3]))
    o = 1
    while o < ng:
        other = np.arange(ng) ^ o
        so, co = s[other], c[other]
        s, c = _kahan(*_kahan(s, c, so), -co)
        o *= 2
    return (s - c)[0]


@pytest.mark.parametrize("d,G", [(16, 4), (4, 1), (64, 4)])
def test_pooled_rows_are_the_documented_sums(d, G):
    B, ng = 1, 32 // -(-d // (4 if G == 4 else 1))
    w = wl.make_workload("tiny", T=200, d=d, Z=d, G=G, M=30000, B=B, cards=("const", 5000),
                         bag=("uniform", 100, 480))
    h, o = gu.make_pair(w)
    out = gu.host(h.forward(gu.cuda(w.indices), gu.cuda(w.offsets), B)).reshape(w.T, d)
    locs, _ = o.locations(w.indices, w.offsets, B)
    want = np.stack([_pool(w.w0[locs[a:b, None] + np.arange(d)], ng)
                     for a, b in zip(w.offsets[:-1], w.offsets[1:])])
    np.testing.assert_array_equal(out, want)
    h.close()
