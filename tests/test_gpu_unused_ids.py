"""Ids outside every bag (offsets[0] > 0, offsets[T*B] < nnz: a padded indices buffer) add nothing,
whatever an earlier batch left in the sorted path's buffers, and malformed offsets never reach past
them.  Dyadic inputs: gradients and SGD steps equal the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

# how the sorted path groups the pairs: (d, Z, batch, options)
SORTS = {
    "local": (64, 32, 700, {binding.OPT_SORT_SCOPE: binding.SORT_LOCAL}),
    "local-touched": (64, 32, 700, {binding.OPT_SORT_SCOPE: binding.SORT_LOCAL,
                                    binding.OPT_UPDATE_MODE: binding.UPDATE_TOUCHED}),
    "local-counted": (16, 8, 45001, {}),
    "counting": (64, 32, 700, {binding.OPT_SORT_SCOPE: binding.SORT_GLOBAL}),
    "counting-touched": (20, 8, 300, {binding.OPT_UPDATE_MODE: binding.UPDATE_TOUCHED}),
    "radix-window": (64, 32, 700, {binding.OPT_DETERMINISTIC: 1}),
    "radix-touched": (16, 16, 3000, {binding.OPT_DETERMINISTIC: 1,
                                     binding.OPT_UPDATE_MODE: binding.UPDATE_TOUCHED}),
}


def _batch(d, Z, B, seed):
    return wl.make_workload("tiny", T=5, d=d, Z=Z, G=4, M=5000, B=B, cards=("const", 60),
                            bag=("uniform", 0, 3), ids=("zipf", 1.1), grad="dyadic", w0="dyadic",
                            seed=seed)


def _pair(w, opts, signed):
    h = binding.PSS(w.cards, dim=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, optimizer="sgd")
    o = oracle.OraclePSS(w.cards, d=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, signed=signed)
    h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_SORTED)
    h.set_option(binding.OPT_SIGNED, int(signed))
    for k, v in opts.items():
        h.set_option(k, v)
    h.set_weights(gu.cuda(w.w0))
    return h, o


def _check(h, o, w, w0, idx, off, B, go):
    """Forward, gradient and SGD step (lr 1/4) of one batch from weights w0; returns the weights."""
    out = gu.host(h.forward(gu.cuda(idx), gu.cuda(off), B)).ravel()
    np.testing.assert_array_equal(out, o.forward(w0, idx, off, B)[0])
    grad = gu.host(h.backward_grad(gu.cuda(go)))
    np.testing.assert_array_equal(grad, o.grad(idx, off, B, go).astype(np.float32))
    h.backward_update(gu.cuda(go), 0.25)
    w1, _, _ = o.step(w0, None, idx, off, B, go, "sgd", 0.25)
    got = gu.host(h.get_weights())
    np.testing.assert_array_equal(got, w1)
    return w1


@pytest.mark.parametrize("signed", [False, True], ids=["unsigned", "signed"])
@pytest.mark.parametrize("sort", list(SORTS))
def test_ids_outside_the_bags_add_nothing(sort, signed):
    d, Z, B, opts = SORTS[sort]
    w = _batch(d, Z, B, seed=3)
    h, o = _pair(w, opts, signed)
    rng = np.random.default_rng(1)
    lead, trail = rng.integers(0, 60, 701), rng.integers(0, 60, 9000)
    # fresh buffers; then, after a batch that fills them, a smaller one with unused ids
    idx, off = np.concatenate([lead, w.indices, trail]), w.offsets + len(lead)
    w1 = _check(h, o, w, w.w0, idx, off, B, w.grad_out)
    w1 = _check(h, o, w, w1, idx, off - off[0], B, w.grad_out)
    B2 = B * 3 // 4 if sort != "local-counted" else B - 2000
    s = _batch(d, Z, B2, seed=4)
    idx = np.concatenate([lead, s.indices, trail])
    _check(h, o, w, w1, idx, s.offsets + len(lead), B2, s.grad_out)
    assert h.get_error() == (binding.PSS_OK, -1)
    h.close()


@pytest.mark.parametrize("sort", list(SORTS))
def test_malformed_offsets_stay_inside_the_buffers(sort):
    d, Z, B, opts = SORTS[sort]
    w = _batch(d, Z, B, seed=3)
    h, o = _pair(w, opts, False)
    nnz, rng = w.indices.shape[0], np.random.default_rng(2)

    def with_(at, value):
        off = w.offsets.copy()
        off[at] = value
        return off

    go = gu.cuda(w.grad_out)
    for off in (with_(0, -3), with_(-1, nnz + 5), with_(100, 1 << 40), with_(117, -(1 << 40)),
                with_(130, 0), rng.integers(0, nnz + 1, w.offsets.shape[0])):
        h.forward(gu.cuda(w.indices), gu.cuda(off), B)
        assert np.isfinite(gu.host(h.backward_grad(go))).all()
        assert h.get_error() == (binding.PSS_ERR_INDEX_RANGE, -2)
    # numbers whose products and successors leave 64 bits
    top = (1 << 63) - 1
    for at, v in ((0, -(1 << 62)), (0, 1 << 62), (0, -top // 3), (-1, 1 << 62), (-1, -(1 << 62)),
                  (-1, top // 3), (-1, top), (0, -top - 1), (96, 1 << 62), (96, -top // 3),
                  (96, top), (101, -top - 1)):
        h.forward(gu.cuda(w.indices), gu.cuda(with_(at, v)), B)
        assert np.isfinite(gu.host(h.backward_grad(go))).all()
        assert h.get_error() == (binding.PSS_ERR_INDEX_RANGE, -2)
    off = w.offsets.copy()
    off[50], off[51] = top, -top - 1
    h.forward(gu.cuda(w.indices), gu.cuda(off), B)
    assert h.get_error() == (binding.PSS_ERR_INDEX_RANGE, -2)
    # an offset inside a tile (of 4, 8, .. 32 bags): that tile's ids add nothing, all others do
    off = with_(5, w.offsets[5] - 100)
    h.forward(gu.cuda(w.indices), gu.cuda(off), B)
    got = gu.host(h.backward_grad(go)).astype(np.float64).sum()
    rows = w.grad_out.reshape(B, w.T, d).astype(np.float64)
    lens = np.diff(w.offsets).reshape(w.T, B)
    per_bag = (lens.T * rows.sum(2)).T.ravel()      # the bags' gradient mass, table-major
    left_out = [per_bag.sum() - per_bag[4 // nb * nb:][:nb].sum() for nb in range(4, 36, 4)]
    assert got in left_out
    assert h.get_error() == (binding.PSS_ERR_INDEX_RANGE, -2)
    # and the next batch is exact
    _check(h, o, w, w.w0, w.indices, w.offsets, B, w.grad_out)
    assert h.get_error() == (binding.PSS_OK, -1)
    h.close()
