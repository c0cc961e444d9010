"""Batches that AUTO sorts below its general threshold (5M adds with chunks of 32 and more, 10M with
shorter ones) keep the atomic path's sums: every contribution is added in fp64, so the gradient is
the rounded fp64 sum, infinities stay infinities and sums beyond fp32 can come back.

Bound: n fp64 additions in any order are off by at most (n - 1) 2^-53 sum|x| (n < 2^17 here), then
one rounding to fp32, 2^-24 |g|."""
import numpy as np
import pytest

import oracle
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

SHAPES = {"L16": (16, 16, 9001), "L8": (16, 8, 9001), "L32": (64, 32, 2201)}   # d, Z, B


def _setup(shape, signed=False):
    d, Z, B = SHAPES[shape]
    w = wl.make_workload("tiny", T=26, d=d, Z=Z, G=4, M=20000, B=B, cards=("const", 300),
                         ids=("zipf", 1.05), grad="normal")
    h = binding.PSS(w.cards, dim=d, M=w.M, Z=Z, G=4, seed=w.seed, optimizer="sgd")
    h.set_option(binding.OPT_SIGNED, int(signed))
    h.set_weights(gu.cuda(w.w0))
    o = oracle.OraclePSS(w.cards, d=d, M=w.M, Z=Z, G=4, seed=w.seed, signed=signed)
    assert 3_500_000 <= w.indices.shape[0] * d < (5_000_000 if Z == 32 else 10_000_000)
    return w, h, o


def _grad(h, w, go):
    h.forward(gu.cuda(w.indices), gu.cuda(w.offsets), w.B)
    return gu.host(h.backward_grad(go))


@pytest.mark.parametrize("signed", [False, True], ids=["unsigned", "signed"])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_gradient_is_the_rounded_fp64_sum(shape, signed):
    w, h, o = _setup(shape, signed)
    got = _grad(h, w, gu.cuda(w.grad_out)).astype(np.float64)
    assert h.info()["last_path"] == binding.PATH_SORTED
    ref = o.grad(w.indices, w.offsets, w.B, w.grad_out)
    A = o.grad(w.indices, w.offsets, w.B, np.abs(w.grad_out)) if not signed else \
        oracle.OraclePSS(w.cards, d=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed).grad(
            w.indices, w.offsets, w.B, np.abs(w.grad_out))
    bound = 2.0 ** -24 * np.abs(ref) * (1 + 1e-6) + 2.0 ** (17 - 53) * A
    worst = np.max(np.abs(got - ref) / np.where(bound > 0, bound, 1))
    assert worst <= 1, worst
    h.close()


@pytest.mark.parametrize("shape", list(SHAPES))
def test_infinities_and_sums_beyond_fp32(shape):
    w, h, o = _setup(shape)
    go = w.grad_out.reshape(w.B, w.T, w.d).copy()
    go[7, 3, 1] = np.inf
    go[100:110, 5, :] = 3e38          # ten rows whose sum leaves fp32 ...
    go[110:120, 5, :] = -3e38         # ... and ten that bring it back
    idx = w.indices.copy()
    at = 5 * w.B
    idx[at + 100:at + 120] = idx[at + 100]
    w.indices = idx
    got = _grad(h, w, gu.cuda(go.ravel()))
    assert h.info()["last_path"] == binding.PATH_SORTED
    ref = o.grad(idx, w.offsets, w.B, go.ravel())
    assert np.isinf(ref).any() and not np.isnan(ref).any()
    np.testing.assert_array_equal(np.isinf(got), np.isinf(ref.astype(np.float32)))
    assert not np.isnan(got).any()
    h.close()


def test_batches_without_such_a_reduce_stay_atomic():
    # deterministic, a touched update (which the counted local sort does not serve), fp32
    # accumulation, a forced global sort, and a gradient that the staged reduce cannot copy
    for shape, key, value, path in (
            ("L16", binding.OPT_DETERMINISTIC, 1, binding.PATH_ATOMIC),
            ("L16", binding.OPT_UPDATE_MODE, binding.UPDATE_TOUCHED, binding.PATH_ATOMIC),
            ("L16", binding.OPT_ACCUM, binding.ACCUM_F32, binding.PATH_ATOMIC),
            ("L32", binding.OPT_SORT_SCOPE, binding.SORT_GLOBAL, binding.PATH_ATOMIC),
            ("L32", binding.OPT_UPDATE_MODE, binding.UPDATE_DENSE, binding.PATH_SORTED)):
        w, h, o = _setup(shape)
        h.set_option(key, value)
        _grad(h, w, gu.cuda(w.grad_out))
        assert h.info()["last_path"] == path, (shape, key)
        h.close()
    w, h, o = _setup("L32")
    t = gu.torch()
    buf = t.empty(w.grad_out.size + 1, dtype=t.float32, device="cuda")
    buf[1:] = gu.cuda(w.grad_out).ravel()
    got = _grad(h, w, buf[1:])
    assert h.info()["last_path"] == binding.PATH_ATOMIC
    gu.check_grad(got, o.grad(w.indices, w.offsets, w.B, w.grad_out),
                  o.grad(w.indices, w.offsets, w.B, np.abs(w.grad_out)))
    h.close()
