"""The staged reduce of the sorted path at the edges of its blocks (32 entries), ranges (64 and
more entries per warp) and local segments (8192 pairs), with dropped ids.  Dyadic gradients: every
partial sum is exact, so the gradient equals the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("signed", [False, True], ids=["unsigned", "signed"])
@pytest.mark.parametrize("mode", ["global", "local", "deterministic"])
@pytest.mark.parametrize("B", [1, 31, 32, 33, 63, 64, 65, 97, 8191, 8192, 8193, 40001])
def test_reduce_edges_bit_exact(B, mode, signed):
    w = wl.make_workload("tiny", T=1, d=32, Z=32, M=4096, B=B, cards=("const", 50), bag=("one",),
                         ids=("zipf", 1.2), grad="dyadic", w0="dyadic")
    idx = w.indices.copy()
    idx[3::7] = 1000                                   # outside the table: dropped
    h = binding.PSS(w.cards, dim=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, optimizer="sgd")
    o = oracle.OraclePSS(w.cards, d=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, signed=signed)
    h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_SORTED)
    h.set_option(binding.OPT_SIGNED, int(signed))
    h.set_option(binding.OPT_SORT_SCOPE,
                 binding.SORT_LOCAL if mode == "local" else binding.SORT_GLOBAL)
    h.set_option(binding.OPT_DETERMINISTIC, int(mode == "deterministic"))
    h.set_weights(gu.cuda(w.w0))
    h.forward(gu.cuda(idx), gu.cuda(w.offsets), B)
    got = gu.host(h.backward_grad(gu.cuda(w.grad_out)))
    assert h.info()["last_path"] == binding.PATH_SORTED
    want = o.grad(idx, w.offsets, B, w.grad_out)
    np.testing.assert_array_equal(got, want.astype(np.float32))
    assert h.get_error()[1] == (3 if B > 3 else -1)
    h.close()


@pytest.mark.parametrize("signed", [False, True], ids=["unsigned", "signed"])
@pytest.mark.parametrize("B", [3100, 8191, 8193, 16385, 40001])
def test_auto_local_sort_counts_distinct_locations(B, signed):
    # more than 3 pairs per block start: grouped within segments, with the
    # distinct locations counted exactly for the collision rate
    w = wl.make_workload("tiny", T=1, d=32, Z=32, M=4096, B=B, cards=("const", 700), bag=("one",),
                         ids=("zipf", 1.05), grad="dyadic", w0="dyadic")
    idx = w.indices.copy()
    idx[5::9] = -1                                     # dropped
    h = binding.PSS(w.cards, dim=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, optimizer="sgd")
    o = oracle.OraclePSS(w.cards, d=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, signed=signed)
    assert B > 3 * h.R
    h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_SORTED)
    h.set_option(binding.OPT_SIGNED, int(signed))
    h.set_weights(gu.cuda(w.w0))
    locs, _ = o.locations(idx, w.offsets, B)
    locs = locs[locs >= 0]
    want = o.grad(idx, w.offsets, B, w.grad_out).astype(np.float32)
    for _ in range(2):                                 # the marks and counts return to zero
        h.forward(gu.cuda(idx), gu.cuda(w.offsets), B)
        got = gu.host(h.backward_grad(gu.cuda(w.grad_out)))
        np.testing.assert_array_equal(got, want)
        gu.torch().cuda.synchronize()
        rate = h.info()["last_collision_rate"]
        assert rate == 1.0 - np.unique(locs).shape[0] / locs.shape[0]
    h.close()


@pytest.mark.parametrize("B", [100, 2047, 2049, 5000])
def test_local_sort_touched_list(B):
    # the local sort's touched list visits exactly what the dense pass does
    w = wl.make_workload("tb", B=B, M=1 << 20, grad="dyadic", w0="dyadic")
    state = []
    for mode in (binding.UPDATE_DENSE, binding.UPDATE_TOUCHED):
        h = binding.PSS(w.cards, dim=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, optimizer="adagrad")
        h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_SORTED)
        h.set_option(binding.OPT_SORT_SCOPE, binding.SORT_LOCAL)
        h.set_option(binding.OPT_UPDATE_MODE, mode)
        h.set_weights(gu.cuda(w.w0))
        for _ in range(2):
            h.forward(gu.cuda(w.indices), gu.cuda(w.offsets), B)
            h.backward_update(gu.cuda(w.grad_out), w.lr)
        state.append([gu.host(x) for x in h.get_state()])
        h.close()
    np.testing.assert_array_equal(state[0][0], state[1][0])
    np.testing.assert_array_equal(state[0][1], state[1][1])
