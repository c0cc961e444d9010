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


@pytest.mark.parametrize("signed", [False, True], ids=["unsigned", "signed"])
@pytest.mark.parametrize("d,Z,B", [(32, 8, 20001), (64, 4, 9000), (16, 32, 45000), (128, 64, 6007),
                                   (96, 64, 5200), (50, 8, 15000), (256, 128, 2800),
                                   (32, 8, 30011), (64, 4, 11003)])
def test_local_reduce_of_other_chunks_bit_exact(d, Z, B, signed):
    # chunks of other lengths, in batches large enough for the local sort
    # (its buckets that share a slot interleave), and rows that they do not tile
    w = wl.make_workload("tiny", T=15, d=d, Z=Z, M=9000, B=B, cards=("const", 900), bag=("one",),
                         ids=("zipf", 1.05), grad="dyadic", w0="dyadic")
    idx = w.indices.copy()
    idx[4::13] = 900                                   # dropped
    h = binding.PSS(w.cards, dim=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, optimizer="sgd")
    o = oracle.OraclePSS(w.cards, d=w.d, M=w.M, Z=w.Z, G=w.G, seed=w.seed, signed=signed)
    h.set_option(binding.OPT_SIGNED, int(signed))
    h.set_weights(gu.cuda(w.w0))
    locs, _ = o.locations(idx, w.offsets, B)
    locs = locs[locs >= 0]
    h.forward(gu.cuda(idx), gu.cuda(w.offsets), B)
    got = gu.host(h.backward_grad(gu.cuda(w.grad_out)))
    want = o.grad(idx, w.offsets, B, w.grad_out)
    # k / 2^8 with |k| < 2^10, summed over at most 2^20 terms: exact in fp64
    # and in every partial sum below 2^16, beyond which fp32 may round once
    small = np.abs(want) < 2.0 ** 15
    np.testing.assert_array_equal(got[small], want.astype(np.float32)[small])
    np.testing.assert_allclose(got, want, rtol=2.0 ** -20, atol=0)
    gu.torch().cuda.synchronize()
    # AUTO sorts batches that add 3.5M elements with blocks that the local sort
    # serves, 10M with blocks of 4; smaller ones take the atomic path, which
    # counts nothing
    if w.nnz * h.J * h.L < (3_500_000 if h.L >= 8 else 10_000_000):
        assert h.info()["last_path"] == binding.PATH_ATOMIC
    else:
        assert h.info()["last_path"] == binding.PATH_SORTED
        assert h.info()["last_collision_rate"] == 1.0 - np.unique(locs).shape[0] / locs.shape[0]
    h.close()
