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
