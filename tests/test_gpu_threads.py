"""Two host threads, each with its own handle and stream, run the deterministic sort with different
digit widths (different sizes of shared memory of one kernel): every call succeeds and every
gradient is the same."""
import threading

import numpy as np
import pytest

from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def test_threads_with_different_digit_widths():
    t = gu.torch()
    w = wl.make_workload("tiny", d=32, Z=32, M=1 << 20, B=64, grad="dyadic", w0="dyadic")
    errors, grads = [], {}

    def work(bits):
        try:
            with t.cuda.stream(t.cuda.Stream()):
                h, _ = gu.make_pair(w)
                h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_SORTED)
                h.set_option(binding.OPT_DETERMINISTIC, 1)
                h.set_option(binding.OPT_SORT_DIGIT_BITS, bits)
                idx, off, go = gu.cuda(w.indices), gu.cuda(w.offsets), gu.cuda(w.grad_out)
                out = None
                grad = t.empty(w.M, dtype=t.float32, device="cuda")
                start.wait()
                for _ in range(3000):
                    out = h.forward(idx, off, w.B, out=out)
                    h.backward_grad(go, grad=grad)
                grads[bits] = gu.host(grad)
                h.close()
        except Exception as e:   # reported below, in the test's own thread
            errors.append((bits, e))

    start = threading.Barrier(2)
    threads = [threading.Thread(target=work, args=(bits,)) for bits in (4, 11)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors
    np.testing.assert_array_equal(grads[4], grads[11])
