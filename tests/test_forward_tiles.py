"""The forward's tiles: one lane per bag, so a tile holds at most 32 bags whatever the row width and
the batch.  The rule is host code and checked over all layouts with the host compiler; rows of one
or two columns (16 or 32 lane groups per warp) are then checked bit for bit at batches large enough
for the widest tiles (dyadic inputs: every partial sum is exact)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2207_10731_gb300", "csrc")


@pytest.fixture(scope="module")
def tile_bags(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    src, lib = d / "tiles.cpp", d / "tiles.so"
    src.write_text('#include "pss_tiles.h"\n'
                   'extern "C" int bags(int64_t T, int J, int log2gs, int64_t rows, int64_t warps)'
                   ' { return pss::tile_bags(T, J, log2gs, rows, warps); }\n')
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True)
    fn = ctypes.CDLL(str(lib)).bags
    fn.argtypes = [ctypes.c_int64, ctypes.c_int, ctypes.c_int, ctypes.c_int64, ctypes.c_int64]
    return fn


def test_every_bag_of_a_tile_has_a_lane(tile_bags):
    for log2gs in range(6):
        ng = 32 >> log2gs
        step = max(ng, 4)
        for J in (1, 2, 3, 4, 7, 16, 33, 128, 512):
            for T in (1, 2, 5, 26, 1000):
                for rows in (1, 2, 31, 33, 257, 4515, 8192, 16384, 65536, 1 << 20, 1 << 26):
                    for ctas in (1, 2, 3, 4, 8):
                        wb = tile_bags(T, J, log2gs, rows, 152 * ctas * 8)
                        what = (log2gs, J, T, rows, ctas, wb)
                        assert step <= wb <= 32 and wb % ng == 0, what
                        assert 32 >> (wb - 1).bit_length() >= 1, what
                        assert wb == step or wb * J <= 512, what


@pytest.mark.gpu
@pytest.mark.parametrize("bad", [False, True], ids=["valid", "bad-ids"])
@pytest.mark.parametrize("bag", [("one",), ("uniform", 0, 5)], ids=["one", "several"])
@pytest.mark.parametrize("d,Z,G", [(1, 1, 1), (2, 2, 1), (2, 1, 1), (4, 4, 4), (8, 8, 4), (8, 4, 4),
                                   (3, 2, 1), (16, 16, 4)])
def test_narrow_rows_large_batches(d, Z, G, bag, bad):
    T, B = 26, 6601
    w = wl.make_workload("tiny", T=T, d=d, Z=Z, G=G, M=5000, B=B, cards=("const", 60), bag=bag,
                         ids=("zipf", 1.1), grad="dyadic", w0="dyadic")
    idx = w.indices.copy()
    if bad:
        idx[2::11] = 60
    h = binding.PSS(w.cards, dim=d, M=w.M, Z=Z, G=G, seed=w.seed, optimizer="sgd")
    o = oracle.OraclePSS(w.cards, d=d, M=w.M, Z=Z, G=G, seed=w.seed)
    h.set_weights(gu.cuda(w.w0))
    ref, first_bad = o.forward(w.w0, idx, w.offsets, B)
    want = o.grad(idx, w.offsets, B, w.grad_out).astype(np.float32)
    for path in (binding.PATH_ATOMIC, binding.PATH_SORTED):
        h.set_option(binding.OPT_BACKWARD_PATH, path)
        out = gu.host(h.forward(gu.cuda(idx), gu.cuda(w.offsets), B)).ravel()
        np.testing.assert_array_equal(out, ref)
        grad = gu.host(h.backward_grad(gu.cuda(w.grad_out)))
        np.testing.assert_array_equal(grad, want)
        assert h.get_error()[1] == first_bad
    h.close()
