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


SHIM = """
#include "pss_tiles.h"
extern "C" int bags(int64_t T, int J, int log2gs, int64_t rows, int64_t warps) {
    return pss::tile_bags(T, J, log2gs, rows, warps);
}
extern "C" int64_t max_tiles() { return pss::kMaxTiles; }
// the first n tiles from tile number `tile` on: t, r, place in the offsets, inside or not
extern "C" void walk(int64_t tile, int64_t nwarps, int64_t T, int64_t tpt, int64_t B, int wb,
                     int by_table, int64_t n, int64_t* out) {
    const pss::TileWalk w((uint32_t)nwarps, (uint32_t)T, (uint32_t)tpt, B, wb, by_table != 0);
    uint32_t t, r;
    w.first((uint32_t)tile, t, r);
    int64_t o = (int64_t)t * B + (int64_t)r * wb;
    for (int64_t i = 0; i < n; ++i, out += 4) {
        out[0] = t, out[1] = r, out[2] = o, out[3] = w.inside(t, r);
        o += w.advance(t, r);
    }
}
"""


@pytest.fixture(scope="module")
def tiles(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    src, lib = d / "tiles.cpp", d / "tiles.so"
    src.write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(src), "-o", str(lib)],
                   check=True)
    lib = ctypes.CDLL(str(lib))
    i, q = ctypes.c_int, ctypes.c_int64
    lib.bags.argtypes = [q, i, i, q, q]
    lib.max_tiles.restype = q
    lib.walk.argtypes = [q, q, q, q, q, i, i, q, ctypes.c_void_p]
    lib.walk.restype = None
    return lib


def _walk(tiles, tile, nwarps, T, tpt, B, wb, by_table, n):
    out = np.zeros((n, 4), np.int64)
    tiles.walk(tile, nwarps, T, tpt, B, wb, int(by_table), n, out.ctypes.data)
    return out


def test_every_bag_of_a_tile_has_a_lane(tiles):
    for log2gs in range(6):
        ng = 32 >> log2gs
        step = max(ng, 4)
        for J in (1, 2, 3, 4, 7, 16, 33, 128, 512):
            for T in (1, 2, 5, 26, 1000):
                for rows in (1, 2, 31, 33, 257, 4515, 8192, 16384, 65536, 1 << 20, 1 << 26):
                    for ctas in (1, 2, 3, 4, 8):
                        wb = tiles.bags(T, J, log2gs, rows, 152 * ctas * 8)
                        what = (log2gs, J, T, rows, ctas, wb)
                        assert step <= wb <= 32 and wb % ng == 0, what
                        assert 32 >> (wb - 1).bit_length() >= 1, what
                        assert wb == step or wb * J <= 512, what


@pytest.mark.parametrize("by_table", [False, True], ids=["by-bag", "by-table"])
def test_the_warps_walk_every_tile_once(tiles, by_table):
    for T, B, wb in ((1, 1, 4), (1, 1000, 4), (26, 131, 16), (5, 20001, 12), (7, 64, 32), (300, 3, 8)):
        tpt = -(-B // wb)
        for nwarps in (8, 56, 8 * 152, 8 * 304):
            seen = np.zeros((T, tpt), np.int64)
            n = T * tpt // nwarps + 4
            for tile in range(min(nwarps, T * tpt + 7)):
                w = _walk(tiles, tile, nwarps, T, tpt, B, wb, by_table, n)
                k = int(w[:, 3].sum())
                assert w[:k, 3].all(), "a tile after the last one"
                t, r, o = w[:k, 0], w[:k, 1], w[:k, 2]
                np.testing.assert_array_equal(o, t * B + r * wb)
                np.add.at(seen, (t, r), 1)
            assert (seen == 1).all(), (T, B, wb, nwarps)


def test_walk_up_to_the_most_tiles(tiles):
    # as many tables (of one tile) as the API's 32-bit count allows: the last tiles of some warps,
    # and the prefetches past them
    T, nwarps = (1 << 31) - 1, 8 * 152 * 4
    assert T < tiles.max_tiles()
    for by_table in (False, True):
        for warp in (0, 1, 77, nwarps - 1):
            left = 5
            first = warp + ((T - 1 - warp) // nwarps - left) * nwarps
            w = _walk(tiles, first, nwarps, T, 1, 1, 4, by_table, left + 4)
            k = int(w[:, 3].sum())
            assert k == left + 1 and w[:k, 3].all()
            np.testing.assert_array_equal(w[:k, 0], first + nwarps * np.arange(k))
            np.testing.assert_array_equal(w[:k, 2], w[:k, 0])


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
