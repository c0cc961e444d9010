"""The forward at the edges of its tiles, lane groups and staged windows: one-id tiles, tiles of
empty and one-id bags, short bags, bags longer than a window, and ids outside their table.  Dyadic
inputs: every partial sum is exact, so rows and gradients equal the oracle's bit for bit."""
import random

import numpy as np
import pytest

import oracle
from paper_2207_10731_gb300 import binding, workloads as wl
from tests import gpu_util as gu

BAGS = {"one": ("one",), "zero-one": ("uniform", 0, 1), "short": ("uniform", 0, 9),
        "long": ("uniform", 200, 330)}


@pytest.mark.gpu
@pytest.mark.parametrize("signed", [False, True], ids=["unsigned", "signed"])
@pytest.mark.parametrize("bad", [False, True], ids=["valid", "bad-ids"])
@pytest.mark.parametrize("bag", list(BAGS))
@pytest.mark.parametrize("d,Z,G,B", [(128, 32, 4, 1), (128, 32, 4, 17), (64, 32, 4, 35),
                                     (16, 32, 4, 131), (20, 8, 4, 33), (128, 32, 1, 19),
                                     (32, 1, 1, 7), (128, 32, 4, 20001)])
def test_forward_edges_bit_exact(d, Z, G, B, bag, bad, signed):
    if bag == "long" and B > 200:
        pytest.skip("the oracle would take long, and the edges are the small batches'")
    w = wl.make_workload("tiny", T=5, d=d, Z=Z, G=G, M=5000, B=B, cards=("const", 60),
                         bag=BAGS[bag], ids=("zipf", 1.1), grad="dyadic", w0="dyadic")
    idx = w.indices.copy()
    if bad:
        idx[2::11] = 60
    h = binding.PSS(w.cards, dim=d, M=w.M, Z=Z, G=G, seed=w.seed, optimizer="sgd")
    o = oracle.OraclePSS(w.cards, d=d, M=w.M, Z=Z, G=G, seed=w.seed, signed=signed)
    h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_SORTED)
    h.set_option(binding.OPT_SIGNED, int(signed))
    h.set_weights(gu.cuda(w.w0))
    out = gu.host(h.forward(gu.cuda(idx), gu.cuda(w.offsets), B)).ravel()
    ref, first_bad = o.forward(w.w0, idx, w.offsets, B)
    np.testing.assert_array_equal(out, ref)
    grad = gu.host(h.backward_grad(gu.cuda(w.grad_out)))
    want = o.grad(idx, w.offsets, B, w.grad_out)
    np.testing.assert_array_equal(grad, want.astype(np.float32))
    assert h.get_error()[1] == first_bad
    h.close()


@pytest.mark.gpu
def test_forward_with_starts_far_apart():
    # G = 2^30: block starts 4 GiB apart, beyond 32-bit byte offsets
    import torch
    G, d, B = 1 << 30, 32, 100
    M = G + 32
    cards = np.array([50, 50], dtype=np.int64)
    w = torch.zeros(M, dtype=torch.float32, device="cuda")
    w[:32] = torch.arange(1.0, 33.0, device="cuda")
    w[G:] = torch.arange(101.0, 133.0, device="cuda")
    h = binding.PSS(cards, dim=d, M=M, Z=32, G=G, seed=3, optimizer="sgd")
    assert h.R == 2
    h.set_weights(w)
    idx = torch.arange(2 * B, device="cuda") % 50
    off = torch.arange(2 * B + 1, device="cuda")
    locs = h.compute_locations(idx, off, B)
    assert set(locs.tolist()) == {0, G}
    out = h.forward(idx, off, B)
    want = w[locs[:, None] + torch.arange(32, device="cuda")].view(2, B, d).transpose(0, 1)
    assert torch.equal(out, want)
    h.close()


def test_short_quotient_is_exact():
    # the forward's 32-bit reduction mod R: q from three of the four partial
    # products of s * floor((2^64 - 1) / R), then two subtractions modulo 2^32
    rnd = random.Random(5)
    m32 = (1 << 32) - 1
    Rs = [1, 2, 3, 5, 7, (1 << 30) - 1, 1 << 30, 624993, 1 << 20] + \
         [rnd.randrange(1, (1 << 30) + 1) for _ in range(300)] + \
         [rnd.randrange(1, 1 << rnd.randrange(1, 31)) for _ in range(300)]
    for R in Rs:
        inv = ((1 << 64) - 1) // R
        rh, rl = inv >> 32, inv & m32
        top = (1 << 61) - 2
        ss = [0, 1, R - 1, R, 2 * R - 1, top, top - top % R, top - top % R - 1] + \
             [rnd.randrange(0, top + 1) for _ in range(40)]
        for s in (x for x in ss if 0 <= x <= top):
            sh, sl = s >> 32, s & m32
            q = (sh * rh + ((sh * rl) >> 32) + ((sl * rh) >> 32)) & m32
            r = (sl - q * R) & m32
            r = min(r, (r - 2 * R) & m32)
            assert min(r, (r - R) & m32) == s % R, (s, R)
