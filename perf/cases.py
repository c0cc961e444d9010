"""The calls that the performance of this library is measured on.

Each case is one call sequence of a program that trains or serves a recommendation model whose
embedding tables share one array: a forward alone (serving), a forward and the gradient (a caller
with its own optimizer), or a forward, the fused update and a read of the weights (training).  The
shapes are the repository's named workloads (8 small tables; Criteo-Kaggle shaped, 26 tables,
d = 16; Criteo-TB shaped, 26 tables, d = 128; multi-hot bags, d = 64; the paper's micro-benchmark)
at the batch sizes that the paper trains, serves and times with.

A case is a dict:
  kind   "infer" (forward, nothing emitted for a backward), "grad" (forward + backward_grad) or
         "step" (forward + backward_update + get_weights)
  T, d, M, Z, G, B     tables, row width, array length, chunk length, start alignment, batch
  cards  the tables' sizes: "const", "kaggle" or "tb"
  bag    mean ids per bag; 1 is exactly one id, more is Poisson (empty bags among them)
  zipf   exponent of the id distribution, 0 for uniform ids
  opt, lr              optimizer of a step
  grad   upstream gradient: "normal", or "ones" (the loss is the sum of the outputs)
  det    run-to-run identical bits asked for
"""
import math

import numpy as np
import torch

from paper_2207_10731_gb300 import binding, workloads

HASH_SEED = 17


def _case(name=None, kind="step", T=26, d=128, M=2_500_000, Z=32, G=4, B=65536, cards="tb", bag=1,
          zipf=1.05, opt="adagrad", lr=0.01, grad="normal", det=False):
    c = dict(kind=kind, T=T, d=d, M=M, Z=Z, G=G, B=B, cards=cards, bag=bag, zipf=zipf, opt=opt,
             lr=lr, grad=grad, det=det)
    if name:
        c["name"] = name
    return c


def _tiny(**k):
    return _case(**{**dict(T=8, d=16, M=16384, Z=16, B=256, cards="const", zipf=0, opt="sgd",
                           lr=0.1), **k})


def _kaggle(**k):
    return _case(**{**dict(d=16, M=1 << 20, B=2048, cards="kaggle"), **k})


def _micro(**k):
    return _case(**{**dict(B=10240, opt="sgd", lr=0.1, grad="ones"), **k})


def listed():
    return [
        # a small model's training step: launches and the call's own time
        _tiny(name="tiny_step"),
        # a serving request for a few dozen users: the latency of one forward
        _kaggle(name="serve_small", kind="infer", B=32),
        # Criteo-Kaggle training at the paper's batch
        _kaggle(name="kaggle_step"),
        # Criteo-TB training at the paper's batch of 2048
        _case(name="tb_batch2k_step", B=2048, opt="sgd", lr=0.1),
        # Criteo-TB training with the large batch that data-parallel training uses per GPU
        _case(name="tb_step"),
        # multi-hot features: long bags of few hot ids
        _case(name="multihot_step", d=64, B=16384, bag=20, zipf=1.2, opt="sgd", lr=0.1),
        # little compression: an array that does not fit in L2, of which a batch touches a part
        _case(name="large_array_step", M=1 << 26, B=16384),
        # Criteo-TB serving at the paper's inference batch
        _case(name="tb_infer", kind="infer", B=16384),
        # the paper's micro-benchmark (loss = sum of the outputs), gradient for the caller's optimizer
        _micro(name="micro_grad", kind="grad"),
        # the same with short chunks, of the paper's chunk-size study
        _micro(name="micro_z8_step", Z=8),
        # block starts at any offset, as the paper prints them; an odd batch
        _case(name="tb_any_start_step", G=1, B=10007),
        # a run that has to be repeatable bit by bit; an odd batch
        _case(name="tb_repeatable_step", B=20011, det=True),
    ]


def _between(rng, lo, hi):
    """Whole number in [lo, hi], spread over the logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    f = rng.randrange(9)
    if f == 0:
        return _tiny(B=_between(rng, 33, 1024), M=_between(rng, 4096, 1 << 18),
                     kind=rng.choice(["step", "infer", "grad"]))
    if f == 1:
        return _kaggle(B=_between(rng, 512, 32768), M=_between(rng, 1 << 17, 1 << 22))
    if f == 2:
        return _case(B=_between(rng, 1024, 65536), M=_between(rng, 1 << 18, 1 << 23),
                     d=rng.choice([64, 96, 128]))
    if f == 3:
        bag = _between(rng, 2, 20)
        return _case(d=64, B=_between(rng, 512, 16384), bag=bag, zipf=rng.choice([1.05, 1.2]),
                     M=_between(rng, 1 << 19, 1 << 22), opt="sgd", lr=0.1)
    if f == 4:
        return _case(M=_between(rng, 1 << 24, 1 << 26), B=_between(rng, 4096, 16384))
    if f == 5:
        if rng.random() < 0.5:
            return _kaggle(kind="infer", B=_between(rng, 8, 16384))
        return _case(kind="infer", B=_between(rng, 128, 16384), M=_between(rng, 1 << 18, 1 << 24))
    if f == 6:
        return _micro(kind=rng.choice(["grad", "step"]), Z=rng.choice([8, 16, 32, 64]),
                      B=_between(rng, 1500, 12000))
    if f == 7:
        return _case(G=1, B=_between(rng, 1024, 16384), M=_between(rng, 1 << 19, 1 << 22))
    return _case(det=True, B=_between(rng, 1024, 32768), M=_between(rng, 1 << 19, 1 << 23))


# ---------------------------------------------------------------------------
def _cards(case):
    """The tables' sizes: part of the model, so the same for every seed."""
    rng = np.random.default_rng(7)
    if case["cards"] == "const":
        return np.full(case["T"], 1000, dtype=np.int64)
    if case["cards"] == "kaggle":
        return workloads.loguniform_cardinalities(rng, case["T"], 3, 10_000_000)
    return workloads.scaled_loguniform_cardinalities(rng, case["T"], 3, workloads.TB_CAP,
                                                     workloads.TB_TOTAL_ROWS)


def _inputs(case, seed):
    """Ids and offsets (table-major CSR), upstream gradient, weights and Adagrad accumulator."""
    T, d, B, M = case["T"], case["d"], case["B"], case["M"]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    cards = torch.from_numpy(_cards(case)).cuda()
    if case["bag"] == 1:
        lens = torch.ones(T * B, dtype=torch.int64, device="cuda")
    else:
        rate = torch.full((T * B,), float(case["bag"]), device="cuda")
        lens = torch.poisson(rate, generator=g).to(torch.int64)
    offsets = torch.zeros(T * B + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=offsets[1:])
    table = torch.arange(T, device="cuda").repeat_interleave(lens.view(T, B).sum(1))
    n = cards[table].double()
    u = torch.rand(table.numel(), dtype=torch.float64, device="cuda", generator=g)
    s = case["zipf"]
    if s == 0:
        ids = (u * n).floor()
    else:
        # ranks with density r^-s on [1/2, n + 1/2), rounded
        lo, hi = 0.5 ** (1 - s), (n + 0.5) ** (1 - s)
        ids = ((hi - lo) * u + lo).pow(1 / (1 - s)).round() - 1
    indices = torch.minimum(ids.clamp_(min=0), n - 1).to(torch.int64)
    del table, n, u
    gout = None
    if case["kind"] != "infer":
        shape = (B, T, d)
        gout = (torch.ones(shape, device="cuda") if case["grad"] == "ones"
                else torch.randn(shape, device="cuda", generator=g))
    w = torch.randn(M, device="cuda", generator=g).mul_(0.01)
    acc = None
    if case["kind"] == "step" and case["opt"] == "adagrad":
        # what earlier steps of the training left in it
        acc = torch.rand(M, device="cuda", generator=g).mul_(4).add_(1)
    return indices, offsets, gout, w, acc


def prepare(case, seed):
    indices, offsets, gout, w, acc = _inputs(case, seed)
    T, d, B = case["T"], case["d"], case["B"]
    h = binding.PSS(_cards(case), dim=d, M=case["M"], Z=case["Z"], G=case["G"], seed=HASH_SEED,
                    optimizer=case["opt"])
    if case["kind"] == "infer":
        # a serving program has no backward to prepare for
        h.set_option(binding.OPT_BACKWARD_PATH, binding.PATH_ATOMIC)
    if case["det"]:
        h.set_option(binding.OPT_DETERMINISTIC, 1)
    if acc is not None:
        h.set_state(w, acc)
    else:
        h.set_weights(w)
    torch.cuda.synchronize()
    state = dict(kind=case["kind"], h=h, indices=indices, offsets=offsets, B=B, lr=case["lr"],
                 out=torch.empty((B, T, d), device="cuda"))
    if case["kind"] == "step":
        state.update(gout=gout, weights=w)
    elif case["kind"] == "grad":
        state.update(gout=gout, grad=w)
    return state


def run(state):
    h = state["h"]
    out = h.forward(state["indices"], state["offsets"], state["B"], out=state["out"])
    if state["kind"] == "infer":
        return {"out": out}
    if state["kind"] == "grad":
        return {"out": out, "grad": h.backward_grad(state["gout"], grad=state["grad"])}
    h.backward_update(state["gout"], state["lr"])
    return {"out": out, "weights": h.get_weights(out=state["weights"])}


def work(case):
    T, d, B, M = case["T"], case["d"], case["B"], case["M"]
    nnz = T * B * case["bag"]
    touched = min(M, nnz * d)                       # elements of the array that a batch can reach
    nbytes = 8 * nnz + 8 * (T * B + 1) + 4 * touched + 4 * T * B * d
    flops = nnz * d
    if case["kind"] != "infer":
        nbytes += 4 * T * B * d                     # the upstream gradient
        flops += nnz * d
    if case["kind"] == "grad":
        nbytes += 4 * M                             # the gradient
    elif case["kind"] == "step":
        # the update reads and writes what it touches; the weights read once and written once
        nbytes += (12 if case["opt"] == "adagrad" else 4) * touched + 4 * M
        flops += (6 if case["opt"] == "adagrad" else 2) * touched
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
def _hash_parameters():
    """A and B0 of the location hash: the first two splitmix64 outputs of the seed."""
    m64, p61, s, got = (1 << 64) - 1, (1 << 61) - 1, HASH_SEED, []
    for _ in range(2):
        s = (s + 0x9E3779B97F4A7C15) & m64
        z = s
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m64
        got.append(z ^ (z >> 31))
    return 1 + got[0] % (p61 - 1), got[1] % p61


def _locations(case, t, ids):
    """Block starts [len(ids), J] of ids of table t: G * (((A*key + B0) mod (2^61-1)) mod R)."""
    p61 = (1 << 61) - 1
    A, B0 = _hash_parameters()
    J = -(-case["d"] // case["Z"])
    R = (case["M"] - min(case["Z"], case["d"])) // case["G"] + 1
    key = (ids[:, None] * case["T"] + t) * J + torch.arange(J, device=ids.device)
    # A*key mod p61 by Horner's rule over 21-bit limbs of A (keys stay below 2^36)
    x = torch.zeros_like(key)
    for limb in (A >> 42, (A >> 21) & 0x1FFFFF, A & 0x1FFFFF):
        x = ((x & ((1 << 40) - 1)) << 21) | (x >> 40)       # x * 2^21 mod p61
        x = (x + (key * limb) % p61) % p61
    return case["G"] * (((x + B0) % p61) % R)


def exact(case, seed):
    indices, offsets, gout, w, acc = _inputs(case, seed)
    T, d, B, M, Z = case["T"], case["d"], case["B"], case["M"], case["Z"]
    col = torch.arange(d, device="cuda")
    bags = torch.arange(B, device="cuda")
    out = torch.zeros((B, T, d), dtype=torch.float64, device="cuda")
    grad = torch.zeros(M, dtype=torch.float64, device="cuda")
    for t in range(T):
        off = offsets[t * B:(t + 1) * B + 1]
        lo, hi = int(off[0]), int(off[-1])
        bag_of = bags.repeat_interleave(off[1:] - off[:-1])
        for a in range(lo, hi, 1 << 16):
            b = min(hi, a + (1 << 16))
            loc = _locations(case, t, indices[a:b])
            at = loc[:, col // Z] + col % Z                   # [ids, d]
            rows = bag_of[a - lo:b - lo]
            out[:, t].index_add_(0, rows, w[at].double())
            if case["kind"] != "infer":
                grad.index_add_(0, at.reshape(-1), gout[rows, t].double().reshape(-1))
    if case["kind"] == "infer":
        return {"out": out}
    if case["kind"] == "grad":
        return {"out": out, "grad": grad}
    w64 = w.double()
    if case["opt"] == "sgd":
        return {"out": out, "weights": w64 - case["lr"] * grad}
    new = acc.double() + grad * grad
    return {"out": out, "weights": w64 - case["lr"] * grad / (new.sqrt() + 1e-10)}
