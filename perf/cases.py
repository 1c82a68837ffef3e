"""What the framework is timed on: the passes a recommendation model has it do, from one small
serving request to the largest training batches.

A pass goes through the package's public calls as a training or serving loop makes them: a lookup
(`robe_forward`), or a lookup and the backward of the same ids with the update fused in
(`robe_backward`, `robe_forward_keep` + `robe_backward_kept`, `robe_backward_adam`,
`robe_backward_adagrad`) or exchanged first (`dp.robe_dp_step` on one rank).  The gradient of the
output rows is an input: the model that produces it is not part of the framework.

Sizes are those of the repository's own workloads (`synth.workload`), whose shapes come from the
paper: 26 tables; rows of 16 elements on a 540 K array (Criteo Kaggle) or of 128 on 25 M (Criteo TB).
"""
import math

import torch

import paper_2108_02191_b200 as robe
from paper_2108_02191_b200 import dp

LR = 0.01  # of the plain SGD steps: with unit gradients an update is the size of the parameters


def _case(name, do, T, d, Z, M, batch, vocab, **more):
    """A case with its options at their defaults unless given.

    do       "infer": lookup only;  "atomic": lookup + atomic backward with SGD;  "binned", "det":
             lookup that keeps its block starts + binned / deterministic backward with SGD on them;
             "adam", "adagrad": lookup + deterministic backward with that optimizer;
             "dense": lookup + data-parallel step (dense gradient, exchange, dense SGD)
    vocab    (smallest, largest) table; sizes in between are spread over their logarithm
    zipf     ids follow Zipf(1.05) instead of being uniform
    bag      mean ids per bag (Poisson, clipped to [1, 4 bag]); 0: one id per table and sample"""
    c = dict(name=name, do=do, T=T, d=d, Z=Z, M=M, batch=batch, vocab_lo=vocab[0], vocab_hi=vocab[1],
             zipf=False, bag=0, array="f32", ids="int64", table_major=False, sign=False)
    c.update(more)
    return c


KAGGLE = (3, 10_131_227)  # smallest and largest table of the Kaggle data
TB = (3, 40_000_000)      # of the terabyte data


def listed():
    return [
        # one request of an online ranker: a few hundred candidates looked up at once, latency counts
        _case("serve_small", "infer", 26, 16, 8, 540_000, 128, KAGGLE, zipf=True),
        # the smallest training step: a toy model, or the last shard of an epoch
        _case("train_tiny", "atomic", 4, 16, 4, 4096, 256, (100, 2000)),
        # bulk scoring with the 100 MB model in place of 100 GB of tables
        _case("infer_zipf", "infer", 26, 128, 32, 25_000_000, 65_536, TB, zipf=True),
        # the same on half-precision parameters, ids as 32-bit per-table lists laid end to end
        _case("infer_bf16", "infer", 26, 128, 32, 25_000_000, 131_072, (10_000_000, 10_000_000),
              array="bf16", ids="int32", table_major=True),
        # an array far beyond the L2: the mildest compression, every block comes from memory
        _case("infer_10g", "infer", 26, 128, 32, 2_500_000_000, 131_072, (10_000_000, 10_000_000)),
        # a training step with one block per row, the layout with the fewest memory fetches
        _case("train_z128", "atomic", 26, 128, 128, 25_000_000, 32_768, TB, zipf=True),
        # a training step with every element hashed on its own (feature hashing as in HashedNet)
        _case("train_z1", "atomic", 26, 128, 1, 25_000_000, 32_768, TB, zipf=True),
        # multi-hot features (click histories) summed per bag, 1 GB array, fastest training step
        _case("train_multihot", "binned", 26, 64, 16, 250_000_000, 16_384, (1_000_000, 1_000_000), bag=20),
        # the same step bit-reproducible from run to run
        _case("train_multihot_det", "det", 26, 64, 16, 250_000_000, 16_384, (1_000_000, 1_000_000), bag=20),
        # the small model as the paper trains it, with Adam
        _case("train_adam", "adam", 26, 16, 8, 540_000, 16_384, KAGGLE, zipf=True),
        # data-parallel training with signed rows of a length no power of two fits, short last block
        _case("train_dp_ragged", "dense", 7, 100, 32, 1_000_003, 3001, (1000, 1_000_000), bag=4, sign=True),
        # long rows, as wider towers use, small tables beside large ones
        _case("train_long_rows", "atomic", 13, 256, 64, 25_000_000, 16_384, (1000, 10_000_000)),
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))


# array lengths that each listed case stands for
_ARRAYS = {
    "serve_small": (4096, 4_000_000), "train_tiny": (4096, 500_000), "train_adam": (50_000, 4_000_000),
    "train_dp_ragged": (50_000, 4_000_000), "infer_10g": (50_000_000, 2_500_000_000),
    "train_multihot": (10_000_000, 250_000_000), "train_multihot_det": (10_000_000, 250_000_000),
}


def draw(rng):
    c = dict(rng.choice(listed()))
    name = c.pop("name")
    most = c["T"] * c["d"] * c["batch"] * max(1, c["bag"])  # elements looked up: never more than listed
    c["T"] = rng.randint(2, 26)
    if c["d"] > 128:
        c["d"] = rng.randint(129, 256)
    else:
        c["d"] = rng.choice((16, 32, 64, 128, rng.randint(8, 128), rng.randint(8, 128)))
    if name == "train_z1":
        c["Z"] = rng.choice((1, 2, 4))
    elif name == "train_z128":
        c["Z"] = c["d"]
    elif name == "train_dp_ragged":
        c["Z"] = rng.randint(4, c["d"])
    else:
        c["Z"] = rng.choice([z for z in (8, 16, 32, 64, 128) if z <= c["d"]])
    c["M"] = _log(rng, *_ARRAYS.get(name, (262_144, 25_000_000)))
    if c["bag"]:
        c["bag"] = rng.randint(2, 20)
    if c["do"] in ("det", "binned"):
        most = most * min(16, c["Z"]) // 16  # nor more blocks to sort
    if name == "serve_small":
        c["batch"] = _log(rng, 1, 512)
    else:
        fits = min(262_144, max(1, most // (c["T"] * c["d"] * max(1, c["bag"]))))
        c["batch"] = _log(rng, max(1, min(fits, c["batch"] // 32)), fits)
    c["vocab_hi"] = _log(rng, max(1000, c["vocab_lo"]), max(1000, c["vocab_hi"]))
    c["vocab_lo"] = min(c["vocab_lo"], c["vocab_hi"])
    c["zipf"] = rng.random() < 0.5
    c["ids"] = rng.choice(("int64", "int32"))
    c["table_major"] = rng.random() < 0.3
    if c["do"] == "infer":
        c["array"] = rng.choice(("f32", "f32", "bf16"))
    if c["do"] == "adam":
        c["do"] = rng.choice(("adam", "adagrad"))
    if c["sign"]:
        c["sign"] = rng.random() < 0.5
    return c


# -- inputs ---------------------------------------------------------------------------------

_S = 1.05       # Zipf exponent
_HEAD = 4096    # ranks whose weight is summed term by term; beyond, by the midpoint integral


def _vocab(c):
    lo, hi, T = c["vocab_lo"], c["vocab_hi"], c["T"]
    return [int(round(lo * (hi / lo) ** (e / max(1, T - 1)))) for e in range(T)]


def _zipf_head():
    total, cdf = 0.0, []
    for r in range(1, _HEAD + 1):
        total += r ** -_S
        cdf.append(total)
    return cdf


_CDF = _zipf_head()
_EDGE = (_HEAD + 0.5) ** (1 - _S)


def _zipf_total(v):
    return _CDF[v - 1] if v <= _HEAD else _CDF[-1] + (_EDGE - (v + 0.5) ** (1 - _S)) / (_S - 1)


def _draw_ids(c, table, gen):
    """One id per entry of `table` (the table each position belongs to)."""
    dev = table.device
    v = torch.tensor(_vocab(c), dtype=torch.float64, device=dev)[table]
    u = torch.rand(table.numel(), dtype=torch.float64, device=dev, generator=gen)
    if not c["zipf"]:
        return (u * v).long()
    head = torch.tensor(_CDF, dtype=torch.float64, device=dev)
    u *= torch.tensor([_zipf_total(n) for n in _vocab(c)], dtype=torch.float64, device=dev)[table]
    rank = torch.searchsorted(head, u, right=True)
    left = (_EDGE - (u - _CDF[-1]).clamp_(min=0.0) * (_S - 1)).clamp_(min=1e-12)
    tail = (left ** (1 / (1 - _S)) - 0.5).floor().long()
    return torch.minimum(torch.where(rank < _HEAD, rank, tail), v.long() - 1)


class State:
    """What a user's program holds between calls: the handle, the array and the buffers it reuses."""

    def __init__(self, c, seed):
        dev = torch.device("cuda")
        gen = torch.Generator(dev).manual_seed(seed)
        T, B, d, M = c["T"], c["batch"], c["d"], c["M"]
        self.do, self.batch, self.step = c["do"], B, 0
        bags = torch.arange(B * T, device=dev)
        table = torch.div(bags, B, rounding_mode="floor") if c["table_major"] else bags % T
        self.offsets = None
        if c["bag"]:
            mean = torch.full((B * T,), float(c["bag"]), device=dev)
            lengths = torch.poisson(mean, generator=gen).clamp_(1, 4 * c["bag"]).long()
            self.offsets = torch.zeros(B * T + 1, dtype=torch.int64, device=dev)
            torch.cumsum(lengths, 0, out=self.offsets[1:])
            table = torch.repeat_interleave(table, lengths)
        self.indices = _draw_ids(c, table, gen).to(getattr(torch, c["ids"]))
        self.array = torch.empty(M, device=dev).uniform_(-0.01, 0.01, generator=gen)
        if c["array"] == "bf16":
            self.array = self.array.to(torch.bfloat16)
        shape = (T, B, d) if c["table_major"] else (B, T, d)
        self.out = torch.empty(shape, device=dev)
        self.h = h = robe.robe_create(M, c["Z"], d, T, 0x0B0E)
        robe.robe_attach_array(h, self.array)
        if c["table_major"]:
            robe.robe_set_option(h, robe.ROBE_OPT_BAG_LAYOUT, robe.ROBE_BAGS_TABLE_MAJOR)
        if c["sign"]:
            robe.robe_set_option(h, robe.ROBE_OPT_SIGN, 1)
        if self.do == "infer":
            return
        self.grad_out = torch.empty(shape, device=dev).normal_(generator=gen)
        mode = {"atomic": robe.ROBE_BWD_ATOMIC, "dense": robe.ROBE_BWD_ATOMIC, "binned": robe.ROBE_BWD_BINNED}
        robe.robe_set_option(h, robe.ROBE_OPT_BWD_MODE, mode.get(self.do, robe.ROBE_BWD_DETERMINISTIC))
        size = robe.robe_backward_workspace_bytes(h, B, self.indices.numel())
        self.workspace = torch.empty(size, dtype=torch.uint8, device=dev) if size else None
        if self.do == "dense":
            self.grad_array = torch.zeros(M, device=dev)
        if self.do in ("adam", "adagrad"):
            self.moments = [torch.zeros(M, device=dev) for _ in range(2 if self.do == "adam" else 1)]

    def __del__(self):
        if hasattr(self, "h"):
            robe.robe_destroy(self.h)


def prepare(case, seed):
    return State(case, seed)


def run(s):
    if s.do in ("binned", "det"):
        robe.robe_forward_keep(s.h, s.indices, s.offsets, s.batch, s.out, s.workspace)
        robe.robe_backward_kept(s.h, s.grad_out, s.indices, s.offsets, s.batch, None, LR, s.workspace)
        return {"out": s.out, "array": s.array}
    robe.robe_forward(s.h, s.indices, s.offsets, s.batch, s.out)
    if s.do == "infer":
        return s.out
    if s.do == "atomic":
        robe.robe_backward(s.h, s.grad_out, s.indices, s.offsets, s.batch, None, LR, s.workspace)
    elif s.do == "dense":
        dp.robe_dp_step(s.h, s.grad_out, s.indices, s.offsets, s.batch, s.grad_array, LR)
        return {"out": s.out, "array": s.array, "grad_array": s.grad_array}
    elif s.do == "adam":
        s.step += 1
        robe.robe_backward_adam(s.h, s.grad_out, s.indices, s.offsets, s.batch, *s.moments, 1e-3, 0.9, 0.999,
                                1e-8, s.step, s.workspace)
    else:
        robe.robe_backward_adagrad(s.h, s.grad_out, s.indices, s.offsets, s.batch, *s.moments, LR, 1e-10,
                                   s.workspace)
    return {"out": s.out, "array": s.array, "moments": getattr(s, "moments", None)}


# -- what a pass cannot do without ----------------------------------------------------------

def _distinct(n, v, zipf):
    """Expected number of different ids among n draws from a table of v."""
    if not zipf:
        return v * -math.expm1(-n / v)
    total, seen, lo = _zipf_total(v), 0.0, 1.0
    while lo <= v:  # ranks [lo, hi) share about one probability
        hi = min(v + 1.0, max(lo + 1.0, lo * 1.05))
        mid = 0.5 * (lo + hi - 1.0)
        seen += (hi - lo) * -math.expm1(-n * mid ** -_S / total)
        lo = hi
    return seen


def work(case):
    """Ids, offsets, output rows and gradient rows once; the part of the array that the ids reach
    read once, and with an update written once, with the optimizer's state likewise."""
    c = case
    bags = c["batch"] * c["T"]
    nnz = bags * max(1, c["bag"])
    ids = sum(_distinct(nnz / c["T"], v, c["zipf"]) for v in _vocab(c))
    slots = c["M"] * -math.expm1(-ids * c["d"] / c["M"])
    size = 2 if c["array"] == "bf16" else 4
    total = nnz * (4 if c["ids"] == "int32" else 8) + 4 * bags * c["d"] + slots * size
    if c["bag"]:
        total += 8 * (bags + 1)
    flops = nnz * c["d"] if c["bag"] else 0
    if c["do"] != "infer":
        states = {"adam": 3, "adagrad": 2}.get(c["do"], 1)
        total += 4 * bags * c["d"] + slots * 4 + (states - 1) * slots * 8
        flops += nnz * c["d"] + 2 * slots
    if c["do"] == "dense":  # the dense gradient is an output of its own, left at zero
        total += 4 * c["M"]
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Lookups and deterministic updates are defined to the bit; atomic ones add in any order in fp32."""
    return {"rel": 1e-5} if case["do"] in ("atomic", "binned", "dense") else "exact"
