"""The work a user of this parameter store has it do, as measurable cases.

`listed()` names a dozen calls and training steps, from one data point's keys to the largest batches of the
repository's workloads; `draw(rng)` gives another case of the same ranges.  `prepare` makes what a user's program has in
hand before the call (a store with rows in it, a batch), `run` makes the call(s) through the public binding, `work` says
what a pass cannot do without, `tolerance` how far two correct implementations may differ.

Every case is one of six paths:
  primitives  pull, push and (localize > 0) localize of one batch of keys on one store
  mf          one SGD minibatch of matrix factorization
  complex     one minibatch of ComplEx with AdaGrad and negative sampling
  rescal      one minibatch of RESCAL with AdaGrad and negative sampling
  sgns        one minibatch of skip-gram with negative sampling
  keymap      arbitrary 64-bit keys translated to dense ones, then pulled

mode: "ordered" (a call reads its batch after everything before it on the stream: the default of a handle),
"pipelined" (ps_set_pipelining: the keys of the batch are sorted beside earlier calls) or "host" (the batch arrives from
pinned host memory through the *_host entry points, pipelined and with ps_set_host_overlap, the way batches are streamed
in; the loss comes back to host memory).
"""
import functools
import math

import numpy as np
import torch

import paper_2002_00655_b200 as ps


# --------------------------------------------------------------------------------------------------- the cases
def _prim(name, keys, row, n, localize, workers, zipf=0.9):
    return {"name": name, "op": "primitives", "keys": keys, "row": row, "n": n, "localize": localize, "workers": workers,
            "zipf": zipf}


def listed():
    return [
        # What a worker exchanges with the store for ONE ComplEx data point (subject, relation, object, 10 negatives;
        # rows of 100 complex dimensions with their accumulators): the access pattern of the paper's own workers.
        _prim("point_13", 500_000, 400, 13, 0, 1, 1.0),
        # The small pull / push / localize batch of the tests: a worker that prefetches for a few hundred data points.
        _prim("primitives_6k", 50_000, 128, 6_000, 600, 8),
        # The large pull / push / localize batch of the benchmark (1M keys, 100k of them relocated), 16M keys of 512 bytes.
        _prim("primitives_1m", 16_000_000, 128, 1_000_000, 100_000, 64),
        # A small matrix: minibatches of 1,024 cells, rank 8, uniform columns, on a handle with its defaults.
        {"name": "mf_1k", "op": "mf", "rows": 1_000, "cols": 1_000, "rank": 8, "n": 1_024, "zipf": 0.0, "mode": "ordered"},
        # The benchmark's matrix: 10M x 1M, rank 100, Zipf columns, 65,536 cells a step, batches on the device.
        {"name": "mf_65k", "op": "mf", "rows": 10_000_000, "cols": 1_000_000, "rank": 100, "n": 65_536, "zipf": 1.1,
         "mode": "pipelined"},
        # The same with batches streamed in from pinned host memory: the end-to-end form of the headline benchmark.
        {"name": "mf_65k_host", "op": "mf", "rows": 10_000_000, "cols": 1_000_000, "rank": 100, "n": 65_536, "zipf": 1.1,
         "mode": "host"},
        # A small knowledge graph: 256 triples a step, 12 complex dimensions, on a handle with its defaults.
        {"name": "complex_256", "op": "complex", "entities": 2_000, "relations": 16, "dim": 12, "n": 256, "neg": 10,
         "mode": "ordered"},
        # The benchmark's knowledge graph: 500k entities, 100 complex dimensions, 8,192 triples with 10 negatives.
        {"name": "complex_8k", "op": "complex", "entities": 500_000, "relations": 1_000, "dim": 100, "n": 8_192, "neg": 10,
         "mode": "pipelined"},
        # The paper's large ComplEx: 4,000 complex dimensions (64 KB rows), 2,048 triples; 200k entities are held here
        # (13 GB of rows) so that two stores and a copy for comparison fit one card.
        {"name": "complex_4000", "op": "complex", "entities": 200_000, "relations": 1_000, "dim": 4_000, "n": 2_048,
         "neg": 10, "mode": "pipelined"},
        # RESCAL at the paper's sizes: 500k entities, 573 relations of 100 x 100, 8,192 triples with 10 negatives.
        {"name": "rescal_8k", "op": "rescal", "entities": 500_000, "relations": 573, "dim": 100, "n": 8_192, "neg": 10,
         "mode": "pipelined"},
        # Skip-gram at the paper's sizes: 1M words, vectors of 300, window 5, 3 negatives, 32,768 centers a step.
        {"name": "sgns_32k", "op": "sgns", "vocab": 1_000_000, "row": 300, "n": 32_768, "window": 5, "neg": 3,
         "mode": "pipelined"},
        # 1M sparse keys a batch in front of a store of 4M keys of 512 bytes; most have been met before.
        {"name": "keymap_1m", "op": "keymap", "keys": 4_000_000, "row": 128, "n": 1_000_000, "zipf": 0.9},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mode(rng):
    return rng.choice(("ordered", "pipelined", "pipelined", "host"))


def draw(rng):
    """One more case: a path, its sizes spread over the logarithm of their ranges, no larger than the listed ones."""
    op = rng.choice(("primitives", "primitives", "mf", "mf", "complex", "complex", "rescal", "sgns", "keymap"))
    if op == "primitives":
        row = 4 * _log(rng, 1, 256)
        n = _log(rng, 1, min(1_000_000, 128_000_000 // row))
        keys = max(1_000, min(16 * n, 2_000_000_000 // row)) + rng.randrange(1_000)
        loc = n // 10 if rng.random() < 0.7 else 0
        c = _prim("", keys, row, n, loc, rng.choice((2, 4, 8, 64)), round(rng.uniform(0.5, 1.1), 2))
    elif op == "mf":
        rank = 4 * _log(rng, 1, 64)
        n = _log(rng, 16, min(131_072, 6_553_600 // rank))
        rows = max(1_000, 150 * n) + rng.randrange(1_000)
        c = {"op": op, "rows": rows, "cols": max(100, rows // 10), "rank": rank, "n": n,
             "zipf": rng.choice((0.0, round(rng.uniform(0.6, 1.1), 2))), "mode": _mode(rng)}
    elif op == "complex":
        dim, neg = _log(rng, 4, 1_000), rng.choice((1, 4, 10, 10, 20))
        n = _log(rng, 16, min(8_192, 10_649_600 // (dim * (3 + neg))))
        c = {"op": op, "entities": max(1_000, 60 * n) + rng.randrange(1_000), "relations": rng.choice((16, 237, 1_000)),
             "dim": dim, "n": n, "neg": neg, "mode": _mode(rng)}
    elif op == "rescal":
        dim = 4 * rng.randrange(2, 33)
        n = _log(rng, 16, min(8_192, 81_920_000 // (dim * dim)))
        c = {"op": op, "entities": max(1_000, 60 * n) + rng.randrange(1_000), "relations": rng.choice((11, 237, 573)),
             "dim": dim, "n": n, "neg": rng.choice((4, 10)), "mode": rng.choice(("ordered", "pipelined"))}
    elif op == "sgns":
        row, window, neg = 4 * _log(rng, 4, 128), rng.randrange(2, 8), rng.randrange(2, 8)
        n = _log(rng, 64, min(32_768, 403_046_400 // (row * (1 + 2 * window * (1 + neg)))))
        c = {"op": op, "vocab": max(1_000, 30 * n) + rng.randrange(1_000), "row": row, "n": n, "window": window, "neg": neg,
             "mode": _mode(rng)}
    else:
        n = _log(rng, 16, 1_000_000)
        c = {"op": op, "keys": max(1_000, 4 * n) + rng.randrange(1_000), "row": 4 * _log(rng, 1, 32), "n": n,
             "zipf": round(rng.uniform(0.5, 1.1), 2)}
    c.pop("name", None)
    return c


# -------------------------------------------------------------------------------------------- inputs, from a seed
def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 64 + salt)
    return g


def _zipf_cdf(n, exponent):
    p = torch.arange(1, n + 1, dtype=torch.float64, device="cuda").pow_(-exponent)
    return torch.cumsum(p, 0).div_(p.sum())


def _sample(cdf, count, g):
    """Ranks with the given distribution (rank 0 the most frequent), int64."""
    u = torch.rand(count, dtype=torch.float64, device="cuda", generator=g)
    return torch.searchsorted(cdf, u).clamp_(max=cdf.numel() - 1)


def _zipf(n, exponent, count, g):
    return _sample(_zipf_cdf(n, exponent), count, g) if exponent else _uniform(n, count, g)


def _uniform(n, count, g):
    return torch.randint(0, n, (count,), device="cuda", generator=g)


def _fill(store, std, g, accumulators=False):
    """Rows N(0, std); with accumulators the second half of a row holds AdaGrad sums as they are some way into training."""
    half = store.L // 2
    step = max(1, (1 << 26) // store.L)
    for first in range(0, store.K, step):
        count = min(step, store.K - first)
        rows = torch.randn((count, store.L), device="cuda", generator=g).mul_(std)
        if accumulators:
            rows[:, half:].square_().mul_(10.0).add_(1e-3)
        store.set_rows(torch.arange(first, first + count, device="cuda"), rows)


def _store(keys, row, max_batch, workers=1, slack=1.0):
    return ps.Store(keys, row, workers, int(math.ceil(slack * -(-keys // workers))), max_batch_keys=max_batch)


def _mode_on(store, case):
    if case["mode"] != "ordered":
        ps.ps_set_pipelining(store.h, True)
    if case["mode"] == "host":
        ps.ps_set_host_overlap(store.h, True)


def _batch(case, *arrays):
    """The batch where the mode has it: device tensors, or pinned host tensors."""
    arrays = [a.contiguous() for a in arrays]
    if case["mode"] != "host":
        return arrays
    return [a.cpu().pin_memory() for a in arrays]


class _State:
    pass


def _triples(case, g):
    n, q = case["n"], case["neg"]
    cdf = _zipf_cdf(case["entities"], 1.0)
    return _batch(case, _sample(cdf, n, g).int(), _uniform(case["relations"], n, g).int(), _sample(cdf, n, g).int(),
                  _uniform(case["entities"], n * q, g).int().view(n, q),
                  torch.randint(0, 2, (n, q), device="cuda", generator=g, dtype=torch.uint8))


def prepare(case, seed):
    s = _State()
    s.case = case
    g = _gen(seed, 1)
    op, n = case["op"], case["n"]
    if op == "primitives":
        s.store = _store(case["keys"], case["row"], n, case["workers"], 1.5 if case["workers"] > 1 else 1.0)
        _fill(s.store, 1.0, g)
        s.keys = _zipf(case["keys"], case["zipf"], n, g)
        s.updates = torch.randn((n, case["row"]), device="cuda", generator=g)
        s.wanted = s.keys[:case["localize"]]
        s.turn = 0                                   # the requester changes from batch to batch
    elif op == "mf":
        s.store = _store(case["rows"] + case["cols"], case["rank"], 2 * n)
        _fill(s.store, 0.1, g)
        s.batch = _batch(case, _uniform(case["rows"], n, g).int(), _zipf(case["cols"], case["zipf"], n, g).int(),
                         torch.randn(n, device="cuda", generator=g).mul_(1.1))
    elif op == "complex":
        s.store = _store(case["entities"] + case["relations"], 4 * case["dim"], (3 + case["neg"]) * n)
        _fill(s.store, 0.1, g, accumulators=True)
        s.batch = _triples(case, g)
    elif op == "rescal":
        d = case["dim"]
        s.store = _store(case["entities"] + case["relations"] * d, 2 * d, (2 + case["neg"] + d) * n)
        _fill(s.store, 0.1, g, accumulators=True)
        s.batch = _triples(case, g)
    elif op == "sgns":
        vocab, w = case["vocab"], case["window"]
        s.store = _store(2 * vocab, case["row"], n * (1 + 2 * w * (1 + case["neg"])))
        _fill(s.store, 0.05, g)                      # vectors some way into training
        s.corpus_len = 4 * n + 2 * w
        s.first = n + w                              # a batch from the middle of the stream
        tokens = _zipf(vocab, 1.0, s.corpus_len, g).int()
        negatives = _zipf(vocab, 0.75, n * 2 * w * case["neg"], g).int()
        if case["mode"] == "host":                   # only the batch's stretch of the stream travels
            s.tok_first = s.first - w
            tokens = tokens[s.tok_first:s.first + n + w]
        s.batch = _batch(case, tokens, negatives)
    elif op == "keymap":
        keys = case["keys"]
        s.store = _store(keys, case["row"], max(n, 65_536))
        _fill(s.store, 1.0, g)
        s.map = ps.KeyMap(keys, max(n, 65_536))
        universe = torch.arange(keys, device="cuda") * -7046029254386353131      # an odd multiplier: a bijection
        met = universe[torch.randperm(keys, device="cuda", generator=g)[:keys * 3 // 4]]
        for part in met.split(max(n, 65_536)):       # what earlier batches brought
            s.map.insert(part)
        s.sparse = universe[_zipf(keys, case["zipf"], n, g)]
    if "mode" in case:
        _mode_on(s.store, case)
        if case["mode"] == "host":
            s.loss_words = torch.zeros(64, dtype=torch.float64).pin_memory()
            s.turn = 0
    torch.cuda.synchronize()
    return s


# -------------------------------------------------------------------------------------------------------- a pass
_MF = (0.002, 0.05)                     # learning rate, lambda
_ADAGRAD = (0.1, 1e-8)                  # learning rate, eps
_SGNS_LR = 2.5e-4                       # small enough that a batch seen again and again stays finite


def run(s):
    case, store = s.case, s.store
    op = case["op"]
    if op == "primitives":
        pulled = store.pull(s.keys)
        store.push(s.keys, s.updates)
        if case["localize"]:
            s.turn = (s.turn + 1) % case["workers"]
            store.localize(s.turn, s.wanted)
        return [pulled, store.store, store.table]
    if op == "keymap":
        dense = s.map.insert(s.sparse)
        return [dense, store.pull(dense)]
    host = case["mode"] == "host"
    if host:                            # every call in flight has a loss word of its own
        s.turn = (s.turn + 1) % 64
        word = s.loss_words[s.turn:s.turn + 1]
    if op == "mf":
        if host:
            ps.ps_step_mf_host(store.h, *s.batch, case["rows"], *_MF, store.loss, word)
        else:
            ps.ps_step_mf(store.h, *s.batch, case["rows"], *_MF, store.loss)
    elif op == "complex":
        if host:
            ps.ps_step_kge_host(store.h, *s.batch, case["neg"], case["entities"], case["dim"], *_ADAGRAD, store.loss, word)
        else:
            ps.ps_step_kge(store.h, *s.batch, case["neg"], case["entities"], case["dim"], *_ADAGRAD, store.loss)
    elif op == "rescal":
        ps.ps_step_rescal(store.h, *s.batch, case["neg"], case["entities"], case["dim"], *_ADAGRAD, store.loss)
    elif op == "sgns":
        if host:
            ps.ps_step_sgns_host(store.h, s.batch[0], s.tok_first, s.first, case["n"], s.corpus_len, case["window"],
                                 s.batch[1], case["neg"], case["vocab"], _SGNS_LR, store.loss, word)
        else:
            ps.ps_step_sgns(store.h, s.batch[0], s.first, case["n"], case["window"], s.batch[1], case["neg"],
                            case["vocab"], _SGNS_LR, store.loss)
    return [word if host else store.loss, store.store]


# ------------------------------------------------------------------------------- what a pass cannot do without
@functools.lru_cache(maxsize=None)
def _weights(n, exponent):
    p = np.arange(1, n + 1, dtype=np.float64) ** -exponent
    return p / p.sum()


def _distinct(n_keys, *draws):
    """Expected distinct keys among draws of (count, Zipf exponent) over the same n_keys keys."""
    miss = np.zeros(n_keys)
    for count, exponent in draws:
        miss += count * np.log1p(-np.minimum(_weights(n_keys, exponent), 1 - 1e-12))
    return float(-np.expm1(miss).sum())


def work(case):
    """Bytes: the batch arrays and a table entry (8 bytes) per distinct key read once, each distinct row read once and
    written once, what is handed back written once.  Operations: those of the method's formulas."""
    op, n = case["op"], case["n"]
    if op == "primitives":
        row = 4 * case["row"]
        u = _distinct(case["keys"], (n, case["zipf"]))
        moved = _distinct(case["keys"], (case["localize"], case["zipf"])) if case["localize"] else 0.0
        pull = 8 * n + u * (8 + row) + n * row
        push = 8 * n + n * row + u * (8 + 2 * row)
        localize = 8 * case["localize"] + moved * (16 + 8 + 2 * row)      # table entry rewritten, a slot each way
        return {"bytes": pull + push + localize, "flops": n * case["row"]}
    if op == "keymap":
        row = 4 * case["row"]
        u = _distinct(case["keys"], (n, case["zipf"]))
        return {"bytes": 8 * n + u * 12 + 2 * 8 * n + u * (8 + row) + n * row, "flops": n}
    if op == "mf":
        row = 4 * case["rank"]
        u = _distinct(case["rows"], (n, 0.0)) + _distinct(case["cols"], (n, case["zipf"]))
        return {"bytes": 12 * n + u * (8 + 2 * row), "flops": n * 14 * case["rank"]}
    if op in ("complex", "rescal"):
        q, d = case["neg"], case["dim"]
        u = _distinct(case["entities"], (2 * n, 1.0), (n * q, 0.0))
        r = _distinct(case["relations"], (n, 0.0))
        batch = n * (12 + 5 * q)
        if op == "complex":             # a score and the gradients of three roles per triple, AdaGrad per occurrence
            return {"bytes": batch + (u + r) * (8 + 8 * 4 * d), "flops": n * (3 + q) * d * 40}
        return {"bytes": batch + (u + r * d) * (8 + 4 * 4 * d), "flops": n * (8 * d * d + 10 * d * d + q * 10 * d)}
    slots = 2 * case["window"] * (1 + case["neg"])
    row = 4 * case["row"]
    out = _distinct(case["vocab"], (n * 2 * case["window"], 1.0), (n * 2 * case["window"] * case["neg"], 0.75))
    u = _distinct(case["vocab"], (n, 1.0)) + out
    return {"bytes": 4 * n * (1 + 2 * case["window"] * case["neg"]) + u * (8 + 2 * row), "flops": n * slots * 6 * case["row"]}


def tolerance(case):
    """32-bit rows whose sums per key are formed in 64 bits and rounded once: implementations differ by the rounding of
    the terms.  Location tables and dense keys are the same."""
    return {"rel": 1e-5}
