"""The work users have this library do, as cases that can be timed: attention over flattened tables
through the public entry points (mate_plan*, mate_attn_fwd, mate_attn_bwd, mate_cell_mean).

A case is one layer's share of a user's step:
  kind "train"  forward + backward on a batch whose plan is in hand (a plan serves every layer of a step)
  kind "infer"  forward, then the mean of the token logits per table cell (cell selection)
  kind "batch"  a batch that has just arrived: plan, forward, backward
pattern: "exact" (row / column heads), "bucketed" (global section + buckets of `radius`), "sat" (row or
column, one pattern for all heads), "packed" (examples of different length without padding).
"""
import math

import numpy as np
import torch

import paper_2109_04312_b200 as mate

_DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, kind, B, N, P, rows, cols, H=12, d=64, dtype="bf16", pattern="exact", law="geometric", param=0.45,
          cap=16, merged=0.0, glob=0, radius=0):
    return {"name": name, "kind": kind, "pattern": pattern, "dtype": dtype, "B": B, "H": H, "N": N, "d": d, "P": P,
            "rows": rows, "cols": cols, "law": law, "param": param, "cap": cap, "merged": merged, "glob": glob,
            "radius": radius}


def listed():
    return [
        # the smallest call there is: a question and a 4 x 3 table in single precision (a unit test, a gradient
        # check, a notebook); nothing but latency
        _case("tiny_f32_train", "train", 1, 40, 8, 4, 3, H=4, d=16, dtype="f32", law="uniform", param=4.0, cap=4),
        # one question about one table arrives at a server: one example, a BERT-base layer, forward only
        _case("serve_one_table", "infer", 1, 512, 64, 16, 8, param=0.5, cap=8),
        # fine-tuning of a BERT-base sized model on ordinary tables
        _case("bert_train", "train", 8, 512, 64, 16, 8, param=0.5, cap=8),
        # tables of the size the paper trains on (2048 tokens)
        _case("medium_train", "train", 4, 2048, 128, 64, 10, param=0.4, cap=12),
        # a long document with a big table: inference ...
        _case("long_infer", "infer", 1, 8192, 256, 400, 8),
        # ... and training (the largest sequence)
        _case("long_train", "train", 1, 8192, 256, 400, 8),
        # cells of very different length and merged rows: segments are skewed
        _case("skew_train", "train", 2, 4096, 128, 120, 30, H=16, law="zipf", param=1.2, cap=64, merged=0.1),
        # examples of different length in one batch, stored one behind the other
        _case("packed_train", "train", 12, 1021, 97, 64, 9, pattern="packed", cap=12),
        # the paper's efficient variant with its constants (G = 116, R = 42)
        _case("bucketed_train", "train", 4, 2048, 64, 64, 10, pattern="bucketed", param=0.4, cap=12, glob=116,
              radius=42),
        # one pattern for all heads: same row or same column
        _case("sat_train", "train", 2, 1024, 96, 40, 9, pattern="sat", param=0.5, cap=12),
        # a training step meets a new batch of tables: the plan is part of the step
        _case("new_batch", "batch", 4, 2048, 128, 64, 10, param=0.4, cap=12),
        # single precision throughout (debugging a model, comparing against a reference)
        _case("f32_train", "train", 2, 512, 64, 16, 8, dtype="f32", param=0.5, cap=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the whole range of the listed ones, odd and ragged ones included."""
    most = max(work(c)["flops"] for c in listed())
    most_f32 = max(work(c)["flops"] for c in listed() if c["dtype"] == "f32")
    while True:
        what = rng.choice(["train"] * 4 + ["infer"] * 3 + ["packed", "bucketed", "sat", "batch", "batch", "plain", "plain"])
        plain = what == "plain"  # single precision, or a head size other than 64: small models and checks
        N = _log_int(rng, 40, 512) if plain else _log_int(rng, 96, 8192)
        B = rng.randint(1, max(1, min(16, 16384 // N)))
        P = min(N, _log_int(rng, 8, max(9, min(256, N // 4))))
        cols = rng.randint(3, 30)
        cell = rng.uniform(1.6, 3.0)  # mean tokens per cell
        rows = max(2, int((N - P) / (cols * cell) * (1.4 if what == "packed" else rng.uniform(0.8, 1.3))))
        c = _case("", "train", B, N, P, rows, cols, H=rng.choice([4, 8, 12, 12, 16]), param=1.0 / cell,
                  cap=rng.choice([8, 12, 16]))
        if rng.random() < 0.2:
            c.update(law="zipf", param=1.2, cap=64, merged=0.1)
        if plain:
            c.update(d=rng.choice([16, 32, 64, 128]), dtype="f32")
            if c["d"] != 64 and rng.random() < 0.5:
                c["dtype"] = "bf16"
        elif what in ("infer", "batch"):
            c["kind"] = what
        elif what == "packed":
            c["pattern"] = "packed"
        elif what == "bucketed":
            c.update(pattern="bucketed", glob=P + rng.randint(0, 64), radius=rng.randint(24, 96))
            c["glob"] = min(c["glob"], N)
        elif what == "sat":
            c["pattern"] = "sat"
        if work(c)["flops"] <= (most_f32 if plain else most):
            del c["name"]
            return c


def _cell_lengths(c, rng, n):
    if c["law"] == "uniform":
        return rng.integers(1, int(c["param"]) + 1, size=n)
    if c["law"] == "zipf":
        k = np.arange(1, c["cap"] + 1)
        p = k ** -float(c["param"])
        return rng.choice(k, size=n, p=p / p.sum())
    return np.minimum(rng.geometric(c["param"], size=n), c["cap"])


def _table(c, rng, n_tokens):
    """(row ids, column ids) of at most n_tokens table tokens, row by row, ids from 1."""
    lens = _cell_lengths(c, rng, c["rows"] * c["cols"]).reshape(c["rows"], c["cols"])
    merged = rng.random(c["rows"]) < c["merged"]  # such a row is one cell under the first column
    lens[merged, 1:] = 0
    r, k = np.meshgrid(np.arange(1, c["rows"] + 1), np.arange(1, c["cols"] + 1), indexing="ij")
    return np.repeat(r.ravel(), lens.ravel())[:n_tokens], np.repeat(k.ravel(), lens.ravel())[:n_tokens]


def _structure(c, seed):
    """Row and column ids of every example, and its prefix length: prefix, table, and (unless packed)
    padding up to N.  Of a packed batch the lengths belong to the case, the tables to the seed."""
    rng = np.random.default_rng(seed)
    lengths = np.random.default_rng(c["N"])
    out = []
    for b in range(c["B"]):
        N, P = c["N"], c["P"]
        if c["pattern"] == "packed":  # from a quarter of the longest length up to all of it
            N = N if b == 0 else int(lengths.integers(max(1, N // 4), N + 1))
            P = min(N, int(lengths.integers(max(1, P // 2), P + 1)))
        r, k = _table(c, rng, N - P)
        if c["pattern"] == "packed" and len(r) < N - P:  # the last cell takes what is left
            r, k = (np.concatenate([x, np.full(N - P - len(x), x[-1])]) for x in (r, k))
        ids = np.full((2, N), -1, np.int32)
        ids[:, :P] = 0
        ids[0, P:P + len(r)], ids[1, P:P + len(r)] = r, k
        out.append((ids[0], ids[1], P))
    return out


def _pairs(c, r, k, P):
    """Unmasked (query, key) pairs of one example, summed over its heads."""
    nv = int((r >= 0).sum())
    G = min(max(P, c["glob"]), nv)
    tr, tk = r[P:nv].astype(np.int64), k[P:nv].astype(np.int64)
    per_view = []
    for ids in (tr, tk):
        ids = np.sort(ids)[G - P:]
        seg = np.bincount(ids) if len(ids) else np.zeros(1, np.int64)
        if c["radius"]:
            n = len(ids)
            t = np.arange(n)
            first = np.searchsorted(ids, ids)
            last = np.searchsorted(ids, ids, side="right")
            w = t // c["radius"] * c["radius"]
            own = np.minimum(last, w + 2 * c["radius"]) - np.maximum(first, w - c["radius"])
            per_view.append(int(own.sum()))
        else:
            per_view.append(int((seg.astype(np.int64) ** 2).sum()))
    base = G * nv + (nv - G) * G
    if c["pattern"] == "sat":
        cell = np.bincount(tr * (c["cols"] + 1) + tk) if len(tr) else np.zeros(1, np.int64)
        return c["H"] * (base + sum(per_view) - int((cell.astype(np.int64) ** 2).sum()))
    n_row = c["H"] // 2
    return n_row * (base + per_view[0]) + (c["H"] - n_row) * (base + per_view[1])


def work(case):
    c = case
    ex = _structure(c, 0)
    pairs = sum(_pairs(c, r, k, P) for r, k, P in ex)
    tokens = sum(len(r) for r, _, _ in ex)
    size = {"bf16": 2, "f32": 4}[c["dtype"]]
    tensor, stat = tokens * c["H"] * c["d"] * size, tokens * c["H"] * 4
    if c["kind"] == "infer":  # Q, K, V -> O, LSE; logits, ids -> mean, count
        cells = c["B"] * (c["rows"] + 1) * (c["cols"] + 1)
        return {"bytes": 4 * tensor + stat + 12 * tokens + 8 * cells, "flops": 4 * c["d"] * pairs}
    # Q, K, V, dO -> O, LSE, dQ, dK, dV (and, for a new batch, the ids)
    return {"bytes": 8 * tensor + stat + (8 * tokens if c["kind"] == "batch" else 0), "flops": 14 * c["d"] * pairs}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    return {"rel": 1e-2}


def prepare(case, seed):
    c = case
    ex = _structure(c, seed)
    n_row = c["H"] // 2
    s = {"kind": c["kind"], "pattern": c["pattern"], "head_view": [0] * n_row + [1] * (c["H"] - n_row), "c": c}
    packed = c["pattern"] == "packed"
    cat = np.concatenate if packed else np.stack
    s["row_ids"] = torch.from_numpy(cat([e[0] for e in ex])).cuda()
    s["col_ids"] = torch.from_numpy(cat([e[1] for e in ex])).cuda()
    s["prefix"] = [e[2] for e in ex]
    s["cu"] = np.concatenate([[0], np.cumsum([len(e[0]) for e in ex])])
    shape = (c["H"], int(s["cu"][-1]), c["d"]) if packed else (c["B"], c["H"], c["N"], c["d"])
    g = torch.Generator(device="cuda").manual_seed(seed)

    def values():
        return (torch.randn(shape, device="cuda", generator=g) * 0.5).to(_DTYPES[c["dtype"]])

    s["Q"], s["K"], s["V"] = values(), values(), values()
    if c["kind"] == "infer":
        s["logits"] = torch.randn((c["B"], c["N"]), device="cuda", generator=g)
    else:
        s["dO"] = values()
    if c["kind"] != "batch":
        s["plan"] = _plan(s)
    return s


def _plan(s):
    c = s["c"]
    if s["pattern"] == "packed":
        return mate.mate_plan_packed(s["row_ids"], s["col_ids"], s["cu"], s["prefix"], s["head_view"], c["rows"], c["cols"])
    if s["pattern"] == "bucketed":
        return mate.mate_plan_bucketed_global(s["row_ids"], s["col_ids"], c["P"], c["glob"], s["head_view"], c["radius"],
                                              c["rows"], c["cols"])
    if s["pattern"] == "sat":
        return mate.mate_plan_sat(s["row_ids"], s["col_ids"], c["P"], c["H"], c["rows"], c["cols"])
    return mate.mate_plan(s["row_ids"], s["col_ids"], c["P"], s["head_view"], c["rows"], c["cols"])


def run(state):
    s = state
    plan = s["plan"] if s["kind"] != "batch" else _plan(s)
    O, LSE = mate.mate_attn_fwd(plan, s["Q"], s["K"], s["V"])
    if s["kind"] == "infer":
        mean, count = mate.mate_cell_mean(plan, s["logits"], s["col_ids"])
        return {"O": O, "LSE": LSE, "mean": mean, "count": count}
    dQ, dK, dV = mate.mate_attn_bwd(plan, s["Q"], s["K"], s["V"], O, LSE, s["dO"])
    return {"O": O, "LSE": LSE, "dQ": dQ, "dK": dK, "dV": dV}
