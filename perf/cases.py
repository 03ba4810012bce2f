"""Workloads for timing the library through its public entry points.

A case is a dict of plain values; `prepare` makes what a program has in hand
(resident tables, compiled predicates, output buffers, a model), `run` makes
one pass of calls and returns their outputs, `work` states the bytes and
operations such a pass cannot do without, and `exact` gives the 64-bit value
of the outputs that are floating-point numbers.

Tables and predicates come from the package's generator: the 32 bytes/row
skewed table (i32, i64, u8 and u16 columns, Zipf keys, correlated codes),
the 1M-row single table, the star schema.  Predicates are conjunctions of one
to six terms ({=, BETWEEN, IN, OR pair, udf}) aimed at selectivities from 1e-6
to 0.9.  The predicates belong to the case; the table's values, the features
and the weights come from the seed.
"""
from __future__ import annotations

import math
import re

import numpy as np
import torch

from paper_1901_01488_gb300 import datagen
from paper_1901_01488_gb300 import esc
from paper_1901_01488_gb300.surrogate import Surrogate

H, F = 128, 64                              # the surrogate's hidden width and features
MLP_SHAPES = (("W1", (H, F)), ("b1", (H,)), ("W2", (H, H)), ("b2", (H,)), ("w3", (H,)), ("b3", (1,)))
MLP_PARAMS = sum(math.prod(s) for _, s in MLP_SHAPES)
QUERY_SELECTIVITY = 1 / 25 * 366 / 2557 * 0.1   # of the single table's predicate, columns independent
LR, BETA1, BETA2, EPS = 1e-3, 0.9, 0.999, 1e-8


def listed():
    return [
        # an optimizer counting the selections of a small dimension table, one call each: call latency
        {"name": "count_10k", "kind": "count", "rows": 10_000, "queries": 8, "first": 11_000},
        # exact counts on the large fact table, one call each
        {"name": "count_60m", "kind": "count", "rows": 60_000_000, "queries": 12, "first": 2_000},
        # a planner's step on the plain 1M-row table: the exact count, then the rows, both waited for
        {"name": "query_1m", "kind": "query", "rows": 1_000_000},
        # sub-queries materialised for the final plan on a mid-sized table of no round size
        {"name": "select_2m", "kind": "select", "rows": 2_000_003, "queries": 8, "first": 5_000},
        # the same on the large fact table, selectivities from 1e-6 to 0.9
        {"name": "select_60m", "kind": "select", "rows": 60_000_000, "queries": 12, "first": 2_100},
        # a prepared batch over tables of many sizes, replayed: every sub-query materialises
        {"name": "batch_96", "kind": "batch", "tables": "10000,200000,2000000,8000000", "queries": 96,
         "waves": 10, "first": 300_000},
        # one wave of the serving loop: requests that just arrived, every fourth materialises
        {"name": "wave_48", "kind": "wave", "tables": "10000,200000,2000000,8000000", "queries": 48,
         "first": 400_000},
        # one table's count requests of a busy serving wave, answered in one pass
        {"name": "shared_32", "kind": "shared", "rows": 8_000_000, "predicates": 32, "first": 500_000},
        # exact labels for the learned estimator: a full pass of predicates
        {"name": "shared_2048", "kind": "shared", "rows": 20_000_000, "predicates": 2048, "first": 600_000},
        # filtered-join counts of a star schema: four dimension bitmaps, then all subsets in one pass
        {"name": "star_120m", "kind": "star", "rows": 120_000_000, "dims": 4},
        # the estimator's inference over a large set of predicates
        {"name": "predict_1m", "kind": "predict", "batch": 1_000_000},
        # one training step of the estimator at its default batch: gradient and Adam
        {"name": "train_4096", "kind": "train", "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["count", "query", "select", "batch", "wave", "shared", "star", "predict", "train"])
    first = rng.randrange(1_000_000, 2_000_000_000)
    if kind == "count":
        return {"kind": kind, "rows": _log_int(rng, 10_000, 60_000_000), "queries": rng.randint(4, 12), "first": first}
    if kind == "query":
        return {"kind": kind, "rows": _log_int(rng, 10_000, 8_000_000)}
    if kind == "select":
        return {"kind": kind, "rows": _log_int(rng, 10_000, 60_000_000), "queries": rng.randint(4, 12), "first": first}
    if kind in ("batch", "wave"):
        sizes = sorted(_log_int(rng, 10_000, 8_000_000) for _ in range(rng.randint(2, 5)))
        case = {"kind": kind, "tables": ",".join(map(str, sizes)), "first": first,
                "queries": rng.randint(16, 96) if kind == "batch" else rng.randint(4, 64)}
        if kind == "batch":
            case["waves"] = rng.choice([1, 4, 10])
        return case
    if kind == "shared":
        return {"kind": kind, "rows": _log_int(rng, 100_000, 20_000_000), "predicates": _log_int(rng, 8, 2048),
                "first": first}
    if kind == "star":
        return {"kind": kind, "rows": _log_int(rng, 1_000_000, 120_000_000), "dims": rng.randint(2, 4)}
    if kind == "predict":
        return {"kind": kind, "batch": _log_int(rng, 1, 1_000_000)}
    return {"kind": kind, "batch": _log_int(rng, 32, 65_536)}


# ---------------------------------------------------------------- the workloads' inputs
def _predicates(first, n):
    """n predicates, targets log-spaced from 1e-6 to 0.9 (one predicate: the middle)."""
    if n == 1:
        return [datagen.random_predicate(first, 1e-3)]
    return datagen.skewed_predicates(n, seed0=first)


def _placed(case):
    """(table index, predicate) of a batch's sub-queries: a fixed uniform choice of tables and targets."""
    sizes = [int(s) for s in case["tables"].split(",")]
    rng = np.random.default_rng(case["first"])
    span = math.log10(0.9) + 6.0
    return sizes, [(int(rng.integers(len(sizes))),
                    datagen.random_predicate(case["first"] + j, 10.0 ** (-6.0 + span * float(rng.random()))))
                   for j in range(case["queries"])]


def _columns_read(text):
    return [c for c in datagen.SKEWED_COLUMNS if re.search(rf"\b{c}\b", text)]


def _width(columns):
    kinds = {"key": 4, "code150": 2, "code25": 1, "code7": 1, "day": 4, "price": 8, "qty": 8, "key2": 4}
    return sum(kinds[c] for c in columns)


def _materialised_bytes(count, text):
    """Output of `count` rows (id and projected values), and the projected values the predicate did not read."""
    unread = [c for c in datagen.SKEWED_PROJECTION if c not in _columns_read(text)]
    return count * (4 + _width(datagen.SKEWED_PROJECTION) + _width(unread))


def _capacity(rows, estimate):
    """Output rows reserved for a sub-query from its estimated selectivity (correlated columns exceed it)."""
    return min(rows, 1024 + int(4 * rows * estimate))


class _Buffers:
    """Output buffers for several sub-queries: one array of row ids and one per
    projected column, each sub-query with its own slice."""

    def __init__(self, capacities, projection=datagen.SKEWED_PROJECTION):
        starts, total = [], 0
        for c in capacities:
            starts.append(total)
            total += (c + 31) // 32 * 32
        size = max(32, total)
        kinds = {"key": torch.int32, "day": torch.int32, "price": torch.int64}
        self.ids = torch.zeros(size, dtype=torch.int32, device="cuda")
        self.columns = [torch.zeros(size, dtype=kinds[p], device="cuda") for p in projection]
        self.rows = [(c, self.ids[s:s + max(1, c)], [t[s:s + max(1, c)] for t in self.columns])
                     for s, c in zip(starts, capacities)]


def _star(case, seed):
    dims = datagen.STAR_DIM_ROWS[:case["dims"]]
    fact = datagen.star_fact(case["rows"], seed, "cuda", dims)
    fact.columns = fact.columns[:len(dims)]      # the measures take no part in the counts
    texts = datagen.star_dim_predicates(4, len(dims))
    tables = [esc.Table.from_datagen(datagen.star_dim(d, n, seed, "cuda")) for d, n in enumerate(dims)]
    return {"fact": esc.Table.from_datagen(fact), "dims": tables,
            "preds": [esc.Predicate(t, s) for t, s in zip(tables, texts)],
            "names": [f"fk{d}" for d in range(len(dims))], "rows": list(dims),
            "bitmaps": [torch.zeros((n + 31) // 32, dtype=torch.int32, device="cuda") for n in dims]}


def _unflatten(p):
    out, o = {}, 0
    for name, shape in MLP_SHAPES:
        n = math.prod(shape)
        out[name] = p[o:o + n].reshape(shape)
        o += n
    return out


def _model_inputs(case, seed):
    """A model in training (weights, moments, step), features and residual targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["batch"]
    model = Surrogate(esc, seed=seed)
    parts = _unflatten(model.params)
    for name in ("b1", "b2", "b3"):
        parts[name] += 0.05 * torch.randn(parts[name].shape, generator=g, device="cuda")
    model.wbf = model.params.to(torch.bfloat16).view(torch.int16).contiguous()
    x = torch.rand((n, F), generator=g, device="cuda")
    x = x * (torch.rand((n, F), generator=g, device="cuda") < 0.5)     # untested columns leave zeros
    state = {"model": model, "x": x.to(torch.bfloat16).view(torch.int16).contiguous()}
    if case["kind"] == "train":
        model.m.copy_(1e-3 * torch.randn(MLP_PARAMS, generator=g, device="cuda"))
        model.v.copy_(1e-4 * (0.5 + torch.rand(MLP_PARAMS, generator=g, device="cuda")))
        model.step = 1000
        state["target"] = 0.3 * torch.randn(n, generator=g, device="cuda")
        state["grad"] = torch.zeros(MLP_PARAMS, device="cuda")
        state["loss"] = torch.zeros(1, device="cuda")
    return state


def prepare(case, seed):
    kind = case["kind"]
    state = {"kind": kind}
    if kind in ("count", "select"):
        table = esc.Table.from_datagen(datagen.skewed_table(case["rows"], seed, "cuda"))
        preds = _predicates(case["first"], case["queries"])
        proj = datagen.SKEWED_PROJECTION if kind == "select" else ()
        state.update(table=table, preds=[esc.Predicate(table, p.text, proj) for p in preds])
        if kind == "select":
            state["out"] = _Buffers([_capacity(case["rows"], p.est) for p in preds])
            state["counts"] = torch.zeros(len(preds), dtype=torch.int64, device="cuda")
            state["words"] = list(state["counts"].split(1))
    elif kind == "query":
        table = esc.Table.from_datagen(datagen.single_table(case["rows"], seed, "cuda"))
        state.update(table=table, pred=esc.Predicate(table, datagen.SINGLE_TABLE_PREDICATE,
                                                     datagen.SINGLE_TABLE_PROJECTION),
                     out=_Buffers([_capacity(case["rows"], QUERY_SELECTIVITY)]))
    elif kind in ("batch", "wave"):
        sizes, placed = _placed(case)
        tables = [esc.Table.from_datagen(datagen.skewed_table(n, seed * 100 + i, "cuda"))
                  for i, n in enumerate(sizes)]
        wants = [kind == "batch" or j % 4 == 3 for j in range(len(placed))]
        preds = [esc.Predicate(tables[ti], p.text, datagen.SKEWED_PROJECTION if w else ())
                 for (ti, p), w in zip(placed, wants)]
        state.update(tables=tables, preds=preds, handles=[tables[ti].handle for ti, _ in placed],
                     programs=[p.handle for p in preds])
        state["out"] = _Buffers([_capacity(sizes[ti], p.est) if w else 0 for (ti, p), w in zip(placed, wants)])
        state["rows"] = [r if w else None for r, w in zip(state["out"].rows, wants)]
        state["counts"] = torch.zeros(len(preds), dtype=torch.int64, device="cuda")
        if kind == "batch":
            state["batch"] = esc.esc_batch_prepare_waves(state["handles"], state["programs"], state["rows"],
                                                         case["waves"])
            state["owner"] = _BatchOwner(state["batch"])
    elif kind == "shared":
        table = esc.Table.from_datagen(datagen.skewed_table(case["rows"], seed, "cuda"))
        texts = [p.text for p in _predicates(case["first"], case["predicates"])]
        state.update(table=table, preds=esc.PredicateSet(table, texts),
                     counts=torch.zeros(len(texts), dtype=torch.int64, device="cuda"))
    elif kind == "star":
        state.update(_star(case, seed))
    else:
        state.update(_model_inputs(case, seed))
    return state


class _BatchOwner:
    """Destroys a prepared batch with the state that holds it."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        esc.esc_batch_destroy(self.handle)


# ---------------------------------------------------------------- one pass
def run(state):
    kind = state["kind"]
    if kind == "count":
        return np.array([esc.count(state["table"], p) for p in state["preds"]], dtype=np.int64)
    if kind == "query":
        n = esc.count(state["table"], state["pred"])
        m, _ = esc.esc_selectivity(state["table"].handle, state["pred"].handle, state["out"].rows[0])
        return [n, m, state["out"].ids, *state["out"].columns]
    if kind == "select":
        for p, r, w in zip(state["preds"], state["out"].rows, state["words"]):
            esc.esc_selectivity_async(state["table"].handle, p.handle, w, r)
        return [state["counts"], state["out"].ids, *state["out"].columns]
    if kind == "batch":
        esc.esc_batch_run(state["batch"], state["counts"])
        return [state["counts"], state["out"].ids, *state["out"].columns]
    if kind == "wave":
        esc.esc_selectivity_batch_async(state["handles"], state["programs"], state["counts"], state["rows"])
        return [state["counts"], state["out"].ids, *state["out"].columns]
    if kind == "shared":
        esc.esc_selectivity_shared_async(state["table"].handle, state["preds"].handles, state["counts"])
        return state["counts"]
    if kind == "star":
        selected = [esc.esc_bitmap_build(t.handle, p.handle, b)
                    for t, p, b in zip(state["dims"], state["preds"], state["bitmaps"])]
        subsets = esc.esc_semijoin_counts(state["fact"].handle, state["names"], state["bitmaps"], state["rows"])
        return [np.array(selected, dtype=np.int64), np.array(subsets, dtype=np.int64), *state["bitmaps"]]
    model = state["model"]
    if kind == "predict":
        return model.predict(state["x"])
    grad, loss = state["grad"], state["loss"]
    grad.zero_()
    loss.zero_()
    esc.esc_mlp_grad(state["x"], state["target"], model.wbf, model.params, grad, loss)
    model.step += 1
    esc.esc_mlp_adam(model.params, model.wbf, grad, model.m, model.v, LR, model.step, BETA1, BETA2, EPS)
    return [grad, loss, model.params, model.wbf.view(torch.bfloat16), model.m, model.v]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "count" or kind == "select":
        preds = _predicates(case["first"], case["queries"])
        b = sum(case["rows"] * _width(_columns_read(p.text)) + 8 for p in preds)
        if kind == "select":
            b += sum(_materialised_bytes(case["rows"] * p.est, p.text) for p in preds)
        return {"bytes": b, "flops": 0}
    if kind == "query":
        # day, price and category read once, the key of the qualifying rows; id, key, day and price written
        return {"bytes": case["rows"] * (4 + 8 + 1 + QUERY_SELECTIVITY * (4 + 4 + 16)), "flops": 0}
    if kind in ("batch", "wave"):
        sizes, placed = _placed(case)
        b = 0
        for j, (ti, p) in enumerate(placed):
            b += sizes[ti] * _width(_columns_read(p.text)) + 8
            if kind == "batch" or j % 4 == 3:
                b += _materialised_bytes(sizes[ti] * p.est, p.text)
        return {"bytes": b, "flops": 0}
    if kind == "shared":
        read = set()
        for p in _predicates(case["first"], case["predicates"]):
            read.update(_columns_read(p.text))
        return {"bytes": case["rows"] * _width(read) + 8 * case["predicates"], "flops": 0}
    if kind == "star":
        dims = datagen.STAR_DIM_ROWS[:case["dims"]]
        # a (4 B) of every dimension, b and c (5 B) of every second; their bitmaps written and read
        b = sum(n * (4 + 5 * (d % 2)) + 2 * n / 8 for d, n in enumerate(dims))
        return {"bytes": b + case["rows"] * 4 * len(dims), "flops": 0}
    n, mac = case["batch"], H * F + H * H + H
    if kind == "predict":
        return {"bytes": n * (2 * F + 4) + 2 * MLP_PARAMS + 4 * (2 * H + 1), "flops": 2 * n * mac}
    # forward, the hidden layer's input gradient, and both weight gradients; Adam reads and writes its state
    return {"bytes": n * (2 * F + 4) + MLP_PARAMS * (2 + 4 + 4 + 3 * 8 + 2),
            "flops": 2 * n * (mac + H * H + H * H + H * F + 2 * H) + 12 * MLP_PARAMS}


# ---------------------------------------------------------------- 64-bit values
def exact(case, seed):
    if case["kind"] not in ("predict", "train"):
        return None                      # counts, row ids and copied values: whole numbers
    s = _model_inputs(case, seed)
    model = s["model"]
    x = s["x"].view(torch.bfloat16)
    w = {k: v.double() for k, v in _unflatten(model.wbf.view(torch.bfloat16)).items()}
    b = {k: v.double() for k, v in _unflatten(model.params).items() if k.startswith("b")}
    n, step = x.shape[0], 1 << 17
    if case["kind"] == "predict":
        y = torch.empty(n, dtype=torch.float64, device="cuda")
        for o in range(0, n, step):
            z1 = (x[o:o + step].double() @ w["W1"].T + b["b1"]).relu_()
            y[o:o + step] = (z1 @ w["W2"].T + b["b2"]).relu_() @ w["w3"] + b["b3"]
        return y
    g = {k: torch.zeros(shape, dtype=torch.float64, device="cuda") for k, shape in MLP_SHAPES}
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    for o in range(0, n, step):
        xs = x[o:o + step].double()
        a1 = xs @ w["W1"].T + b["b1"]
        z1 = a1.relu()
        a2 = z1 @ w["W2"].T + b["b2"]
        z2 = a2.relu()
        e = z2 @ w["w3"] + b["b3"] - s["target"][o:o + step].double()
        dy = 2.0 / n * e
        d2 = torch.outer(dy, w["w3"]) * (a2 > 0)
        d1 = (d2 @ w["W2"]) * (a1 > 0)
        loss += (e * e).sum()
        for k, v in (("W1", d1.T @ xs), ("b1", d1.sum(0)), ("W2", d2.T @ z1), ("b2", d2.sum(0)),
                     ("w3", dy @ z2), ("b3", dy.sum().reshape(1))):
            g[k] += v
    grad = torch.cat([g[k].reshape(-1) for k, _ in MLP_SHAPES])
    # the entry point takes its rates as 32-bit numbers
    lr, b1, b2, eps = (float(np.float32(v)) for v in (LR, BETA1, BETA2, EPS))
    t = model.step + 1
    m = b1 * model.m.double() + (1.0 - b1) * grad
    v = b2 * model.v.double() + (1.0 - b2) * grad * grad
    p = model.params.double() - lr * (m / (1.0 - b1 ** t)) / ((v / (1.0 - b2 ** t)).sqrt() + eps)
    return [grad, loss, p, p, m, v]
