"""Which shared scans are looked up and which interpreted, by what there is to
look up; and the lookup at the edges of its tiles and over general programs,
on tables large enough for it."""
import numpy as np
import pytest
import torch

import oracle
from tests._helpers import as_columns, host_table, random_preds

pytestmark = pytest.mark.gpu
# six terms: more than 16 disjoint boxes
UNDECOMPOSED = "(" + " OR ".join(f"(a = {k} AND d > {k * 1000})" for k in range(6)) + ")"


def conjunction(k, rng):
    lo = int(rng.integers(-60, 50))
    c = int(rng.integers(-(1 << 40), 1 << 40))
    return [f"a BETWEEN {lo} AND {lo + int(rng.integers(0, 60))}",
            f"c > {c} AND b IN ({k % 256}, {(k * 7) % 256}, 255, 0)",
            f"d <= {int(rng.integers(0, 65536))} AND NOT a = {lo}",
            f"e >= {int(rng.integers(-(1 << 31), 1 << 31))} AND udf(a, b, 97) < {int(rng.integers(-96, 97))}",
            f"c IN ({-(1 << 63)}, {(1 << 63) - 1}, {c}, 0, -1) AND d NOT IN (1, 2, 65535)"][k % 5]


def shared(esc, rows, texts, seed=5):
    """Counts checked against the oracle; (lookup passes, interpreted passes)."""
    cols = {k: v[:rows] for k, v in host_table(max(rows, 8), seed=seed).items()}
    t = esc.Table(as_columns(cols, "cuda"), rows)
    ps = esc.PredicateSet(t, texts)
    dev = torch.full((len(texts),), -1, dtype=torch.int64, device="cuda")
    before = esc.esc_debug_shared_passes()
    esc.esc_selectivity_shared_async(t.handle, ps.handles, dev)
    after = esc.esc_debug_shared_passes()
    assert dev.tolist() == [oracle.count(x, cols) for x in texts]
    return after[0] - before[0], after[1] - before[1]


@pytest.mark.parametrize("rows,looked_up,rest,passes", [
    (50_000, 32, 0, (1, 0)), (50_000, 40, 3, (1, 1)),
    (50_000, 31, 1, (0, 1)), (50_000, 2, 30, (0, 1)), (50_000, 0, 32, (0, 1)),   # too few that decompose
    (9_999, 32, 0, (0, 1)), (9_999, 127, 0, (0, 1)), (10_000, 32, 0, (1, 0)),    # too few rows
    (9_999, 128, 0, (1, 0)), (300, 140, 5, (1, 1)), (300, 127, 20, (0, 1)), (0, 40, 0, (0, 0))])
def test_rule(rows, looked_up, rest, passes):
    from paper_1901_01488_gb300 import esc
    rng = np.random.default_rng(rows + looked_up)
    texts = [conjunction(k, rng) for k in range(looked_up)] + [UNDECOMPOSED] * rest
    assert shared(esc, rows, [texts[i] for i in rng.permutation(len(texts))]) == passes


def test_a_pass_that_leaves_a_few():
    """More udfs than a pass holds, in an order that fills pass after pass: what a full pass leaves
    for the next is too little to be looked up, and joins one interpreted pass."""
    from paper_1901_01488_gb300 import esc
    texts = [f"udf(a, d, {m}) > {m // 3}" for m in range(100, 164)]
    assert shared(esc, 20_000, texts) == (0, 1)
    texts = [f"udf(a, d, {100 + m}) > {k}" for m in range(9) for k in range(32 if m < 8 else 3)]
    assert shared(esc, 20_000, texts) == (1, 1)


@pytest.mark.parametrize("rows", [10_000, 10_239, 10_240, 10_241, 10_752, 11_263])
@pytest.mark.parametrize("npred", [32, 50, 110])
def test_tile_edges(rows, npred):
    """1, 2 and 4 words a thread; rows around multiples of the tiles' 512 and 1024."""
    from paper_1901_01488_gb300 import esc
    rng = np.random.default_rng(npred)
    assert shared(esc, rows, [conjunction(k, rng) for k in range(npred)], seed=rows) == (1, 0)


@pytest.mark.parametrize("rows", [10_001, 60_001])
def test_general_programs(rows):
    """Nested AND / OR / NOT, constants and a few udfs, all in passes of their own."""
    from paper_1901_01488_gb300 import esc
    cols = host_table(16, seed=5)
    t = esc.Table(as_columns(cols, "cuda"), 16)
    texts = []
    for x in random_preds(1500, seed=92):
        if x.count("udf(") > 1 or ("udf(" in x and ", 7)" not in x):
            continue
        try:
            esc.Predicate(t, x)
            texts.append(x)
        except esc.EscError:
            pass
    texts += ["TRUE", "FALSE", "NOT (a > 3 OR (b < 9 AND NOT (c > 0 OR d = 7)))"]
    assert len(texts) > 300
    looked_up, interpreted = shared(esc, rows, texts)
    assert looked_up >= 1 and interpreted <= 1
