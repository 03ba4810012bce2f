"""Shared scans counted by table lookup, against the oracle: every way a row's
words are held (one, two or four words a thread, many words a warp), tiles'
edges, and the forms of tests an operand's intervals must separate."""
import numpy as np
import pytest
import torch

import oracle
from tests._helpers import as_columns, host_table, random_preds

pytestmark = pytest.mark.gpu


def shared(esc, t, texts):
    ps = esc.PredicateSet(t, texts)
    dev = torch.full((len(texts),), -1, dtype=torch.int64, device="cuda")
    esc.esc_selectivity_shared_async(t.handle, ps.handles, dev)
    return dev.tolist()


@pytest.mark.parametrize("rows", [1, 511, 513, 1024, 1025, 4097, 100_003])
@pytest.mark.parametrize("npred", [32, 50, 110, 700])
def test_conjunctions(rows, npred):
    """One box a predicate: 1, 2, 4 and 22 words."""
    from paper_1901_01488_gb300 import esc
    cols = host_table(max(rows, 8), seed=rows)
    cols = {k: v[:rows] for k, v in cols.items()}
    t = esc.Table(as_columns(cols, "cuda"), rows)
    rng = np.random.default_rng(npred)
    texts = []
    for k in range(npred):
        lo = int(rng.integers(-60, 50))
        c = int(rng.integers(-(1 << 40), 1 << 40))
        texts.append([f"a BETWEEN {lo} AND {lo + int(rng.integers(0, 60))}",
                      f"c > {c} AND b IN ({k % 256}, {(k * 7) % 256}, 255, 0)",
                      f"d <= {int(rng.integers(0, 65536))} AND NOT a = {lo}",
                      f"e >= {int(rng.integers(-(1 << 31), 1 << 31))} AND udf(a, b, 97) < {int(rng.integers(-97, 97))}",
                      f"c IN ({-(1 << 63)}, {(1 << 63) - 1}, {c}, 0, -1) AND d NOT IN (1, 2, 65535)"][k % 5])
    assert shared(esc, t, texts) == [oracle.count(x, cols) for x in texts]


@pytest.mark.parametrize("rows", [777, 60_001])
def test_general_programs(rows):
    """Nested AND / OR / NOT (several boxes, some too many), constants, more
    udfs than a pass holds, moduli on both sides of 2^16 and 2^31."""
    from paper_1901_01488_gb300 import esc
    cols = host_table(rows, seed=5)
    t = esc.Table(as_columns(cols, "cuda"), rows)
    texts = []
    for x in random_preds(400, seed=91):
        try:
            esc.Predicate(t, x)
            texts.append(x)
        except esc.EscError:
            pass
    texts += [f"udf(c, e, {m}) BETWEEN {-m // 3} AND {m // 5}" for m in (1, 65535, 65536, 2**31 - 1, 2**31, 2**62 + 1)]
    texts += ["(" + " OR ".join(f"(a = {k} AND d > {k * 1000})" for k in range(-9, 9)) + ")",   # more than 16 boxes
              "TRUE", "FALSE", "NOT (a > 3 OR (b < 9 AND NOT (c > 0 OR d = 7)))"]
    assert shared(esc, t, texts) == [oracle.count(x, cols) for x in texts]


def test_many_cuts():
    """Thousands of distinct cuts (sorted on the GPU), many equal ones, and a
    single operand; the counters' planes fill up more than once."""
    from paper_1901_01488_gb300 import esc
    rows = 1_500_000
    rng = np.random.default_rng(2)
    cols = {"a": rng.integers(-(1 << 31), (1 << 31) - 1, rows).astype(np.int32),
            "c": rng.integers(-(1 << 62), 1 << 62, rows).astype(np.int64)}
    cols["a"][:4] = [-(1 << 31), (1 << 31) - 1, 0, -1]
    t = esc.Table(as_columns(cols, "cuda"), rows)
    sa, sc = np.sort(cols["a"]), np.sort(cols["c"])
    texts, want = [], []
    for k in range(2048):
        col, s, span = ("a", sa, 31) if k % 2 else ("c", sc, 62)
        lo = int(rng.integers(-(1 << span), 1 << span)) if k % 5 else 0     # every fifth shares a bound
        hi = (1 << 63) - 1 if k % 7 == 0 else lo + int(rng.integers(0, 1 << span))
        texts.append(f"{col} BETWEEN {lo} AND {hi}")
        want.append(int(np.searchsorted(s, min(hi, int(s[-1])), "right") - np.searchsorted(s, lo, "left")))
    assert shared(esc, t, texts) == want
