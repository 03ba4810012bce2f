"""Shared scans whose operands are searched by way of buckets, against numpy:
cuts spread evenly, crowded into one bucket, in buckets of one value, at the
ends of the types; values outside the cuts; cuts sorted on the GPU."""
import numpy as np
import pytest
import torch

from tests._helpers import as_columns

pytestmark = pytest.mark.gpu

I32 = (-(1 << 31), (1 << 31) - 1)


def bounds(kind, n, rng):
    """n (lo, hi) ranges for the i32 column, by where their cuts lie."""
    if kind == "even":
        lo = rng.integers(-(1 << 31), 1 << 31, n)
        return lo, np.minimum(lo + rng.integers(0, 1 << 30, n), I32[1])
    if kind == "crowded":      # one bucket holds all but two cuts
        lo = rng.integers(1000, 1200, n)
        lo[0] = -(1 << 30)
        hi = lo + rng.integers(0, 100, n)
        hi[1] = 1 << 30
        return lo, hi
    if kind == "single":       # a bucket per value
        lo = rng.integers(-40, 300, n)
        return lo, lo + rng.integers(0, 30, n)
    lo = rng.integers(I32[0], I32[0] + 3, n)    # the ends of the type
    hi = rng.integers(I32[1] - 2, I32[1] + 1, n)
    mid = rng.integers(-5, 5, n)
    return np.where(np.arange(n) % 3 == 0, mid, lo), np.where(np.arange(n) % 3 == 1, mid, hi)


@pytest.mark.parametrize("kind", ["even", "crowded", "single", "ends"])
@pytest.mark.parametrize("npred", [16, 40, 600, 2048])
def test_against_counting(kind, npred):
    from paper_1901_01488_gb300 import esc
    rows = 40_961
    rng = np.random.default_rng(npred)
    lo, hi = bounds(kind, npred, rng)
    a = rng.integers(I32[0], I32[1] + 1, rows).astype(np.int32)
    near = np.concatenate([lo - 1, lo, lo + 1, hi - 1, hi, hi + 1])
    a[:rows // 2] = np.clip(rng.choice(near, rows // 2), *I32).astype(np.int32)
    a[:4] = [I32[0], I32[1], 0, -1]
    c = a.astype(np.int64)
    c[::7] *= 1 << 20           # an i64 column, searched with its values saturated
    d = rng.integers(0, 65536, rows).astype(np.uint16)
    cols = {"a": a, "c": c, "d": d}
    t = esc.Table(as_columns(cols, "cuda"), rows)
    texts, want = [], []
    for k in range(npred):
        l, h = int(lo[k]), int(hi[k])
        name = ("a", "c")[k % 2]
        m = int(rng.integers(1, 500)) * 100
        texts.append(f"{name} BETWEEN {l} AND {h} AND d < {m}")
        want.append(int(((cols[name] >= l) & (cols[name] <= h) & (d < m)).sum()))
    ps = esc.PredicateSet(t, texts)
    dev = torch.full((npred,), -1, dtype=torch.int64, device="cuda")
    esc.esc_selectivity_shared_async(t.handle, ps.handles, dev)
    assert dev.tolist() == want


@pytest.mark.parametrize("rows", [9_999_999, 10_000_000])
def test_eight_predicates(rows):
    """On both sides of the size from which eight predicates are looked up."""
    from paper_1901_01488_gb300 import esc
    rng = np.random.default_rng(8)
    cols = {"a": rng.integers(-1000, 1000, rows).astype(np.int32), "b": rng.integers(0, 256, rows).astype(np.uint8)}
    t = esc.Table(as_columns(cols, "cuda"), rows)
    texts = [f"a BETWEEN {-900 + 100 * k} AND {37 * k} AND b >= {9 * k}" for k in range(8)]
    ps = esc.PredicateSet(t, texts)
    dev = torch.full((8,), -1, dtype=torch.int64, device="cuda")
    esc.esc_selectivity_shared_async(t.handle, ps.handles, dev)
    assert dev.tolist() == [int(((cols["a"] >= -900 + 100 * k) & (cols["a"] <= 37 * k) & (cols["b"] >= 9 * k)).sum())
                            for k in range(8)]


def test_largest_pass():
    """A pass at all its limits: 16 i64 columns, 24 operands, 8192 boxes, 256
    buckets for every operand, more shared memory than there is."""
    from paper_1901_01488_gb300 import esc
    rows, top = 3001, 1 << 20
    rng = np.random.default_rng(24)
    names = [f"c{k}" for k in range(16)]
    cols = {n: rng.integers(-5, top + 5, rows) for n in names}
    t = esc.Table(as_columns(cols, "cuda"), rows)
    m = 1 << 21
    values = [(n, cols[n]) for n in names]
    values += [(f"udf({names[2 * k]}, {names[2 * k + 1]}, {m})", np.fmod(cols[names[2 * k]] * cols[names[2 * k + 1]], m))
               for k in range(8)]
    texts, want = [], []
    for k in range(2048):
        ops = [values[(4 * k + j) % 24] for j in range(4)]
        lo = [1 if k < 6 else int(rng.integers(1, top - 2)) for _ in ops]    # the first six meet every operand
        hi = [top - 2 if k < 6 else int(rng.integers(x, top - 1)) for x in lo]
        texts.append(" OR ".join(f"{n} BETWEEN {a} AND {b}" for (n, _), a, b in zip(ops, lo, hi)))
        hit = np.zeros(rows, bool)
        for (_, v), a, b in zip(ops, lo, hi):
            hit |= (v >= a) & (v <= b)
        want.append(int(hit.sum()))
    ps = esc.PredicateSet(t, texts)
    dev = torch.full((2048,), -1, dtype=torch.int64, device="cuda")
    esc.esc_selectivity_shared_async(t.handle, ps.handles, dev)
    assert dev.tolist() == want
