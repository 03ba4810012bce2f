"""Shared scans by table lookup where their counters and indexes are largest:
bit-sliced counters (2,047 at most between flushes) that overflow many times,
two passes over a bit row, and tables of the most rows there may be.  Nearly
every row passes, so that the counters fill.  Columns repeat with a short
period: the counts over one period give those over the table."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def counts(masks, rows):
    """Rows that pass, from masks [predicates][period]."""
    q, rem = divmod(rows, masks.shape[1])
    return (q * masks.sum(1, dtype=np.int64) + masks[:, :rem].sum(1, dtype=np.int64)).tolist()


def shared(esc, t, texts):
    ps = esc.PredicateSet(t, texts)
    dev = torch.full((len(texts),), -1, dtype=torch.int64, device="cuda")
    before = esc.esc_debug_shared_passes()
    esc.esc_selectivity_shared_async(t.handle, ps.handles, dev)
    after = esc.esc_debug_shared_passes()
    assert (after[0] - before[0], after[1] - before[1]) == (1, 0)
    return dev.tolist()


@pytest.mark.parametrize("npred,boxes", [(200, 1), (700, 1), (2048, 1), (2048, 3)])
def test_counters_overflow(npred, boxes):
    """7, 22, 64 and 192 words (the last in two passes over a bit row) shared by 2 to 32 lanes."""
    from paper_1901_01488_gb300 import esc
    rows, mods = 40_000_003, (7, 11, 13)
    dtypes = {"a": torch.uint8, "b": torch.int32, "c": torch.int64}
    cols = [(n, {torch.uint8: "u8", torch.int32: "i32", torch.int64: "i64"}[dt],
             (torch.arange(rows, device="cuda") % m).to(dt)) for (n, dt), m in zip(dtypes.items(), mods)]
    t = esc.Table(cols, rows)
    r = np.arange(7 * 11 * 13)
    a, b, c = (r % m for m in mods)
    texts, masks = [], []
    for k in range(npred):
        x, y, z = k % 3, k // 3 % 4, k // 12 % 13
        if boxes == 3:
            texts.append(f"a > {x} OR b > {y} OR c != {z}")
            masks.append((a > x) | (b > y) | (c != z))
        else:
            texts.append(f"a >= {x} AND b >= {y} AND c != {z}")
            masks.append((a >= x) & (b >= y) & (c != z))
    assert shared(esc, t, texts) == counts(np.array(masks), rows)


@pytest.fixture(scope="module")
def limit():
    from paper_1901_01488_gb300 import esc
    n = esc.MAX_ROWS
    a, b = torch.empty(n, dtype=torch.uint8, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")
    step = 1 << 28
    for s in range(0, n, step):
        e = min(n, s + step)
        v = torch.arange(s, e, dtype=torch.int64, device="cuda")
        a[s:e] = v % 251
        b[s:e] = v % 241 * 1_000_003 - 120_000_000
        del v
    t = esc.Table([("a", "u8", a), ("b", "i32", b)], n)
    yield esc, n, t
    t.close()
    del a, b
    torch.cuda.empty_cache()


@pytest.mark.parametrize("npred", [8, 50, 110, 300])
def test_row_limit(limit, npred):
    """2^32 - 2^16 rows: 1, 2, 4 words a thread, and words shared by lanes."""
    esc, n, t = limit
    r = np.arange(251 * 241)
    a, b = r % 251, r % 241 * 1_000_003 - 120_000_000
    texts, masks = [], []
    for k in range(npred):
        lo, hi = k % 11, 250 - k % 7
        cut = -119_000_000 + 700_000 * (k % 17)
        texts.append(f"a BETWEEN {lo} AND {hi} AND b > {cut}")
        masks.append((a >= lo) & (a <= hi) & (b > cut))
    assert shared(esc, t, texts) == counts(np.array(masks), n)
