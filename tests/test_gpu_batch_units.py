"""Compaction units of a batch: one size for a whole write launch, from 8 to
256 groups, against the oracle at the sizes where units begin and end."""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_01488_gb300 import datagen

pytestmark = pytest.mark.gpu

# rows of the tables of one launch: alone below one unit, around a unit of 8
# groups, and next to a table large enough for units of more than 8 groups
SIZES = [(1, 255, 256, 257), (2047, 2048, 2049, 0), (300, 2_500_001, 65_537), (4_000_003, 3_999_744, 10_000)]


@pytest.mark.parametrize("sizes", SIZES)
@pytest.mark.parametrize("waves", [1, 3])
def test_batch_units(sizes, waves):
    from paper_1901_01488_gb300 import esc
    proj = datagen.SKEWED_PROJECTION
    tabs = [datagen.skewed_table(n, seed=70 + i, device="cuda") for i, n in enumerate(sizes)]
    etabs = [esc.Table.from_datagen(t) for t in tabs]
    hosts = [t.host() for t in tabs]
    # no row, few, most, all but few; a constant; one sub-query counts only
    texts = ["price < 100", "price BETWEEN 100 AND 5000", "day < 2000", "qty != 7 AND code7 != 2", "TRUE"]
    preds, tabh, expect, rows = [], [], [], []
    for i, t in enumerate(etabs):
        for j, text in enumerate(texts):
            p = esc.Predicate(t, text, proj)
            ids, vals = oracle.select(text, hosts[i], proj)
            cap = len(ids) if j != 2 else len(ids) // 2 + 1      # truncated in the middle of a unit
            preds.append(p)
            tabh.append(t.handle)
            expect.append((ids, vals))
            rows.append(None if (i, j) == (1, 1) else p.alloc_rows(cap))
    handles = [p.handle for p in preds]

    def check(counts):
        for (ids, vals), r, c in zip(expect, rows, counts):
            assert c == len(ids)
            if r is not None:
                k = min(len(ids), r[0])
                assert np.array_equal(r[1][:k].cpu().numpy().view(np.uint32), ids[:k])
                for name, col in zip(proj, r[2]):
                    assert np.array_equal(col[:k].cpu().numpy(), vals[name][:k]), name

    counts = torch.zeros(len(preds), dtype=torch.int64, device="cuda")
    b = esc.esc_batch_prepare_waves(tabh, handles, rows, waves)
    for _ in range(2):
        for r in rows:
            if r is not None:
                r[1].fill_(-1)
        esc.esc_batch_run(b, counts)
        check(counts.tolist())
    esc.esc_batch_destroy(b)
    counts.zero_()
    for r in rows:
        if r is not None:
            r[1].fill_(-1)
    esc.esc_selectivity_batch_async(tabh, handles, counts, rows)
    check(counts.tolist())
