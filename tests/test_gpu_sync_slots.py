"""Synchronous calls report through a bounded set of slots: more calls at once
than slots, on threads and streams of their own, and programs of every size."""
import threading

import numpy as np
import pytest
import torch

import oracle
from paper_1901_01488_gb300 import datagen

pytestmark = pytest.mark.gpu
TEXTS = ["price < 5000", "code7 = 3 AND day BETWEEN 100 AND 900", "udf(price, qty, 97) > 60 OR key2 > 9000000",
         "code25 IN (1, 2, 3, 20) AND NOT (code150 IN (5, 100) OR qty < 25) AND key BETWEEN 10 AND 16000000"]


def test_more_calls_than_slots():
    from paper_1901_01488_gb300 import esc
    sizes = (1, 300, 10_000, 700_001)
    tabs = [datagen.skewed_table(n, seed=90 + i, device="cuda") for i, n in enumerate(sizes)]
    etabs = [esc.Table.from_datagen(t) for t in tabs]
    hosts = [t.host() for t in tabs]
    proj = ("price", "code7")
    preds = [[esc.Predicate(t, x, proj) for x in TEXTS] for t in etabs]
    want = [[oracle.select(x, h, proj) for x in TEXTS] for h in hosts]
    dims = datagen.star_fact(50_000, 4, "cuda", (2_000, 300))
    fact = esc.Table.from_datagen(dims)
    full = [torch.full(((n + 31) // 32,), -1, dtype=torch.int32, device="cuda") for n in (2_000, 300)]
    torch.cuda.synchronize()
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        try:
            for r in range(12):
                i, j = (k + r) % len(sizes), (k // 4 + r) % len(TEXTS)
                ids, vals = want[i][j]
                if esc.count(etabs[i], preds[i][j], st) != len(ids):
                    bad.append(("count", i, j))
                with torch.cuda.stream(st):
                    rows = preds[i][j].alloc_rows(len(ids))
                    words = torch.zeros((sizes[i] + 31) // 32, dtype=torch.int32, device="cuda")
                n, _ = esc.esc_selectivity(etabs[i].handle, preds[i][j].handle, rows, st)
                c = esc.esc_bitmap_build(etabs[i].handle, preds[i][j].handle, words, st)
                got = rows[1][:n].cpu().numpy().view(np.uint32)
                bits = np.unpackbits(words.cpu().numpy().view(np.uint8), bitorder="little")[:sizes[i]]
                if n != len(ids) or c != n or not np.array_equal(got, ids) or not np.array_equal(np.flatnonzero(bits), ids):
                    bad.append(("rows", i, j))
                if esc.esc_semijoin_counts(fact.handle, ["fk0", "fk1"], full, [2_000, 300], st) != [50_000] * 4:
                    bad.append(("semijoin",))
        except Exception as e:   # noqa: BLE001
            bad.append(e)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(40)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[:3]


def test_calls_around_a_capture():
    """A count while another stream is being captured; asynchronous calls inside
    the capture, replayed."""
    from paper_1901_01488_gb300 import esc
    t = esc.Table.from_datagen(datagen.skewed_table(40_000, 5, "cuda"))
    p = [esc.Predicate(t, x) for x in TEXTS]
    want = [esc.count(t, x) for x in p]
    out = torch.zeros(len(p), dtype=torch.int64, device="cuda")
    rows = [x.alloc_rows(c + 1) for x, c in zip(p, want)]
    ids = [esc.select(t, x)[1].clone() for x in p]
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        for k, x in enumerate(p):
            esc.esc_selectivity_async(t.handle, x.handle, out[k:k + 1], rows[k] if k % 2 else None)
        assert esc.count(t, p[0], side) == want[0]
    for _ in range(2):
        out.zero_()
        for r in rows:
            r[1].fill_(-1)
        g.replay()
        assert out.tolist() == want
        for k in range(1, len(p), 2):
            assert torch.equal(rows[k][1][:want[k]], ids[k]) and rows[k][1][want[k]].item() == -1
