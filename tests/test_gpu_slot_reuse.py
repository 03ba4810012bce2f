"""Call slots after an expired wait: the call reports it, and no later call
meets what its launch left in the slot.  The expiry's marks are put there
from the host (esc_debug_taint_slot)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_01488_gb300 import datagen

pytestmark = pytest.mark.gpu
ROWS = 3_000_017      # many more work units than blocks: the blocks have work left when they see the flag
TEXT = "day BETWEEN 200 AND 1500 AND code25 != 3"


@pytest.fixture(scope="module")
def world():
    from paper_1901_01488_gb300 import build
    build.build()
    from paper_1901_01488_gb300 import esc
    t = datagen.skewed_table(ROWS, seed=31, device="cuda")
    tbl = esc.Table.from_datagen(t)
    ids, vals = oracle.select(TEXT, t.host(), ("price",))
    return esc, tbl, ids, vals["price"]


def call(esc, tbl, kind, n):
    p = esc.Predicate(tbl, TEXT, ("price",) if kind == "select" else ())
    if kind == "count":
        return esc.count(tbl, p), None, None
    if kind == "bitmap":
        words = torch.zeros((ROWS + 31) // 32, dtype=torch.int32, device="cuda")
        return esc.esc_bitmap_build(tbl.handle, p.handle, words), words, None
    rows = p.alloc_rows(n)
    return esc.esc_selectivity(tbl.handle, p.handle, rows)[0], rows[1], rows[2][0]


def check(kind, got, ids, vals):
    assert got[0] == len(ids)
    if kind == "bitmap":
        bits = np.unpackbits(got[1].cpu().numpy().view(np.uint8), bitorder="little")[:ROWS]
        assert np.array_equal(np.flatnonzero(bits), ids)
    if kind == "select":
        assert np.array_equal(got[1].cpu().numpy().view(np.uint32), ids)
        assert np.array_equal(got[2].cpu().numpy(), vals)


@pytest.mark.parametrize("kind,when", [("count", 1), ("bitmap", 1), ("count", 2), ("bitmap", 2), ("select", 2)])
def test_expired_call(world, kind, when):
    esc, tbl, ids, vals = world
    check(kind, call(esc, tbl, kind, len(ids)), ids, vals)
    for _ in range(40):                              # more often than there are slots
        esc.esc_debug_taint_slot(when)
        with pytest.raises(esc.EscError) as ei:
            call(esc, tbl, kind, len(ids))
        assert ei.value.status == esc.ESC_ETIMEOUT
        check(kind, call(esc, tbl, kind, len(ids)), ids, vals)
    torch.cuda.synchronize()


def test_hook_is_off_by_default(world):
    esc, tbl, ids, vals = world
    with pytest.raises(esc.EscError):
        esc.esc_debug_taint_slot(3)
    esc.esc_debug_taint_slot(1)
    esc.esc_debug_taint_slot(0)
    check("count", call(esc, tbl, "count", len(ids)), ids, vals)


def test_materialising_after_an_expired_scan(world):
    """The write pass over a bitmap that the scan did not finish (what its
    memory held before is there instead): no row past the table, nothing
    past the buffers."""
    esc, tbl, ids, vals = world
    rows = ROWS // 256 * 256 + 10                    # the last group's other rows are set in what memory holds
    small = datagen.skewed_table(rows, seed=32, device="cuda")
    stbl = esc.Table.from_datagen(small)
    p, every = esc.Predicate(stbl, TEXT, ("price",)), esc.Predicate(tbl, "day >= 0 AND code25 < 200", ())
    for _ in range(4):
        out = every.alloc_rows(ROWS)
        esc.esc_selectivity(tbl.handle, every.handle, out)
        got = torch.zeros(rows + 64, dtype=torch.int32, device="cuda")
        col = torch.full((rows + 64,), -7, dtype=torch.int64, device="cuda")
        got[rows:] = -7
        esc.esc_debug_taint_slot(1)
        with pytest.raises(esc.EscError) as ei:
            esc.esc_selectivity(stbl.handle, p.handle, (rows, got, [col]))
        assert ei.value.status == esc.ESC_ETIMEOUT
        torch.cuda.synchronize()
        assert bool((got[:rows] >= 0).all()) and int(got[:rows].max()) < rows
        assert bool((got[rows:] == -7).all()) and bool((col[rows:] == -7).all())
    check("select", call(esc, tbl, "select", len(ids)), ids, vals)
