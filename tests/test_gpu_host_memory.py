"""Calls that run out of host memory (injected) return ESC_ENOMEM, give back
the device memory they took, and leave the next call right."""
import pytest
import torch

import oracle
from paper_1901_01488_gb300 import datagen

pytestmark = pytest.mark.gpu
ROWS = 50_000


@pytest.fixture(scope="module")
def world():
    from paper_1901_01488_gb300 import build
    build.build()
    from paper_1901_01488_gb300 import esc
    t = datagen.skewed_table(ROWS, seed=51, device="cuda")
    return esc, esc.Table.from_datagen(t), t.host()


@pytest.mark.parametrize("npred", [8, 40, 2000])      # interpreted; looked up by rows and by words
def test_shared_scan(world, npred):
    esc, tbl, host = world
    texts = [p.text for p in datagen.skewed_predicates(npred, seed0=7)]
    ps = esc.PredicateSet(tbl, texts)
    out = torch.zeros(npred, dtype=torch.int64, device="cuda")
    esc.esc_selectivity_shared_async(tbl.handle, ps.handles, out)
    want = out.tolist()
    for k in range(0, npred, 1 + npred // 10):
        assert want[k] == oracle.count(texts[k], host)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(400):
        esc.esc_debug_fail_host_allocs(1)
        with pytest.raises(esc.EscError) as ei:
            esc.esc_selectivity_shared_async(tbl.handle, ps.handles, out)
        assert ei.value.status == esc.ESC_ENOMEM
    esc.esc_debug_fail_host_allocs(0)
    torch.cuda.synchronize()
    # (the library's pool grows by 32 MB at a time; 400 passes of 2,000 predicates hold over 1 GB)
    assert free - torch.cuda.mem_get_info()[0] <= 64 << 20
    out.zero_()
    esc.esc_selectivity_shared_async(tbl.handle, ps.handles, out)
    assert out.tolist() == want


def test_batch(world):
    esc, tbl, host = world
    texts = [p.text for p in datagen.skewed_predicates(30, seed0=9)]
    ps = [esc.Predicate(tbl, x) for x in texts]
    out = torch.zeros(30, dtype=torch.int64, device="cuda")
    esc.esc_debug_fail_host_allocs(1)
    with pytest.raises(esc.EscError) as ei:
        esc.esc_selectivity_batch_async([tbl.handle] * 30, [p.handle for p in ps], out)
    assert ei.value.status == esc.ESC_ENOMEM
    esc.esc_selectivity_batch_async([tbl.handle] * 30, [p.handle for p in ps], out)
    assert out.tolist() == [oracle.count(x, host) for x in texts]
