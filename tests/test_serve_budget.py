"""The serving loop's memory budget covers its shared passes: the bound on
their scratch, which passes run, and (on the GPU) that a budget too small for
any is kept, with the same counts."""
import os
import subprocess
import sys

import pytest

from paper_1901_01488_gb300 import datagen, esc, serve
from paper_1901_01488_gb300.serve import Request, fit_groups, wave_groups

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_scratch_bound():
    got = [esc.esc_shared_scratch_bytes(n) for n in (1, 8, 32, 512, 2048)]
    assert got == sorted(got) and got[0] > 4096          # a compiled query is ~3.7 KB
    assert got[1] < 2 << 20                              # small groups reserve little
    assert (64 << 20) < got[-1] < 160 << 20
    assert esc.esc_shared_scratch_bytes(100_000) == got[-1]     # passes follow one another
    with pytest.raises(esc.EscError):
        esc.esc_shared_scratch_bytes(0)


def test_fit_groups():
    reqs = [Request(i, t, f"x < {i}", arrival=i * 1e-4) for i, t in enumerate([0, 0, 1, 0, 1, 1, 1, 2])]
    groups, rest = wave_groups(reqs, 3)
    assert [[r.rid for r in g] for g in groups] == [[0, 1, 3], [2, 4, 5, 6]]
    size = lambda n: 100 * n
    g, r, extra = fit_groups(groups, rest, 1000, size)
    assert g == groups and r == rest and extra == 400           # one after the other: the larger one's
    g, r, extra = fit_groups(groups, rest, 399, size)
    assert [[x.rid for x in k] for k in g] == [[0, 1, 3]] and [x.rid for x in r] == [2, 4, 5, 6, 7] and extra == 300
    g, r, extra = fit_groups(groups, rest, 0, size)
    assert g == [] and [x.rid for x in r] == list(range(8)) and extra == 0
    g, r, extra = fit_groups(groups, rest, -5, size)
    assert g == [] and extra == 0


@pytest.mark.gpu
@pytest.mark.parametrize("budget,shared", [(8 << 30, True), (300_000, False)])
def test_budget_holds_with_shared_passes(budget, shared):
    tabs = [datagen.skewed_table(n, seed=60 + i, device="cuda") for i, n in enumerate((20_000, 300_000))]
    etabs = [esc.Table.from_datagen(t) for t in tabs]
    work = datagen.batch_workload(160, seed=24, sizes=[t.nrows for t in tabs])
    reqs = [Request(j, ti, p.text, 0.0) for j, (ti, p) in enumerate(work)]
    srv = serve.Server(esc, etabs, mem_budget=budget, max_batch=64, streams=2)
    for r in srv.run(reqs):
        assert r.count == esc.count(etabs[r.table], esc.Predicate(etabs[r.table], r.text))
    assert (srv.shared_launches > 0) == shared
    assert srv.peak_bytes <= budget
    if shared:                                           # what the passes hold is in the account
        assert srv.peak_bytes >= esc.esc_shared_scratch_bytes(8)
    assert srv.in_flight_bytes == 0


_FOOTPRINT = r"""
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_1901_01488_gb300 import esc
n, kind = int(sys.argv[2]), sys.argv[3]
a = torch.arange(4000, dtype=torch.int32, device="cuda")
cols = [(f"c{k}", "i32", a * (k + 1)) for k in range(16)]
t = esc.Table(cols, 4000)
if kind == "lists":
    texts = [f"c{k % 16} IN ({', '.join(str(977 * k + 13 * j) for j in range(16))})" for k in range(n)]
else:
    texts = [" OR ".join(f"c{(k + j) % 16} BETWEEN {k * 31 + j} AND {k * 37 + 50 * j}" for j in range(4)) for k in range(n)]
ps = esc.PredicateSet(t, texts)
out = torch.zeros(n, dtype=torch.int64, device="cuda")
few = esc.PredicateSet(t, texts[:1])
esc.esc_selectivity_shared_async(t.handle, few.handles, out)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
passes = esc.esc_debug_shared_passes()[0]
esc.esc_selectivity_shared_async(t.handle, ps.handles, out)
torch.cuda.synchronize()
assert esc.esc_debug_shared_passes()[0] > passes
print(free - torch.cuda.mem_get_info()[0])
"""


@pytest.mark.gpu
@pytest.mark.parametrize("n,kind", [(128, "ranges"), (2048, "ranges"), (2048, "lists")])
def test_bound_against_the_pool(n, kind):
    """What a first shared scan adds to the device memory in use (the pool grows by up to 64 MB at a time)."""
    r = subprocess.run([sys.executable, "-c", _FOOTPRINT, ROOT, str(n), kind], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    assert int(r.stdout) <= esc.esc_shared_scratch_bytes(n) + (64 << 20)
