"""Shared scans under the checked build, each in a process of its own: the
lookup's and the interpreter's paths meet no index out of range, and a check
that fires is reported with its site."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run(args, timeout=900):
    from paper_1901_01488_gb300 import build
    build.build()
    r = subprocess.run([sys.executable] + args, env=dict(os.environ, ESC_CHECKED="1"), cwd=ROOT,
                       capture_output=True, text=True, timeout=timeout)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    return r.stdout


@pytest.mark.parametrize("module", ["test_gpu_shared_boxes.py", "test_gpu_shared_buckets.py",
                                    "test_gpu_shared_rule.py"])
def test_every_path(module):
    """Rows' words in registers or shared by lanes, with and without buckets, ragged tables, cuts sorted on the
    GPU, passes at their limits, predicates left to the interpreter."""
    out = run(["-m", "pytest", os.path.join("tests", module), "-q", "-x", "-p", "no:cacheprovider"])
    assert " passed" in out and "skipped" not in out, out[-2000:]


_REPORT = r"""
import sys
sys.path.insert(0, sys.argv[1])
import torch
from paper_1901_01488_gb300 import esc

assert esc.esc_build_checked()
rows = 12000
a = (torch.arange(rows, dtype=torch.int32, device="cuda") * 7919) % 3000
t = esc.Table([("a", "i32", a)], rows)
for n in (40, 700):          # rows' words in registers; shared by lanes
    texts = [f"a BETWEEN {k} AND {2 * k + 900}" for k in range(n)]
    ps = esc.PredicateSet(t, texts)
    want = [int(((a >= k) & (a <= 2 * k + 900)).sum()) for k in range(n)]
    for shrink in (0, 1, 1 << 20, 0):
        esc.esc_debug_shrink_table(shrink)
        out = torch.zeros(n, dtype=torch.int64, device="cuda")
        try:
            esc.esc_selectivity_shared_async(t.handle, ps.handles, out)
            status, text = esc.ESC_OK, ""
        except esc.EscError as e:
            status, text = e.status, str(e)
        if shrink:
            assert status == esc.ESC_EBOUNDS and "site 41" in text, (n, shrink, status, text)
        else:
            assert status == esc.ESC_OK and out.tolist() == want, (n, shrink, text)
print("ok")
"""


def test_a_check_that_fires_is_reported():
    assert run(["-c", _REPORT, ROOT]).strip().endswith("ok")


def test_release_build_has_no_such_hook():
    from paper_1901_01488_gb300 import esc
    if esc.esc_build_checked():
        pytest.skip("the checked build is loaded")
    with pytest.raises(esc.EscError) as ei:
        esc.esc_debug_shrink_table(1)
    assert ei.value.status == esc.ESC_EINVAL
