"""A wait for the tensor cores that gives up (made to in the checked build, in
a process of its own): the samples not computed are NaN in y, the loss is
NaN and nothing that depends on the wait is added to the gradient, and the
next call works (the block waited for its products and freed its tensor
memory)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_RUN = r"""
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np
import torch
from paper_1901_01488_gb300 import esc
from tests.test_gpu_mlp_tiles import setup

assert esc.esc_build_checked()
sms = torch.cuda.get_device_properties(0).multi_processor_count
N = esc.MLP_PARAMS


def forward(B, dx, dw, dp):
    y = torch.full((B + 8,), 7.0, device="cuda")
    esc.esc_mlp_forward(dx, dw, dp, y)
    assert bool((y[B:] == 7.0).all())
    return y[:B]


def gradient(dx, dt, dw, dp):
    grad, loss = torch.zeros(N, device="cuda"), torch.zeros(1, device="cuda")
    esc.esc_mlp_grad(dx, dt, dw, dp, grad, loss)
    return grad, loss.item()


# forward: a tile has three waits
for B in (100, 1000, 128 * (2 * sms + 5)):
    _, _, _, dx, dw, dp, _ = setup(esc, B, B, 0)
    want = forward(B, dx, dw, dp)
    assert bool(torch.isfinite(want).all())
    for wait in range(1, 8):
        esc.esc_debug_mlp_give_up(wait)
        y = forward(B, dx, dw, dp)
        esc.esc_debug_mlp_give_up(0)
        done = (wait - 1) // 3 * 2 * sms * 128        # samples of the tiles before
        assert torch.equal(y[:done], want[:done]), wait
        assert bool(torch.isnan(y[done:]).all()), wait
        assert torch.equal(forward(B, dx, dw, dp), want), wait

# gradient: five
W2 = slice(8192 + 128, 8192 + 128 + 128 * 128)
for B in (100, 128):                                   # one block: an entry is added once (b3: four times)
    _, _, _, dx, dw, dp, dt = setup(esc, B, B, 0)
    want, loss = gradient(dx, dt, dw, dp)
    assert bool(torch.isfinite(want).all()) and np.isfinite(loss)
    for wait in range(1, 7):
        esc.esc_debug_mlp_give_up(wait)
        grad, lost = gradient(dx, dt, dw, dp)
        esc.esc_debug_mlp_give_up(0)
        if wait <= 5:
            assert np.isnan(lost), wait
            if wait == 5:                              # the second layer's weights had been added
                assert torch.equal(grad[W2], want[W2])
                grad[W2] = 0
            assert bool((grad[:-1] == 0).all()), wait
        else:
            assert torch.equal(grad[:-1], want[:-1])
        again, l2 = gradient(dx, dt, dw, dp)
        assert torch.equal(again[:-1], want[:-1]) and np.isfinite(l2), wait
B = 128 * (sms + 1)                                    # a second tile in one block
_, _, _, dx, dw, dp, dt = setup(esc, B, 3, 0)
want, loss = gradient(dx, dt, dw, dp)
for wait in range(6, 12):
    esc.esc_debug_mlp_give_up(wait)
    grad, lost = gradient(dx, dt, dw, dp)
    esc.esc_debug_mlp_give_up(0)
    assert np.isnan(lost) == (wait <= 10), wait
torch.cuda.synchronize()
print("ok")
"""


def test_waits_that_give_up():
    from paper_1901_01488_gb300 import build
    build.build()
    env = dict(os.environ, ESC_CHECKED="1")
    r = subprocess.run([sys.executable, "-c", _RUN, ROOT], env=env, cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout[-3000:] + r.stderr[-3000:]


def test_release_build_has_no_such_hook():
    from paper_1901_01488_gb300 import esc
    if esc.esc_build_checked():
        pytest.skip("the checked build is loaded")
    with pytest.raises(esc.EscError) as ei:
        esc.esc_debug_mlp_give_up(1)
    assert ei.value.status == esc.ESC_EINVAL
