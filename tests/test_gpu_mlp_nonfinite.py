"""The gradient of a batch with infinities, NaN or products that overflow:
only what such a sample reaches becomes non-finite, and everything else is as
accurate as without it.  A unit that a sample leaves inactive has no gradient
from it, whatever the sample's residual.

The bounds of the finite entries are test_gpu_mlp_tiles.py's."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from tests.test_gpu_mlp_tiles import U, layers, setup

pytestmark = pytest.mark.gpu
BIG = float(np.finfo(np.float32).max)


def reference(P, x, t):
    """Gradient (units a sample leaves inactive get nothing from it), entries' bounds, entries whose gate is unclear."""
    B = len(t)
    a1, z1, a2, y, m1, m2, my = layers(P, x)
    e = y - t
    dy = 2 / B * e
    g2, g1 = a2 > 0, a1 > 0
    d2 = np.where(g2, np.outer(dy, P["w3"]), 0.0)
    d1 = np.where(g1, d2 @ P["W2"], 0.0)
    ok = np.isfinite(t)
    D2 = np.outer(2 / B * (my + np.where(ok, np.abs(t), 0.0)), np.abs(P["w3"])) * ok[:, None]
    D1 = D2 @ np.abs(P["W2"])
    u2, u1 = np.abs(a2) <= U * m2, np.abs(a1) <= U * m1
    E2 = 4 * U * D2 + u2 * D2
    E1 = 4 * U * D1 + (u2 * D2) @ np.abs(P["W2"]) + u1 * D1
    want = {"W1": d1.T @ x, "b1": d1.sum(0), "W2": d2.T @ z1, "b2": d2.sum(0),
            "w3": dy @ np.maximum(a2, 0), "b3": np.array([dy.sum()])}
    bound = {"W1": E1.T @ np.abs(x), "b1": E1.sum(0), "W2": E2.T @ m1, "b2": E2.sum(0),
             "w3": 4 * U * ((2 / B * (my + np.where(ok, np.abs(t), 0.0)) * ok) @ m2),
             "b3": np.array([4 * U * (2 / B * (my + np.where(ok, np.abs(t), 0.0)) * ok).sum()])}
    return want, bound, (u1, u2)


def compare(grad, want, bound):
    got = omlp.unflatten(grad.cpu().numpy().astype(np.float64))
    seen = 0
    for k in want:
        w, b, g = want[k], bound[k], got[k]
        finite = np.isfinite(w) & (np.abs(w) + b < 0.9 * BIG)
        lost = ~np.isfinite(w) | (np.abs(w) - b > 1.1 * BIG)       # (between: either)
        assert (np.abs(g[finite] - w[finite]) <= b[finite]).all(), k
        assert not np.isfinite(g[lost]).any(), k
        if k in ("W1", "b1", "W2", "b2"):
            assert finite.any() and lost.any(), k
        seen += int(finite.sum())
    assert seen > 5000


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("B,at", [(1, [0]), (128, [0, 127]), (300, [5, 131, 299]), (20_000, [19_968])])
def test_residuals(B, at, value):
    from paper_1901_01488_gb300 import esc
    P, x, t, dx, dw, dp, dt = setup(esc, B, 40 + B, 0)
    dt[at] = value
    t[at] = value
    grad = torch.zeros(esc.MLP_PARAMS, device="cuda")
    loss = torch.zeros(1, device="cuda")
    esc.esc_mlp_grad(dx, dt, dw, dp, grad, loss)
    want, bound, (u1, u2) = reference(P, x, t)
    assert not (u1[at].any() or u2[at].any())        # what these samples reach is certain
    compare(grad, want, bound)
    assert not np.isfinite(loss.item())


@pytest.mark.parametrize("B,at", [(2, [1]), (4, [1, 3])])
def test_products_that_overflow(B, at):
    """dy and dy * w3 are finite, dy * z1 is not."""
    from paper_1901_01488_gb300 import esc
    P, x, t, dx, dw, dp, dt = setup(esc, B, 70 + B, 0)
    x[at] = float(np.array([0x3f66 << 16], np.uint32).view(np.float32)[0])    # 0.9 in bfloat16
    dx[at] = 0x3f66
    for s in at:
        dt[s] = -min(BIG, 1e38 * B)
        t[s] = float(dt[s].item())
    grad = torch.zeros(esc.MLP_PARAMS, device="cuda")
    loss = torch.zeros(1, device="cuda")
    esc.esc_mlp_grad(dx, dt, dw, dp, grad, loss)
    want, bound, _ = reference(P, x, t)
    z1 = np.maximum(x[at] @ P["W1"].T + P["b1"], 0)
    assert (2 / B * -t[at][:, None] * z1 > BIG).any()
    got = omlp.unflatten(grad.cpu().numpy().astype(np.float64))
    for k in ("W1", "b1", "W2", "b2"):
        clear = np.abs(want[k]) + bound[k] < 0.5 * BIG
        assert clear.sum() > clear.size // 2
        assert (np.abs(got[k] - want[k])[clear] <= bound[k][clear]).all(), k


def test_dead_unit_with_a_bad_bias():
    """A unit that no sample activates has no gradient, also when its bias or a weight is NaN."""
    from paper_1901_01488_gb300 import esc
    B = 100
    P, x, t, dx, dw, dp, dt = setup(esc, B, 90, 0)
    b2 = 8192 + 128 + 128 * 128
    out = []
    for bias in (-1e30, float("nan")):
        dp[b2 + 3] = bias
        grad = torch.zeros(esc.MLP_PARAMS, device="cuda")
        esc.esc_mlp_grad(dx, dt, dw, dp, grad, torch.zeros(1, device="cuda"))
        out.append(grad)
    assert bool(torch.isfinite(out[1]).all())
    # one block adds each entry once; b3's is the sum of four warps' in any order
    assert torch.equal(out[0][:-1], out[1][:-1])
    assert abs(out[0][-1] - out[1][-1]).item() <= 2.0 ** -21 * (2 / B * (layers(P, x)[6] + np.abs(t))).sum()
    assert out[1][b2 + 3].item() == 0.0 and out[1][b2 + 128 + 3].item() == 0.0


def expected(x, t, p):
    """y and the gradient with infinite parameters, in float64: 0 times infinity is NaN, which ReLU takes to 0."""
    P = {k: v.double() for k, v in omlp_torch(p).items()}
    x = x.double()
    relu = lambda a: torch.where(a > 0, a, torch.zeros((), dtype=torch.float64))
    prod = lambda a, w: (a[:, None, :] * w[None, :, :]).sum(2)        # (a library's product may skip zeros)
    a1 = prod(x, P["W1"]) + P["b1"]
    z1 = relu(a1)
    a2 = prod(z1, P["W2"]) + P["b2"]
    z2 = relu(a2)
    y = (z2 * P["w3"]).sum(1) + P["b3"]
    dy = 2.0 / len(t) * (y - t.double())
    d2 = torch.where(a2 > 0, dy[:, None] * P["w3"], torch.zeros((), dtype=torch.float64))
    d1 = torch.where(a1 > 0, prod(d2, P["W2"].T.contiguous()), torch.zeros((), dtype=torch.float64))
    g = {"W1": prod(d1.T, x.T.contiguous()), "b1": d1.sum(0), "W2": prod(d2.T, z1.T.contiguous()), "b2": d2.sum(0),
         "w3": prod(dy[None], z2.T.contiguous())[0], "b3": dy.sum()[None]}
    return y, g


def omlp_torch(p):
    out, o = {}, 0
    for name, s in omlp.sizes().items():
        n = int(np.prod(s))
        out[name] = p[o:o + n].reshape(s)
        o += n
    return out


@pytest.mark.parametrize("where", ["W2", "W2 unreached", "-W2", "w3", "w3 dead"])
@pytest.mark.parametrize("B", [1, 130])
def test_infinite_weights(B, where):
    """Small whole numbers throughout, so that the parts of an activation that are 0 (all but the
    first) and every sum are exact: finite values are compared exactly."""
    from paper_1901_01488_gb300 import esc
    rng = np.random.default_rng(B)
    p = torch.from_numpy(rng.integers(-2, 3, esc.MLP_PARAMS).astype(np.float32))
    P = omlp_torch(p)
    P["b1"][5], P["W1"][5] = 3.0, 0.0               # an active unit of the first layer, and an inactive one
    P["b1"][6], P["W1"][6] = -3.0, 0.0
    P["b2"][9], P["W2"][9] = -8.0, 0.0              # a unit that no sample activates
    inf = float("inf")
    if where == "W2":
        P["W2"][7][5] = inf
        P["w3"][7] = 2.0
    elif where == "W2 unreached":
        P["W2"][7][6] = inf                          # 0 times it: NaN, so the unit is inactive
    elif where == "-W2":
        P["W2"][7][5] = -inf
    elif where == "w3":
        P["w3"][7] = inf
    else:
        P["w3"][9] = inf
    x = torch.from_numpy(rng.integers(0, 2, (B, 64)).astype(np.float32))
    t = torch.from_numpy(rng.integers(-3, 4, B).astype(np.float32))
    y, g = expected(x, t, p)
    dx, dw, dp = x.to(torch.bfloat16).view(torch.int16).cuda(), p.to(torch.bfloat16).view(torch.int16).cuda(), p.cuda()
    out = torch.full((B,), 7.0, device="cuda")
    esc.esc_mlp_forward(dx, dw, dp, out)
    same = lambda a, b: torch.equal(torch.isfinite(a), torch.isfinite(b))
    out = out.cpu().double()
    assert same(out, y) and torch.equal(out[torch.isfinite(y)], y[torch.isfinite(y)])
    assert torch.equal(out == inf, y == inf) and torch.equal(out == -inf, y == -inf)
    grad, loss = torch.zeros(esc.MLP_PARAMS, device="cuda"), torch.zeros(1, device="cuda")
    esc.esc_mlp_grad(dx, dt := t.cuda(), dw, dp, grad, loss)
    got = omlp_torch(grad.cpu().double())
    for k, want in g.items():
        assert same(got[k], want), k
        f = torch.isfinite(want)
        assert bool(((got[k] - want).abs()[f] <= 2.0 ** -14 * (want.abs()[f] + 1e4)).all()), k
