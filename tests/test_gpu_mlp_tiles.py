"""The surrogate's tensor-core kernels at the edges of their 128-sample tiles,
with unaligned arrays and with infinities, against 64-bit arithmetic.

Bounds: a value computed in float32 from exact products, by at most 32 sums
one after the other (each truncated or rounded), is off by at most 2^-18 of
the sum of its terms' magnitudes; a gradient entry chains three such values:
2^-16 of the same sum with every factor replaced by its magnitude.  Where a
pre-activation is too close to 0 to tell its sign, either gate is right."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu
U = 2.0 ** -18


def setup(esc, B, seed, shift):
    """Inputs; arrays start `shift` elements into their storage."""
    rng = np.random.default_rng(seed)
    p = np.concatenate([rng.normal(0, 1 / np.sqrt(s[1] if len(s) > 1 else 4), int(np.prod(s))).ravel()
                        for s in omlp.sizes().values()]).astype(np.float32)
    x = (rng.random((B, 64)) * (rng.random((B, 64)) < 0.6)).astype(np.float32)
    t = rng.normal(0, 1, B).astype(np.float32)

    def place(a, dtype=None):
        a = torch.from_numpy(a).cuda()
        a = a.to(torch.bfloat16).view(torch.int16) if dtype == "bf16" else a
        out = torch.zeros(a.numel() + 16, dtype=a.dtype, device="cuda")[shift:shift + a.numel()].view(a.shape)
        return out.copy_(a)

    P = omlp.unflatten(p.astype(np.float64))
    for k in ("W1", "W2", "w3"):
        P[k] = omlp.round_bf16(P[k].astype(np.float32)).astype(np.float64)
    return P, omlp.round_bf16(x).astype(np.float64), t.astype(np.float64), place(x, "bf16"), place(p, "bf16"), place(p), place(t)


def layers(P, x):
    a1 = x @ P["W1"].T + P["b1"]
    z1 = np.maximum(a1, 0)
    a2 = z1 @ P["W2"].T + P["b2"]
    y = np.maximum(a2, 0) @ P["w3"] + P["b3"]
    # magnitudes of the terms
    m1 = np.abs(x) @ np.abs(P["W1"]).T + np.abs(P["b1"])
    m2 = m1 @ np.abs(P["W2"]).T + np.abs(P["b2"])
    my = m2 @ np.abs(P["w3"]) + np.abs(P["b3"])
    return a1, z1, a2, y, m1, m2, my


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("B", [1, 127, 128, 129, 1000, 40_000])
def test_forward(B, shift):
    from paper_1901_01488_gb300 import esc
    P, x, _, dx, dw, dp, _ = setup(esc, B, B + shift, shift)
    y = torch.full((B + 8,), 7.0, device="cuda")
    esc.esc_mlp_forward(dx, dw, dp, y)
    *_, ref, _, _, my = layers(P, x)
    out = y.cpu().numpy().astype(np.float64)
    assert (np.abs(out[:B] - ref) <= U * my).all()
    assert (out[B:] == 7.0).all()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("B", [1, 127, 129, 300, 20_000])
def test_gradient(B, shift):
    from paper_1901_01488_gb300 import esc
    P, x, t, dx, dw, dp, dt = setup(esc, B, 10 + B + shift, shift)
    grad = torch.zeros(esc.MLP_PARAMS + 16, device="cuda")[shift:shift + esc.MLP_PARAMS]
    loss = torch.zeros(1, device="cuda")
    esc.esc_mlp_grad(dx, dt, dw, dp, grad, loss)
    a1, z1, a2, y, m1, m2, my = layers(P, x)
    e = y - t
    d2 = np.outer(2 / B * e, P["w3"])
    g2, g1 = a2 > 0, a1 > 0
    d1 = ((d2 * g2) @ P["W2"]) * g1
    D2 = np.outer(2 / B * (my + np.abs(t)), np.abs(P["w3"]))            # magnitudes
    D1 = D2 @ np.abs(P["W2"])
    u2, u1 = np.abs(a2) <= U * m2, np.abs(a1) <= U * m1                  # gates that may go either way
    E2 = 4 * U * D2 + u2 * D2                                            # possible error of d2, d1, z1
    E1 = 4 * U * D1 + (u2 * D2) @ np.abs(P["W2"]) + u1 * D1
    want = {"W1": d1.T @ x, "b1": d1.sum(0), "W2": (d2 * g2).T @ z1, "b2": (d2 * g2).sum(0),
            "w3": (2 / B * e) @ np.maximum(a2, 0), "b3": np.array([2 / B * e.sum()])}
    bound = {"W1": E1.T @ np.abs(x), "b1": E1.sum(0), "W2": E2.T @ m1, "b2": E2.sum(0),
             "w3": 4 * U * ((2 / B * (my + np.abs(t))) @ m2), "b3": np.array([4 * U * 2 / B * (my + np.abs(t)).sum()])}
    got = omlp.unflatten(grad.cpu().numpy().astype(np.float64))
    for k in want:
        assert (np.abs(got[k] - want[k]) <= bound[k]).all(), k
    assert abs(loss.item() - (e * e).sum()) <= 8 * U * ((my + np.abs(t)) ** 2).sum()


def test_infinite_activation():
    """An activation that overflows stays infinite (not NaN), and only its own sample's output does."""
    from paper_1901_01488_gb300 import esc
    p = torch.zeros(esc.MLP_PARAMS, device="cuda")
    p[0] = 3e38                                     # W1[0][0]
    p[8192 + 128:8192 + 128 + 128 * 128] = 1.0      # W2: ones
    p[24832:24960] = 1.0                            # w3
    x = torch.zeros((130, 64), device="cuda")
    x[:, 0] = 0.5
    x[5, 0], x[129, 0] = 1000.0, -1000.0
    y = torch.zeros(130, device="cuda")
    esc.esc_mlp_forward(x.to(torch.bfloat16).view(torch.int16), p.to(torch.bfloat16).view(torch.int16), p, y)
    assert y[5].item() == float("inf") and y[129].item() == 0.0
    others = torch.cat([y[:5], y[6:129]])
    assert bool((others == others[0]).all()) and others[0].item() > 1e38
