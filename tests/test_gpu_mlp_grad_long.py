"""The cost model's gradient over many samples, where a lane adds the
contributions of many groups of 32 one after another in float32: the measured
training size and one of several million.

Reference: the same network in float64, in chunks.  Tolerance per parameter, in
units of 2^-24 of the sum of the contributions' magnitudes: 96 additions within a
sample's contribution and its products (100 rounding steps allowed), 32 additions
per round of the grid of 456 blocks of four groups, the block's four warps, and
the final rounding.  A unit whose pre-activation lies within its own rounding
(35 steps of 2^-24 of its magnitude sum; 70 behind the first layer) of zero may be
on or off: what it contributes is allowed on top.
"""
import math

import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def reference(X, y, P):
    """(loss, gradient, magnitudes, allowance for undecided units), float64"""
    W1, b1 = P[:96].view(32, 3), P[96:128]
    W2, b2 = P[128:1152].view(32, 32), P[1152:1184]
    W3, b3 = P[1184:1216], P[1216]
    ns = len(X)
    loss = 0.0
    G, A, S = (torch.zeros(md.MLP_NPARAMS, dtype=torch.float64, device=X.device) for _ in range(3))

    def add(out, d1, d2, dy, X, a1, a2):
        out += torch.cat([(d1.T @ X).ravel(), d1.sum(0), (d2.T @ a1).ravel(), d2.sum(0),
                          (dy[:, None] * a2).sum(0), dy.sum()[None]])

    for k in range(0, ns, 1 << 18):
        x, t = X[k:k + (1 << 18)], y[k:k + (1 << 18)]
        z1 = x @ W1.T + b1
        m1 = x.abs() @ W1.abs().T + b1.abs()
        a1 = z1.clamp(min=0)
        z2 = a1 @ W2.T + b2
        m2 = m1 @ W2.abs().T + b2.abs()
        a2 = z2.clamp(min=0)
        e = a2 @ W3 + b3 - t
        dy = 2 * e / ns
        loss += float((e * e).sum())
        on1, on2 = (z1 > 0).double(), (z2 > 0).double()
        d2 = dy[:, None] * W3 * on2
        add(G, (d2 @ W2) * on1, d2, dy, x, a1, a2)
        # magnitudes: the error of e is of the size of its own sum's terms
        me = (m2 @ W3.abs() + b3.abs() + t.abs()) * 2 / ns
        q2 = me[:, None] * W3.abs() * on2
        add(A, (q2 @ W2.abs()) * on1, q2, me, x.abs(), a1, a2)
        # units within rounding of zero
        u1 = (z1.abs() <= 35 * U * m1).double()
        u2 = (z2.abs() <= 70 * U * m2).double()
        full2 = dy.abs()[:, None] * W3.abs()
        p2 = full2 * u2
        add(S, (p2 @ W2.abs()) + ((full2 * (on2 + u2)) @ W2.abs()) * u1, p2,
            torch.zeros_like(dy), x.abs(), a1, a2)
    return loss / ns, G, A, S


@pytest.mark.parametrize("ns", [541199, 4_000_037])
def test_gradient_over_many_rounds(ns):
    u = inputs.uniform(29, 4 * ns + md.MLP_NPARAMS).astype(np.float32)
    X, y = u[:3 * ns].reshape(ns, 3), u[3 * ns:4 * ns]
    P = (u[4 * ns:] - 0.5) * 0.8
    Xd, yd, Pd = (torch.tensor(t, device="cuda") for t in (X, y, P))
    G = torch.full((md.MLP_NPARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    md.md_mlp_loss_grad(Xd, yd, Pd, G, loss)
    l0, G0, A, S = reference(Xd.double(), yd.double(), Pd.double())
    rounds = math.ceil(math.ceil(ns / 32) / (456 * 4))
    steps = 100 + 32 * rounds + 4 + 1
    err = (G.double() - G0).abs()
    tol = steps * U * A + S + 1e-30
    worst = float((err / tol).max())
    print("ns %d: %d rounds, largest error %.3g of the bound, %.3g of the gradient's largest"
          % (ns, rounds, worst, float(err.max() / G0.abs().max())))
    assert worst <= 1.0
    assert abs(float(loss) - l0) <= steps * U * l0 + 1e-12
