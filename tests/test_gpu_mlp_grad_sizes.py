"""The cost model's gradient kernel at the sizes where its grouping can go
wrong: one sample, one short of / exactly / one past a warp's 32 samples, a
block's 128, and the whole grid's 456 blocks, and a second round of the grid.

Reference: the same network in float64.  Tolerance per parameter: every
product and sum of a sample's contribution is rounded to float32 along at most
32 + 32 + 32 additions, then at most two rounds of 32 samples are added, so the
error is below 300 x 2^-24 times the sum of the contributions' magnitudes; a
pre-activation within rounding of zero may also switch one unit of one sample,
which moves the gradient by at most the largest single contribution (allowed
once, above 1,000 samples only).
"""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu


def reference(X, y, P):
    W1, b1 = P[:96].reshape(32, 3), P[96:128]
    W2, b2 = P[128:1152].reshape(32, 32), P[1152:1184]
    W3, b3 = P[1184:1216], P[1216]
    z1 = X @ W1.T + b1
    a1 = np.maximum(z1, 0)
    z2 = a1 @ W2.T + b2
    a2 = np.maximum(z2, 0)
    e = a2 @ W3 + b3 - y
    dy = 2 * e / len(X)
    d2 = dy[:, None] * W3[None] * (z2 > 0)
    d1 = (d2 @ W2) * (z1 > 0)
    # magnitudes of the same sums, without cancellation
    ad1 = (np.abs(d2) @ np.abs(W2)) * (z1 > 0)
    one = np.ones((len(X), 1))

    def parts(d1, d2, dy):
        return [(d1, np.abs(X) if d1 is ad1 else X), (d1, one), (d2, a1), (d2, one),
                (dy[:, None], a2), (dy[:, None], one)]

    G = np.concatenate([(d.T @ a).ravel() for d, a in parts(d1, d2, dy)])
    mags = [(np.abs(d), np.abs(a)) for d, a in parts(ad1, d2, dy)]
    A = np.concatenate([(d.T @ a).ravel() for d, a in mags])
    top = np.concatenate([np.outer(d.max(0), a.max(0)).ravel() for d, a in mags])
    return float(np.mean(e * e)), G, A, top


@pytest.mark.parametrize("ns", [1, 31, 32, 33, 127, 128, 129, 456 * 128 - 1, 456 * 128 + 1,
                                2 * 456 * 128 + 33])
def test_gradient_at_group_edges(ns):
    u = inputs.uniform(17 + ns, 3 * ns + ns + md.MLP_NPARAMS).astype(np.float32)
    X, y = u[:3 * ns].reshape(ns, 3), u[3 * ns:4 * ns]
    P = (u[4 * ns:] - 0.5) * 0.8
    Xd, yd, Pd = (torch.tensor(t, device="cuda") for t in (X, y, P))
    G = torch.full((md.MLP_NPARAMS,), float("nan"), device="cuda")
    loss = torch.full((1,), float("nan"), device="cuda")
    md.md_mlp_loss_grad(Xd, yd, Pd, G, loss)
    l0, G0, A, top = reference(X.astype(np.float64), y.astype(np.float64), P.astype(np.float64))
    tol = 300 * 2.0 ** -24 * A + (top if ns > 1000 else 0.0) + 1e-30
    g = G.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(g - G0) <= tol), np.max(np.abs(g - G0) / tol)
    assert abs(float(loss) - l0) <= 300 * 2.0 ** -24 * l0 + 1e-12
