"""The union-list build's test in expanded form,
    |x|^2 - 2 m.x + (|m|^2 + |u|^2/4 - hi) < |u.x - u.m|   (u = x1 - x0),
evaluated in float32 with one rounding per multiply-add, never drops a candidate
within r_list of either atom: its rounding error stays below the margin
2^-14 r_list^2 that hi = r_list^2 (1 + 2^-14) adds.  Candidates lie in any of the
27 cells around the slot's, cells of 1 to 4/3 list radii (a box of three cells is
the widest), in units of very different size."""
import numpy as np
import pytest

F = np.float32


def fma(a, b, c):
    return (a.astype(np.float64) * b + c.astype(np.float64)).astype(F)


@pytest.mark.parametrize("unit", [1.0, 1e-10, 3.7e6])
@pytest.mark.parametrize("width", [1.0, 1.18, 4.0 / 3.0])
def test_no_candidate_is_lost(unit, width):
    rng = np.random.default_rng(int(width * 1000))
    n = 400000
    rl = 2.8 * unit
    w = np.float32(width * rl)
    hi = F(float(rl) ** 2 * (1 + 2.0 ** -14))
    q0 = (rng.uniform(-0.5, 0.5, (n, 3)) * float(w)).astype(F)
    q1 = (rng.uniform(-0.5, 0.5, (n, 3)) * float(w)).astype(F)
    s = rng.integers(-1, 2, (n, 3)).astype(F)
    # candidates on the shell |x - x0| = r_list (within 1e-5), where they fall
    # into one of the 27 cells; cell-relative positions
    d = rng.normal(size=(n, 3))
    d *= (rl * (1 - 1e-5 * rng.uniform(0, 1, (n, 1)))) / np.linalg.norm(d, axis=1)[:, None]
    cell = np.rint((q0 + d) / float(w))
    ok = np.all(np.abs(cell) <= 1, axis=1)
    s[ok] = cell[ok].astype(F)
    x = (q0.astype(np.float64) + d - s * float(w)).astype(F)
    x = np.clip(x, -0.5 * float(w), 0.5 * float(w)).astype(F)
    # as the kernel computes it
    u = q1 - q0
    m = (q0 + F(0.5) * u).astype(F)
    lim = (F(0.25) * fma(u[:, 0], u[:, 0], fma(u[:, 1], u[:, 1], u[:, 2] * u[:, 2])) - hi).astype(F)
    sm = fma(-s, np.full_like(s, w), m)
    k1 = (fma(sm[:, 0], sm[:, 0], fma(sm[:, 1], sm[:, 1], sm[:, 2] * sm[:, 2])) + lim).astype(F)
    k2 = -fma(u[:, 0], sm[:, 0], fma(u[:, 1], sm[:, 1], u[:, 2] * sm[:, 2]))
    wsq = fma(x[:, 0], x[:, 0], fma(x[:, 1], x[:, 1], x[:, 2] * x[:, 2]))
    r = (wsq + k1).astype(F)
    p = k2
    for k in range(3):
        r = fma(x[:, k], F(-2) * sm[:, k], r)
        p = fma(x[:, k], u[:, k], p)
    accept = r < np.abs(p)
    # exactly, for the same float32 positions
    e = x.astype(np.float64) + s * float(w)
    near = np.minimum(((e - q0) ** 2).sum(1), ((e - q1) ** 2).sum(1))
    within = near < rl * rl
    assert within.sum() > n // 4
    assert np.all(accept[within])
    # the form's error against the exact squared distance, of both signs
    err = np.abs((r.astype(np.float64) - np.abs(p) + float(hi)) - near).max()
    assert err < 0.5 * 2.0 ** -14 * rl * rl, err / (rl * rl)
