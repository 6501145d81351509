"""Where several lanes share an atom, the lanes' float32 sums are added with more
than float32's digits, as the chunks of a one-lane row are.

An atom between two close neighbours, whose forces on it cancel exactly, and a
third, weak one: the three entries lie in rows' quads of their own, so three
lanes hold them, and entries past r_c (between the cutoff and r_list) fill the
quads.  Tolerance: the weak pair's term is right to 2^-20 of itself (a dozen
float32 roundings), while the close pairs' is 4e5 and added in float32 would round
the sum to multiples of 2^-6."""
import numpy as np
import pytest

from paper_1611_00075_gb300 import md

pytestmark = pytest.mark.gpu


def one_atom():
    """Nine cells of side 3 per plane; everything sits in the middle cell, whose
    atoms are listed in the order of their ids."""
    box = np.full(3, 9.0)
    c = np.full(3, 4.5)
    corner = [np.array([x, y, z]) * 1.47 for x in (-1, 1) for y in (-1, 1) for z in (-1, 1)]
    weak = np.array([0.9, 1.1, 0.25])
    rel = [np.zeros(3), [0.5, 0, 0], *corner[0:3], [-0.5, 0, 0], *corner[3:6], weak, *corner[6:8]]
    pos = c + np.array(rel, dtype=np.float64)
    # 32 more atoms far from the first one and from each other
    g = np.array([[x, y, z] for x in (0.75, 8.25) for y in (0.75, 3.0, 6.0, 8.25)
                  for z in (0.75, 3.0, 6.0, 8.25)])
    return np.concatenate([pos, g]), box


@pytest.mark.parametrize("typed", [False, True])
def test_cancelling_lanes(typed):
    pos, box = one_atom()
    n = len(pos)
    r = pos[1:] - pos[0]
    r -= box * np.round(r / box)
    r2 = (r * r).sum(1)
    # 11 entries within r_list, and the third quad's weak one at place 8
    listed = np.flatnonzero(r2 < 2.8 ** 2)
    assert list(listed[:11]) == list(range(11)) and np.all(r2[1:4] > 2.5 ** 2)
    near = r2 < 2.5 ** 2
    s6 = r2 ** -3
    fs = 48.0 / r2 * s6 * (s6 - 0.5)
    want = -(np.where(near, fs, 0.0)[:, None] * r).sum(0)
    kw = {}
    if typed:
        kw["species"] = (np.zeros(n, np.int32), np.ones((2, 2)), np.ones((2, 2)), np.ones(2))
    with md.System(pos, np.zeros_like(pos), box, precision="mixed", **kw) as a:
        f = a.state()[2].cpu().numpy()[0]
    weak = 48.0 * np.linalg.norm(want)  # bounds each product of the term
    assert np.all(np.abs(f - want) <= 2.0 ** -20 * weak), (f, want)
