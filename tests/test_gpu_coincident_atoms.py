"""Two atoms at one position: 1/r is infinite, so the energy is not finite and
a step reports MD_ERR_NONFINITE -- in float64 as in mixed precision, for every
count of lanes per atom of the float64 passes (16, 8, 4 and 1).  Atoms so close
that r^2 is below float32's range, but not float64's, have their finite energy."""
import math

import numpy as np
import pytest

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu


def duplicated(s):
    pos = s.pos.copy()
    pos[1] = pos[0]
    return pos


def expect_nonfinite(a):
    ke, pe = a.energy()
    assert not math.isfinite(pe), pe
    with pytest.raises(md.MDError) as err:
        a.step(3)
    assert err.value.status == md.MD_ERR_NONFINITE


@pytest.mark.parametrize("precision,nc", [("fp64", 6), ("fp64", 10), ("fp64", 16), ("fp64", 21),
                                          ("mixed", 6)])
def test_lennard_jones(precision, nc):
    s = inputs.lj_fcc(nc=nc, T=0.5)
    with md.System(duplicated(s), s.vel, s.box, precision=precision) as a:
        expect_nonfinite(a)


@pytest.mark.parametrize("precision,nc", [("fp64", 6), ("fp64", 21), ("mixed", 6)])
def test_two_species(precision, nc):
    s = inputs.lj_alloy(nc=nc)
    p = s.params
    with md.System(duplicated(s), s.vel, s.box, precision=precision, rc=p["rc"], skin=p["skin"],
                   dt=p["dt"],
                   species=(p["types"], p["t_eps"], p["t_sigma"], p["t_mass"])) as a:
        expect_nonfinite(a)


@pytest.mark.parametrize("precision,nc,n_exp,m_exp", [("fp64", 7, 9, 6), ("fp64", 7, 10, 6),
                                                      ("fp64", 21, 9, 6), ("mixed", 7, 9, 6)])
def test_sutton_chen(precision, nc, n_exp, m_exp):
    s = inputs.sc_fcc(nc=nc, n_exp=float(n_exp), m_exp=float(m_exp))
    p = s.params
    with md.System(duplicated(s), s.vel, s.box, potential="sc", precision=precision,
                   eps=p["eps"], sigma=p["sigma"], c=p["c"], n_exp=p["n_exp"], m_exp=p["m_exp"],
                   rc=p["rc"], skin=p["skin"], dt=p["dt"]) as a:
        expect_nonfinite(a)


@pytest.mark.parametrize("d", [1e-9, 1e-8, 1.05e-8, 1.1e-8, 2e-8, 1e-6])
def test_distance_below_float32(d):
    """Lengths in units of 1e-11, two atoms d sigma apart: below d = 1.08e-8, r^2
    is below float32's normal range, but 1/r^2 is a finite float64.  The pair's
    energy is 4 (sigma / r)^12 to float64's rounding (a few units of 2^-53 per
    factor); r^-6 and the other pairs add less than that."""
    s, u = inputs.lj_fcc(nc=6, T=0.5), 1e-11
    box = s.box * u
    pos = s.pos * u
    near = np.argsort(((s.pos - 0.5 * s.box) ** 2).sum(1))[:2]
    pos[near] = 0.5 * box  # the middle of a cell: its frame holds the distance exactly
    pos[near[1], 0] += d * u
    sep = pos[near[1], 0] - pos[near[0], 0]
    with md.System(pos, np.zeros_like(pos), box, precision="fp64", sigma=u, rc=2.5 * u,
                   skin=0.3 * u) as a:
        ke, pe = a.energy()
    want = 4.0 * (u / sep) ** 12
    assert abs(pe - want) <= 1e-13 * want, (pe, want)
