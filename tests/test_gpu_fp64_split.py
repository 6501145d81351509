"""The float64 passes on both sides of their lanes-per-atom limits (16 up to
3,072 atoms, 8 up to 8,192, 4 up to 32,768, then one), with lists whose last
quad is ragged, and in units whose squared lengths float32 cannot hold.

Tolerance: a force is a sum of about 60 (Sutton-Chen: 150) terms of at most
some 30 times the rms force, each right to a few units of 2^-53, so it is
within 1e-11 of the oracle's, relative to max(|f|, rms).
"""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.lib()
    return oracle


def close(f, f0):
    fn = np.linalg.norm(f0, axis=1)
    rms = np.sqrt(np.mean(fn * fn))
    err = np.linalg.norm(f - f0, axis=1) / np.maximum(fn, rms)
    assert err.max() < 1e-11, err.max()


def jitter(s, amp, seed):
    return np.mod(s.pos + amp * inputs.gaussian(seed, s.pos.size).reshape(-1, 3), s.box)


@pytest.mark.parametrize("nc", [6, 10, 11, 20, 21])  # 864 | 4000, 5324 | 32000 | 37044 atoms
def test_lj(orc, nc):
    s = inputs.lj_fcc(nc=nc, T=0.5)
    pos = jitter(s, 0.06, 300 + nc)
    U, f0 = orc.forces_once(orc.make_params(potential=orc.POT_LJ, rc=2.5, skin=0.3, dt=0.005),
                            pos, s.box)
    with md.System(pos, s.vel, s.box, precision="fp64") as a:
        ke, pe = a.energy()
        close(a.state()[2].cpu().numpy(), f0)
        assert abs(pe - U) < 1e-11 * abs(U)


@pytest.mark.parametrize("nc,n_exp,m_exp", [(7, 9, 6), (7, 12, 7), (11, 9, 6), (11, 10, 5)])
def test_sutton_chen(orc, nc, n_exp, m_exp):
    s = inputs.sc_fcc(nc=nc, n_exp=float(n_exp), m_exp=float(m_exp))
    p = s.params
    pos = jitter(s, 0.02, 320 + nc)
    kw = dict(eps=p["eps"], sigma=p["sigma"], c=p["c"], n_exp=p["n_exp"], m_exp=p["m_exp"],
              rc=p["rc"], skin=p["skin"], dt=p["dt"])
    U, f0 = orc.forces_once(orc.make_params(potential=orc.POT_SC, **kw), pos, s.box)
    with md.System(pos, s.vel, s.box, potential="sc", precision="fp64", **kw) as a:
        close(a.state()[2].cpu().numpy(), f0)


@pytest.mark.parametrize("nc", [6, 11, 21])
def test_two_species(orc, nc):
    s = inputs.lj_alloy(nc=nc)
    p = s.params
    pos = jitter(s, 0.03, 340 + nc)
    off, ids = orc.neighbors_cells(pos, s.box, p["rc"] + p["skin"])
    f0 = orc.lj_typed_list(pos, s.box, off, ids, p["types"], p["t_eps"], p["t_sigma"])[1]
    with md.System(pos, s.vel, s.box, precision="fp64", rc=p["rc"], skin=p["skin"], dt=p["dt"],
                   species=(p["types"], p["t_eps"], p["t_sigma"], p["t_mass"])) as a:
        close(a.state()[2].cpu().numpy(), f0)


def test_units_beyond_float32(orc):
    """Lengths of 1e-15: the float32 screen is off, every entry and candidate is
    decided in float64, and 1/x comes from the division."""
    s = inputs.lj_fcc(nc=6, T=0.5)
    pos, u = jitter(s, 0.06, 361), 1e-15
    _, f0 = orc.forces_once(orc.make_params(potential=orc.POT_LJ, rc=2.5, skin=0.3, dt=0.005),
                            pos, s.box)
    off, ids = orc.neighbors_cells(pos, s.box, 2.8)
    with md.System(pos * u, np.zeros_like(pos), s.box * u, precision="fp64", sigma=u, rc=2.5 * u,
                   skin=0.3 * u) as a:
        goff, gids = a.neighbors()
        f = a.state()[2].cpu().numpy() * u
    np.testing.assert_array_equal(goff.cpu().numpy(), off)
    np.testing.assert_array_equal(gids.cpu().numpy(), ids)
    close(f, f0)
