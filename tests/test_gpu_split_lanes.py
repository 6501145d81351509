"""The mixed passes on both sides of their lanes-per-item limits (eight lanes up
to 16,384 atoms or slots, four up to 65,536, then one) and where the list
capacity alone forbids a split, against the oracle with the mixed path's bar
(2e-4 relative, 1e-5 of the rms; atoms with a pair within rounding of the cutoff
left out); forces stored by a step (the split epilogue) against a fresh
evaluation at the same positions, which runs the same kernel without it."""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md
from test_gpu_paired import near_cutoff

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.lib()
    return oracle


def jitter(s, amp, seed):
    return np.mod(s.pos + amp * inputs.gaussian(seed, s.pos.size).reshape(-1, 3), s.box)


def check(f, f0, bad):
    fn = np.linalg.norm(f0, axis=1)
    rms = np.sqrt(np.mean(fn * fn))
    ok = np.linalg.norm(f - f0, axis=1) <= 2e-4 * fn + 1e-5 * max(1.0, rms)
    assert np.all(ok | bad), int((~(ok | bad)).sum())


@pytest.mark.parametrize("variant,nc", [("full", 16), ("full", 17), ("full", 25), ("full", 26),
                                        ("paired", 20), ("paired", 21), ("paired", 32),
                                        ("paired", 33)])
def test_lj_sizes(orc, variant, nc):
    s = inputs.lj_fcc(nc=nc, T=0.5)
    pos = jitter(s, 0.05, 400 + nc)
    off, ids = orc.neighbors_cells(pos, s.box, 2.8)
    _, f0 = orc.lj_list(pos, s.box, off, ids)
    bad = near_cutoff(pos, s.box, off, ids, 2.5, 1e-5)
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    with md.System(pos, s.vel, s.box, precision="mixed", force_variant=fv) as a:
        check(a.state()[2].cpu().numpy(), f0, bad)
        a.step(3)
        x, v, f = a.state()
        U = sum(a.energy())
        md.md_set_state(a.h, x, v)
        md.md_forces(a.h)
        g = a.state()[2]
        # the list is new, so the order of the sums may differ: float32 rounding
        rms = float(torch.sqrt((g * g).mean()))
        assert float((f - g).abs().max()) < 2e-4 * max(rms, float(g.abs().max()))
        assert abs(sum(a.energy()) - U) < 1e-6 * abs(U)


@pytest.mark.parametrize("variant", ["full", "paired"])
def test_two_species(orc, variant):
    s = inputs.lj_alloy(nc=7)
    p = s.params
    pos = jitter(s, 0.03, 441)
    off, ids = orc.neighbors_cells(pos, s.box, p["rc"] + p["skin"])
    f0 = orc.lj_typed_list(pos, s.box, off, ids, p["types"], p["t_eps"], p["t_sigma"])[1]
    bad = near_cutoff(pos, s.box, off, ids, p["rc"], 1e-5)
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    with md.System(pos, s.vel, s.box, precision="mixed", force_variant=fv, rc=p["rc"],
                   skin=p["skin"], dt=p["dt"],
                   species=(p["types"], p["t_eps"], p["t_sigma"], p["t_mass"])) as a:
        check(a.state()[2].cpu().numpy(), f0, bad)


@pytest.mark.parametrize("cap", [252, 256, 260, 508, 512, 516])
def test_capacity_limits_the_split(orc, cap):
    """Lists of up to cap entries: four lanes carry 256, eight 512."""
    s = inputs.lj_fcc(nc=6, T=0.5)
    pos = jitter(s, 0.05, 451)
    off, ids = orc.neighbors_cells(pos, s.box, 2.8)
    _, f0 = orc.lj_list(pos, s.box, off, ids)
    bad = near_cutoff(pos, s.box, off, ids, 2.5, 1e-5)
    with md.System(pos, s.vel, s.box, precision="mixed", max_neighbors=cap) as a:
        check(a.state()[2].cpu().numpy(), f0, bad)


@pytest.mark.parametrize("unit", [1.0, 1e-12, 1e-14, 1e13])
def test_two_species_cutoff_in_other_units(orc, unit):
    """The cutoff by a saturated multiply-add (r_c^2 well inside float32's
    range) and by comparison (1e-14 and 1e13: too close to its ends), two atoms
    per thread: the same forces in every unit of length."""
    s = inputs.lj_alloy(nc=6)
    p = s.params
    pos = jitter(s, 0.03, 461)
    off, ids = orc.neighbors_cells(pos, s.box, p["rc"] + p["skin"])
    f0 = orc.lj_typed_list(pos, s.box, off, ids, p["types"], p["t_eps"], p["t_sigma"])[1]
    bad = near_cutoff(pos, s.box, off, ids, p["rc"], 1e-5)
    with md.System(pos * unit, np.zeros_like(pos), s.box * unit, precision="mixed",
                   force_variant=md.MD_FORCE_PAIRED, rc=p["rc"] * unit, skin=p["skin"] * unit,
                   dt=p["dt"], species=(p["types"], p["t_eps"], p["t_sigma"] * unit,
                                        p["t_mass"])) as a:
        f = a.state()[2].cpu().numpy() * unit
        pe = a.energy()[1]
    check(f, f0, bad)
    if unit == 1.0:
        pe1 = orc.lj_typed_list(pos, s.box, off, ids, p["types"], p["t_eps"], p["t_sigma"])[0]
        assert abs(pe - pe1) < 2e-5 * abs(pe1)


@pytest.mark.parametrize("variant,nc", [("full", 7), ("full", 17), ("full", 18), ("paired", 7),
                                        ("paired", 23), ("paired", 24)])
def test_sutton_chen_sizes(orc, variant, nc):
    """Eight lanes up to 20,480 atoms or 24,576 slots, one above."""
    s = inputs.sc_fcc(nc=nc)
    p = s.params
    pos = jitter(s, 0.02, 470 + nc)
    kw = dict(eps=p["eps"], sigma=p["sigma"], c=p["c"], n_exp=p["n_exp"], m_exp=p["m_exp"],
              rc=p["rc"], skin=p["skin"], dt=p["dt"])
    U, f0 = orc.forces_once(orc.make_params(potential=orc.POT_SC, **kw), pos, s.box)
    off, ids = orc.neighbors_cells(pos, s.box, p["rc"] + p["skin"])
    bad = near_cutoff(pos, s.box, off, ids, p["rc"], 1e-5)
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    with md.System(pos, s.vel, s.box, potential="sc", precision="mixed", force_variant=fv, **kw) as a:
        check(a.state()[2].cpu().numpy(), f0, bad)
        ke, pe = a.energy()
        assert abs(pe - U) < 2e-6 * abs(U) + 1e-3 * bad.sum()


@pytest.mark.parametrize("variant,nc", [("full", 8), ("full", 18), ("full", 19), ("paired", 8),
                                        ("paired", 24)])
def test_embedded_atom_sizes(orc, variant, nc):
    """Eight lanes up to 12,288 atoms or slots, one above."""
    s = inputs.eam_bcc(nc=nc)
    p = s.params
    keys = ("phi_r", "phi_a", "psi_r", "psi_a", "F_sqrt", "F_quad")
    pos = jitter(s, 0.04, 480 + nc)
    off, ids = orc.neighbors_cells(pos, s.box, p["rc"] + p["skin"])
    f0 = orc.eam_list(pos, s.box, off, ids, orc.make_eam(*[p[k] for k in keys]), p["rc"])[1]
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    with md.System(pos, s.vel, s.box, precision="mixed", force_variant=fv, rc=p["rc"],
                   skin=p["skin"], dt=p["dt"], eam={k: p[k] for k in keys}) as a:
        check(a.state()[2].cpu().numpy(), f0, np.zeros(len(pos), bool))
