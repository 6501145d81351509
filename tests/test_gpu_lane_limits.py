"""The Lennard-Jones mixed passes on both sides of each layout's limit of four
lanes per item (47,104 atoms, 61,440 slots of two; one lane above) and of eight
(16,384 of either), against the oracle with the mixed path's bar (2e-4
relative, 1e-5 of the rms; atoms with a pair within rounding of the cutoff left
out)."""
import numpy as np
import pytest

from paper_1611_00075_gb300 import inputs, md
from test_gpu_paired import near_cutoff
from test_gpu_split_lanes import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.lib()
    return oracle


@pytest.mark.parametrize("variant,nc,n", [
    ("full", 17, 16384), ("full", 17, 16385), ("full", 23, 47104), ("full", 23, 47105),
    ("paired", 21, 32768), ("paired", 21, 32770), ("paired", 32, 122880),
    ("paired", 32, 122882)])
def test_limits(orc, variant, nc, n):
    s = inputs.lj_fcc(nc=nc, T=0.5)
    keep = np.sort(np.argsort(inputs.uniform(860 + nc, s.n))[:n])  # vacancies at random
    pos = np.mod(s.pos + 0.05 * inputs.gaussian(861, s.pos.size).reshape(-1, 3), s.box)[keep]
    off, ids = orc.neighbors_cells(pos, s.box, 2.8)
    U, f0 = orc.lj_list(pos, s.box, off, ids)
    bad = near_cutoff(pos, s.box, off, ids, 2.5, 1e-5)
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    with md.System(pos, s.vel[keep], s.box, precision="mixed", force_variant=fv) as a:
        check(a.state()[2].cpu().numpy(), f0, bad)
        assert abs(a.energy()[1] - U) <= 2e-6 * abs(U) + 0.02 * bad.sum()
