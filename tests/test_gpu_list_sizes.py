"""Neighbour lists on both sides of the limit up to which a warp builds each
row (24,576 atoms, or slots of two): exact sets against the oracle on every
layout and precision, with cells of more than a warp's candidates, one-atom
cells and ragged rows."""
import numpy as np
import pytest

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.lib()
    return oracle


CASES = [("full", "mixed", 18), ("full", "mixed", 19), ("full", "fp64", 18), ("full", "fp64", 19),
         ("half", "mixed", 18), ("half", "mixed", 19), ("paired", "mixed", 22),
         ("paired", "mixed", 24)]


@pytest.mark.parametrize("variant,precision,nc", CASES)
def test_lists_at_the_limit(orc, variant, precision, nc):
    s = inputs.lj_fcc(nc=nc, T=0.5)
    pos = s.pos + 0.07 * inputs.gaussian(500 + nc, s.pos.size).reshape(-1, 3)
    # a density wave: cells of 10 to 40 atoms
    pos[:, 0] += 0.5 * s.box[0] / (2 * np.pi) * np.sin(2 * np.pi * pos[:, 0] / s.box[0])
    pos = np.mod(pos, s.box)
    off, ids = orc.neighbors_cells(pos, s.box, 2.8, half=variant == "half")
    fv = {"full": md.MD_FORCE_FULL, "half": md.MD_FORCE_HALF_ATOMIC,
          "paired": md.MD_FORCE_PAIRED}[variant]
    with md.System(pos, s.vel, s.box, precision=precision, force_variant=fv) as a:
        goff, gids = a.neighbors(half=variant == "half")
        st = a.stats()
        md.md_build_neighbors(a.h)
        assert a.stats()["slot_entries"] == st["slot_entries"]
    np.testing.assert_array_equal(goff.cpu().numpy(), off)
    np.testing.assert_array_equal(gids.cpu().numpy(), ids)
