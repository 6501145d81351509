"""md_bin_cells re-sorts the atoms and leaves the list as it was built: what
md_stats says of the last list (longest row, entries, slots) stays until the
next list is built."""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu

KEYS = ("max_count", "list_entries", "slot_entries", "slot_max", "slots", "builds")


@pytest.mark.parametrize("variant", ["full", "paired"])
@pytest.mark.parametrize("nc", [6, 40])
def test_binning_keeps_the_list_counts(variant, nc):
    s = inputs.lj_fcc(nc=nc, T=0.5)
    pos = np.mod(s.pos + 0.05 * inputs.gaussian(801, s.pos.size).reshape(-1, 3), s.box)
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    with md.System(pos, s.vel, s.box, precision="mixed", force_variant=fv) as a:
        a.neighbors()  # per-atom rows under either layout
        a.step(3)
        f = a.state()[2]
        before = a.stats()
        md.md_bin_cells(a.h)
        after = a.stats()
        assert {k: after[k] for k in KEYS} == {k: before[k] for k in KEYS}
        md.md_forces(a.h)  # a new list, its counts from zero
        again = a.stats()
        assert again["builds"] == before["builds"] + 1
        key = "slot_entries" if variant == "paired" else "list_entries"
        assert abs(again[key] - before[key]) < 0.05 * before[key]
        g = a.state()[2]
    assert float((f - g).abs().max()) < 2e-4 * float(f.abs().max())
