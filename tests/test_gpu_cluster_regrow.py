"""A cluster list that has to grow between two runs of steps: the steps after
it must use the new list, not one that earlier captured steps hold.

The cluster list's rows are sized from the largest cell, the per-atom rows from
the longest row, so a state with one much fuller cell whose atoms still fit the
(preset) row capacity replaces the cluster list alone.  Forces after the steps
against the oracle with the mixed path's bar (2e-4 relative, 1e-5 of the rms;
atoms with a pair within rounding of the cutoff left out)."""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md
from test_gpu_paired import near_cutoff
from test_gpu_split_lanes import check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.lib()
    return oracle


def lattices():
    """The same 864 atoms in the same box twice: spread evenly (cells of about
    13), and drawn together so that the fullest cell holds over four times as many."""
    s = inputs.lj_fcc(nc=6, T=0.3)
    box = s.box * 1.5
    even = s.pos * 1.5
    # a smooth map of the box onto itself, denser around its middle
    x = even / box
    tight = (x + 0.08 * np.sin(2 * np.pi * x)) * box
    g = inputs.gaussian(731, even.size).reshape(-1, 3)
    return np.mod(even + 0.02 * g, box), np.mod(tight + 0.01 * g, box), s.vel, box


@pytest.mark.parametrize("side", [False, True])
def test_steps_after_a_larger_cluster_list(orc, side):
    even, tight, vel, box = lattices()
    st = torch.cuda.Stream() if side else torch.cuda.default_stream()
    with torch.cuda.stream(st):
        with md.System(even, vel, box, precision="mixed", force_variant=md.MD_FORCE_CLUSTER,
                       max_neighbors=400, dt=1e-4, stream=st if side else None) as a:
            a.step(21)  # captured and replayed steps of every kind
            s0 = a.stats()
            md.md_set_state(a.h, torch.as_tensor(tight, device="cuda"),
                            torch.as_tensor(vel, device="cuda"))
            md.md_build_neighbors(a.h)
            s1 = a.stats()
            a.step(21)
            x, v, f = (t.cpu().numpy() for t in a.state())
    # the fullest cell outgrew the headroom of the list, the rows did not
    assert s1["max_cell"] > 1.25 * s0["max_cell"] + 8 and s1["cap"] == s0["cap"]
    off, ids = orc.neighbors_cells(x, box, 2.8)
    _, f0 = orc.lj_list(x, box, off, ids)
    check(f, f0, near_cutoff(x, box, off, ids, 2.5, 1e-5))
