"""Slot lists built a thread per slot where the slots of one warp scan cells of
very different sizes -- empty ones, one-atom ones and ones of several rounds --
in one box and in a batch: forces against the oracle with the mixed path's bar
(2e-4 relative, 1e-5 of the rms; atoms with a pair within rounding of the cutoff
left out)."""
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


def blobs(nc, seed):
    """A porous crystal with a tenth of its atoms taken out at random, squeezed
    along x by a wave: neighbouring cells of none to about 60 atoms."""
    s = inputs.lj_porous(nc=nc, fraction=0.35, rmin=2.0, rmax=5.0)
    keep = inputs.uniform(seed, s.n) > 0.1
    pos = s.pos[keep] + 0.03 * inputs.gaussian(seed + 1, 3 * int(keep.sum())).reshape(-1, 3)
    L = s.box[0]
    pos[:, 0] += 0.35 * L / (2 * np.pi) * np.sin(2 * np.pi * pos[:, 0] / L)
    return np.mod(pos, s.box), s.box


def compare(orc, f, pos, box):
    off, ids = orc.neighbors_cells(pos, box, 2.8)
    _, f0 = orc.lj_list(pos, box, off, ids)
    check(f, f0, near_cutoff(pos, box, off, ids, 2.5, 1e-5))


def test_one_box(orc):
    pos, box = blobs(32, 840)
    assert len(pos) // 2 > 24576
    _, _, start, _ = orc.bin_cells(pos, box, 2.8)
    cells = np.diff(start)
    assert cells.min() == 0 and cells.max() > 28 and (cells == 1).any()
    with md.System(pos, np.zeros_like(pos), box, precision="mixed",
                   force_variant=md.MD_FORCE_PAIRED) as a:
        compare(orc, a.state()[2].cpu().numpy(), pos, box)


def test_batch(orc):
    reps = [blobs(nc, 850 + nc) for nc in (22, 7, 24, 9, 23)]
    with md.Batch([(p, np.zeros_like(p), b) for p, b in reps], precision="mixed",
                  force_variant=md.MD_FORCE_PAIRED) as a:
        assert a.n // 2 > 24576
        f = a.state()[2].cpu().numpy()
        for r, (p, b) in enumerate(reps):
            compare(orc, f[a.offsets[r]:a.offsets[r + 1]], p, b)


@pytest.mark.parametrize("half", [False, True])
@pytest.mark.parametrize("nc", [9, 20, 24])  # a warp per row (1.6 and 18 thousand atoms), a thread per row
def test_rows_around_one_atom_cells(orc, nc, half):
    """Per-atom rows of the same systems: exact sets, empty and one-atom cells
    among their stencils."""
    pos, box = blobs(nc, 850 + nc)
    assert (len(pos) <= 24576) == (nc < 24)
    off, ids = orc.neighbors_cells(pos, box, 2.8, half=half)
    cells = np.diff(orc.bin_cells(pos, box, 2.8)[2])
    assert cells.min() == 0 and (cells == 1).any()
    fv = md.MD_FORCE_HALF_ATOMIC if half else md.MD_FORCE_FULL
    with md.System(pos, np.zeros_like(pos), box, precision="mixed", force_variant=fv) as a:
        goff, gids = a.neighbors(half=half)
    np.testing.assert_array_equal(goff.cpu().numpy(), off)
    np.testing.assert_array_equal(gids.cpu().numpy(), ids)
