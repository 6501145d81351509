"""Per-replica energies of a batch where the sums' blocks have no atoms, one
partial round of threads, and more than one round (8,192 atoms per round)."""
import numpy as np
import pytest

from paper_1611_00075_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("cells", [(6,), (7, 16, 6), (13, 12, 20, 6)])
def test_replica_energies_equal_the_boxes_alone(cells):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_00075_gb300 import build, md
    build.build()
    reps = []
    for nc in cells:
        s = inputs.lj_fcc(nc=nc, T=1.0)
        g = inputs.gaussian(inputs.SEED_BASE + 700 + nc, s.pos.size).reshape(-1, 3)
        reps.append((np.mod(s.pos + 0.05 * g, s.box), s.vel, s.box))
    with md.Batch(reps, precision="mixed") as b:
        ke, pe = b.energies()
    for r, (pos, vel, box) in enumerate(reps):
        with md.System(pos, vel, box, precision="mixed") as a:
            pe1 = a.energy()[1]
        # two float64 sums of n positive terms, each within n 2^-53 of the exact
        # sum, of terms that carry a few roundings
        assert abs(ke[r] - 0.5 * np.sum(vel ** 2)) <= 2 * (len(pos) + 8) * 2.0 ** -53 * ke[r]
        # the same pairs in float32 chunks of possibly different lanes
        assert abs(pe[r] - pe1) <= 2e-6 * abs(pe1)
