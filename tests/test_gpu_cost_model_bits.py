"""Sampling and profiling the cost model time force passes of the persistent
kernel; they do not change what the system computes next.  A run with both calls
between its steps ends in the same bits as a run without, on sizes whose steps
share an atom between lanes and on sizes that do not."""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["full", "paired"])
@pytest.mark.parametrize("sched", ["grid", "mlp"])
@pytest.mark.parametrize("nc", [6, 20, 42])
def test_profiling_keeps_the_trajectory(variant, sched, nc):
    s = inputs.lj_fcc(nc=nc, T=0.72)
    pos = np.mod(s.pos + 0.05 * inputs.gaussian(811, s.pos.size).reshape(-1, 3), s.box)
    fv = md.MD_FORCE_PAIRED if variant == "paired" else md.MD_FORCE_FULL
    sc = md.MD_SCHED_MLP if sched == "mlp" else md.MD_SCHED_GRID
    out = []
    for profile in (False, True):
        with md.System(pos, s.vel, s.box, precision="mixed", force_variant=fv,
                       scheduler=sc) as a:
            a.step(4)
            if profile:
                assert md.md_cost_model(a.h, md.MD_COST_SAMPLE) > 0
                a.step(3)
                md.md_cost_model(a.h, md.MD_COST_PROFILE)
                a.step(3)
            else:
                a.step(3)
                a.step(3)
            out.append(a.state())
    for x, y in zip(*out):
        assert torch.equal(x, y)


def test_profiling_adds_no_timed_force_pass():
    s = inputs.lj_fcc(nc=6, T=0.72)
    with md.System(s.pos, s.vel, s.box, precision="mixed") as a:
        a.step(4)
        md.md_set_timing(a.h, True)
        md.md_cost_model(a.h, md.MD_COST_SAMPLE)
        a.step(5)
        assert a.stats()["count"]["force"] == 5
