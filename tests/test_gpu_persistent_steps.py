"""The persistent step kernels on systems large enough for them (more items than
the resident CTAs hold: nine of 128 threads per SM, eight in float64): runs of
steps with rebuilds inside end in the bits of the grid launch, under every
scheduler and over per-atom rows, float64 rows and slots of two."""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu

LAYOUTS = {"full": (44, "mixed", 9), "fp64": (44, "fp64", 8), "paired": (56, "mixed", 9)}
SCHEDS = {"paircount": md.MD_SCHED_PAIRCOUNT, "mlp": md.MD_SCHED_MLP,
          "dynamic": md.MD_SCHED_DYNAMIC}


@pytest.fixture(scope="module", params=list(LAYOUTS))
def grid_run(request):
    nc, precision, ctas = LAYOUTS[request.param]
    s = inputs.lj_porous(nc=nc, fraction=0.4, rmin=2.0, rmax=6.0, T=1.2)
    pos = np.mod(s.pos + 0.05 * inputs.gaussian(821, s.pos.size).reshape(-1, 3), s.box)
    fv = md.MD_FORCE_PAIRED if request.param == "paired" else md.MD_FORCE_FULL
    items = (s.n + 1) // 2 if request.param == "paired" else s.n
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert items > sms * ctas * 128, "the grid launch would serve this size"

    def run(sched):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            with md.System(pos, s.vel, s.box, precision=precision, force_variant=fv,
                           scheduler=sched, stream=st) as a:
                b0 = a.stats()["builds"]
                a.step(1)
                a.step(30)
                assert a.stats()["builds"] - b0 >= 2
                return [t.cpu() for t in a.state()]

    return run, run(md.MD_SCHED_GRID)


@pytest.mark.parametrize("sched", list(SCHEDS))
def test_bits_of_the_grid_launch(grid_run, sched):
    run, want = grid_run
    for x, y in zip(run(SCHEDS[sched]), want):
        assert torch.equal(x, y)
