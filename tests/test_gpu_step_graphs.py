"""Replayed steps against launched ones.  md_step replays captured runs of eight,
two and one steps and a captured last step, one set per parity of the double
buffer, on side streams and on the default stream alike; with per-launch timing
on, every kernel is launched by itself, which makes it the plain run here.  Calls
of all lengths around those runs, from either parity, with rebuilds inside them,
end in the same bits, whatever the layout, potential and precision."""
import numpy as np
import pytest
import torch

from paper_1611_00075_gb300 import inputs, md

pytestmark = pytest.mark.gpu

CALLS = [1, 2, 3, 4, 9, 10, 12, 18, 19]  # odd sums between them: both parities


def system(name):
    kw = dict(precision="mixed", dt=0.005)
    if name == "sc":
        s = inputs.sc_fcc(nc=8)
        p = s.params
        kw.update(potential="sc", eps=p["eps"], sigma=p["sigma"], c=p["c"], n_exp=p["n_exp"],
                  m_exp=p["m_exp"], rc=p["rc"], skin=p["skin"], dt=p["dt"])
    elif name == "eam":
        s = inputs.eam_bcc(nc=9)
        p = s.params
        keys = ("phi_r", "phi_a", "psi_r", "psi_a", "F_sqrt", "F_quad")
        kw.update(eam={k: p[k] for k in keys}, rc=p["rc"], skin=p["skin"], dt=p["dt"])
    elif name == "alloy":
        s = inputs.lj_alloy(nc=7)
        p = s.params
        kw.update(rc=p["rc"], skin=p["skin"], dt=p["dt"],
                  species=(p["types"], p["t_eps"], p["t_sigma"], p["t_mass"]))
    else:
        s = inputs.lj_fcc(nc=8, T=1.0)
        kw["precision"] = "fp64" if name == "fp64" else "mixed"
        kw["force_variant"] = {"cluster": md.MD_FORCE_CLUSTER, "paired": md.MD_FORCE_PAIRED,
                               "color": md.MD_FORCE_HALF_COLOR}.get(name, md.MD_FORCE_FULL)
    return s, kw


@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("name", ["full", "paired", "fp64", "color", "cluster", "overlap", "sc",
                                  "eam", "alloy"])
def test_replay_equals_launches(name, first):
    s, kw = system(name)
    out = []
    for mode in ("plain", "side", "default"):
        st = torch.cuda.default_stream() if mode == "default" else torch.cuda.Stream()
        with torch.cuda.stream(st):
            # every seventh step rebuilds, so that runs of eight hold a rebuild
            with md.System(s.pos, s.vel, s.box, rebuild_every=7,
                           stream=None if mode == "default" else st, **kw) as a:
                if name == "overlap":
                    md.md_set_decomposition(a.h, 2, 2, 2)
                md.md_set_timing(a.h, mode == "plain")
                b0 = a.stats()["builds"]
                got = []
                for n in [1] * first + CALLS:
                    a.step(n)
                    got.append([t.cpu() for t in a.state()])
                assert a.stats()["builds"] - b0 >= 8
        out.append(got)
    for other in out[1:]:
        for n, (x, y) in enumerate(zip(out[0], other)):
            for p, q in zip(x, y):
                assert torch.equal(p, q), (name, n)
