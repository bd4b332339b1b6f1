"""GPU tests of a batch whose members are all retired and replaced by others
of the same number and shape but another kind (precision, pipeline, fixed-count
selection, counting plane): the steps of the later members are those of a
handle that steps alone, so nothing captured for the earlier ones is replayed.
"""
import math

import numpy as np
import pytest

from paper_1808_03801_gb300 import workloads as W
from tests._util import KB_M_AR, assert_particles_close, by_pid

pytestmark = pytest.mark.gpu

VSCALE = math.sqrt(KB_M_AR * W.T0)
NY, PPC = 40, 60
KINDS = {
    "plain_fp32": ("fp32", "plain", {}),
    "plain_fp64": ("fp64", "plain", {}),
    "fused": ("fp32", "fused", {}),
    "fused_fixed_count": ("fp32", "fused", {"selection": "fixed_count"}),
    "fused_counting": ("fp32", "fused", {"flux_axis": 2, "flux_pos": 0.0}),
}


@pytest.fixture(scope="module")
def usp():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1808_03801_gb300 import usp as U
    U.lib()
    return U


def _sim(usp, kind, seed):
    precision, pipeline, extra = KINDS[kind]
    w = W.couette(ny=NY, ppc=PPC, precision=precision)
    w["params"].update(extra, pipeline=pipeline)
    if "flux_axis" in extra:
        w["params"]["flux_pos"] = 0.5 * w["grid"]["hi"][1]
    H = w["grid"]["hi"][1]
    pos, vel, pid = W.bimaxwellian(NY * PPC, seed=seed, y_range=(0.0, H))
    return usp.Simulation(w).set_particles(pos, vel, pid), H / NY


@pytest.mark.parametrize("first,second", [("plain_fp32", "plain_fp64"), ("plain_fp64", "plain_fp32"),
                                          ("fused", "plain_fp32"), ("plain_fp32", "fused"),
                                          ("fused", "fused_fixed_count"), ("fused", "fused_counting")])
def test_batch_refilled_with_members_of_another_kind(usp, first, second):
    """One step (the first is decided by the loaded state alone): FP64 to
    rounding, FP32 within rounding of its sums."""
    B = usp.Batch(hbm_budget=1 << 30, max_sims=2)
    for kind in (first, second):
        sims = [_sim(usp, kind, seed)[0] for seed in (21, 22)]
        for s in sims:
            assert B.admit(s) == 0
        B.step(1)
        for s in sims:
            B.retire(s)
    rtol = 1e-12 if second == "plain_fp64" else 1e-4
    for s, seed in zip(sims, (21, 22)):
        alone, dy = _sim(usp, second, seed)
        alone.step(1)
        a, b = s.info(), alone.info()
        assert a["step"] == 1 and a["counters"][5] == 0
        assert a["counters"][7] == b["counters"][7]
        assert_particles_close(s.particles(), alone.particles(), VSCALE, dy, rtol=rtol, check_cells=False)
        assert np.array_equal(s.sample()[15], alone.sample()[15])
    B.close()


def test_batch_of_every_kind_steps_as_each_alone(usp):
    """1-D and 2-D members with and without ablations, more cells in all than
    the block-per-cell form is used for: one kernel for each kind, side by side.
    Three steps; a particle within rounding of a face or of a selection may change
    its cells: three cells of a member at most."""
    def workloads(seed):
        out = [W.sod(ny=1000, ppc_left=80, seed=seed), W.couette(ny=700, ppc=60, seed=seed),
               W.cavity(n=25, ppc=40, Kn=0.05, seed=seed), W.poiseuille(ny=60, ppc=90, seed=seed),
               W.cavity(n=20, ppc=50, Kn=0.05, seed=seed), W.slit(nx=40, ny=20, ppc=30, seed=seed)]
        out = [W.with_precision(w, "fp32") for w in out]
        for w in out:
            w["params"]["pipeline"] = "fused"
        out[3]["params"]["selection"] = "fixed_count"
        out[4]["params"].update(mode="spesbgk", es_sampler="gallis_torczynski")
        return out

    ws = workloads(31)
    states = [usp.Simulation(w).init_particles().particles() for w in ws]
    sims = [usp.Simulation(w).set_particles(P["pos"], P["vel"], P["pid"]) for w, P in zip(ws, states)]
    alone = [usp.Simulation(w).set_particles(P["pos"], P["vel"], P["pid"]) for w, P in zip(ws, states)]
    assert sum(s.K for s in sims) > 1520 and all(s.tuning()["fused_R"] > 4 for s in alone)
    B = usp.Batch(hbm_budget=4 << 30, max_sims=len(ws))
    for s in sims:
        assert B.admit(s) == 0
    B.step(3)
    for s, a in zip(sims, alone):
        B.retire(s)
        a.step(3)
        assert s.info()["counters"][5] == 0
        assert abs(s.info()["counters"][4] - a.info()["counters"][4]) <= 3 * 100
        P, Q = (by_pid(x.particles()) for x in (s, a))
        assert np.array_equal(P["pid"], Q["pid"])
        bad = np.abs(P["vel"] - Q["vel"]).max(1) > 1e-4 * VSCALE
        assert len(set(Q["cell"][bad].tolist())) <= 3, (s.w["params"], bad.sum())
    B.close()
