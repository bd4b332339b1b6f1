"""GPU test of a fused domain that outgrows its storage: a supersonic inflow
into a closed end.  The tight bucket layout runs past the capacity, so that the
last cells have no bucket, and the spill list is too short for what arrives in
them: cells with arrivals and not one particle kept.  The steps end, the loss is
reported as CAPACITY, and the handle can be loaded again."""
import numpy as np
import pytest

from paper_1808_03801_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def usp():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1808_03801_gb300 import usp as U
    U.lib()
    return U


@pytest.mark.parametrize("R", [4, 8, 12])
@pytest.mark.parametrize("dim", [1, 2])
def test_fused_domain_that_outgrows_its_storage(usp, dim, R):
    n, ppc = (64, 400) if dim == 1 else (16, 400)
    w = (W.homogeneous_column(ny=n, ppc=ppc, Kn=0.02, dt_over_tauc=30.0, precision="fp32") if dim == 1
         else W.cavity(n=n, ppc=ppc, Kn=0.01))
    flow = [0.0, 0.0, 0.0]
    flow[2 - dim] = 600.0
    for f in range(4):
        if dim == 2 or f >= 2:
            w["faces"][f] = {"kind": "specular", "T": W.T0, "u": (0.0, 0.0, 0.0), "n": 0.0}
    w["faces"][0 if dim == 2 else 2] = {"kind": "reservoir", "T": W.T0, "u": tuple(flow), "n": W.N0}
    w["params"].update(reservoir_cols=2, pipeline="fused", ppc_ref=ppc)
    g = usp.Simulation(w).init_particles(regions=[])
    cells = n ** dim
    # even at the reservoir's density the particles exceed the storage of an empty start, by more than the spill list
    cap = 24 * cells + 4 * 2 * n ** (dim - 1) * ppc + 4096 + 4
    assert cells * ppc > cap + 4096
    g.set_tuning(fused_R=R)
    for _ in range(15):
        g.step(20)
    with pytest.raises(usp.UspError) as e:
        g.synchronize()
    assert e.value.status == -4
    pos, vel, pid = W.bimaxwellian(100, seed=3, y_range=(0.0, w["grid"]["hi"][1]), x_range=(0.0, w["grid"]["hi"][0]))
    g.set_particles(pos, vel, pid).step(1)
    inf = g.info()
    assert inf["counters"][5] == 0 and inf["step"] == 1
    assert np.all(np.isfinite(g.sample()))
