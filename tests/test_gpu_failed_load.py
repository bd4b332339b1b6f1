"""GPU tests of loads that replace a stepped handle's storage.  One that runs
out of memory: whichever allocation fails, the handle has no state to step
(STATE), is not left with part of its storage, and loads and steps again once
there is memory.  Storage goes back to the caller's allocator only when no step
uses it any more."""
import ctypes
import math

import numpy as np
import pytest

from paper_1808_03801_gb300 import workloads as W
from tests._util import KB_M_AR, assert_particles_close

pytestmark = pytest.mark.gpu

VSCALE = math.sqrt(KB_M_AR * W.T0)


@pytest.fixture(scope="module")
def usp():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1808_03801_gb300 import usp as U
    U.lib()
    return U


class Memory:
    """Device memory whose allocations fail after `left` more (None: never)."""

    def __init__(self, usp):
        import torch
        self.left, self.held, self.on_free = None, {}, None

        def alloc(nbytes, ctx):
            if self.left is not None:
                if self.left == 0:
                    return None
                self.left -= 1
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.held[t.data_ptr()] = t
            return t.data_ptr()

        def free(p, ctx):
            if self.on_free:
                self.on_free()
            del self.held[p]

        self.struct = usp.Allocator()
        self.struct.alloc = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)(alloc)
        self.struct.free = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)(free)
        self.struct.ctx = None


@pytest.fixture
def memory(usp, monkeypatch):
    m = Memory(usp)
    monkeypatch.setattr(usp, "_torch_allocator", lambda: (m.struct, m))
    return m


def _state(n, H, seed):
    return W.bimaxwellian(n, seed=seed, y_range=(0.0, H))


@pytest.mark.parametrize("how", ["set", "init"])
@pytest.mark.parametrize("pipeline", ["plain", "fused"])
def test_a_load_that_runs_out_of_memory(usp, memory, pipeline, how):
    w = W.couette(ny=30, ppc=400, precision="fp64" if pipeline == "plain" else "fp32")
    w["params"]["pipeline"] = pipeline
    H = w["grid"]["hi"][1]
    small, large = _state(300, H, 1), _state(12000, H, 2)

    def load(g):
        return g.set_particles(*large) if how == "set" else g.init_particles()

    ref = load(usp.Simulation(w)).step(1)
    for k in range(20):
        memory.left = None
        g = usp.Simulation(w, allocator="torch").set_particles(*small).step(2)
        memory.left = k
        try:
            load(g)
            failed = False
        except usp.UspError as e:
            assert e.status == -2, e
            failed = True
            with pytest.raises(usp.UspError) as s:
                g.step(1)
            assert s.value.status == -6
            with pytest.raises(usp.UspError) as s:   # a retry fails alike
                memory.left = 0
                load(g)
            assert s.value.status == -2
            memory.left = None
            load(g)
        g.step(1)
        assert_particles_close(g.particles(), ref.particles(), VSCALE, H / 30,
                               rtol=1e-12 if pipeline == "plain" else 1e-4, check_cells=False)
        g.close()
        if not failed:
            break
    assert 6 < k < 20 and not memory.held


def test_storage_is_given_back_when_no_step_uses_it(usp, memory):
    """Steps are still running when a larger state is loaded."""
    w = W.cavity(n=100, ppc=100)
    w["params"]["pipeline"] = "fused"
    g = usp.Simulation(w, allocator="torch").init_particles().step(8)
    g.synchronize()
    idle = []
    memory.on_free = lambda: idle.append(g.stream.query())
    pos, vel, pid = W.bimaxwellian(3_000_000, seed=4, y_range=(0.0, 1.0e-4), x_range=(0.0, 1.0e-4))
    g.step(2000)
    assert not g.stream.query()
    g.set_particles(pos, vel, pid)
    memory.on_free = None
    assert len(idle) >= 7 and all(idle)
    assert g.step(1).info()["counters"][5] == 0
    g.close()
