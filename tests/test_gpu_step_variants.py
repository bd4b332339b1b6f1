"""GPU tests of the forms a step's kernels take by size: tile and staging
edges, cells larger than what a block keeps, domains on both sides of a
layout's limit, cell faces, and the FP64 draws against extended precision.

FP64 is compared with the oracle per particle.  The fused FP32 forms are
compared with one another per particle: they take the same words from the same
counters, so with every particle relaxed (dt >> 1/nu) and P_ne given they
differ by FP32 rounding of the sums, about 1e-6 of the thermal speed; 1e-4 is
allowed.  A particle within rounding of a face (about 1e-6 of a cell) may end a
step in the next cell on one side only and shift both cells' corrections: at
most three cells may differ for that, and not the same ones for two seeds.
What no form may change is checked for each: no particle lost or doubled,
cells consistent with their counts, momentum and energy of a periodic domain.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1808_03801_gb300 import workloads as W
from tests._util import KB_M_AR, assert_particles_close, by_pid

pytestmark = pytest.mark.gpu

VSCALE = math.sqrt(KB_M_AR * W.T0)
EDGES = [16, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257, 383, 384, 385, 447, 448, 449, 511, 512, 513, 1023,
         1024, 1025, 1500]


@pytest.fixture(scope="module")
def usp():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1808_03801_gb300 import usp as U
    U.lib()
    return U


def _state(w, counts, seed):
    """counts[k] particles, uniform in cell k (by rows), of a uniform gas."""
    gr = w["grid"]
    nx = gr["nx"] if gr["dim"] == 2 else 1
    n = int(np.sum(counts))
    _, vel, pid = W.bimaxwellian(n, seed=seed, u=(20.0, -10.0, 5.0))
    rng = np.random.default_rng(seed + 1)
    cell = np.repeat(np.arange(len(counts)), counts)
    d = [(gr["hi"][a] - gr["lo"][a]) / m for a, m in ((0, nx), (1, gr["ny"]))]
    pos = np.empty((n, 2))
    pos[:, 0] = gr["lo"][0] + (cell % nx + rng.uniform(0.001, 0.999, n)) * d[0]
    pos[:, 1] = gr["lo"][1] + (cell // nx + rng.uniform(0.001, 0.999, n)) * d[1]
    return pos, vel, pid


def _domain(dim, ncells, ppc, reach):
    """Cells of a gas in which one step of 60 collision times crosses about
    `reach` cells."""
    kn = reach / 60.0
    if dim == 1:
        w = W.homogeneous_column(ny=ncells, ppc=ppc, Kn=kn, dt_over_tauc=60.0, mode="fixed", fixed_pne=0.4)
    else:
        n = math.isqrt(ncells)
        w = W.cavity(n=n, ppc=ppc, Kn=kn / n, dt_over_tauc=60.0, seed=3)
        w["params"].update(mode="fixed", fixed_pne=0.4)
    w["params"]["ppc_ref"] = ppc
    return W.with_precision(w, "fp32")


def _stepped(usp, w, st, R):
    pos, vel, pid = st
    w = dict(w, params=dict(w["params"], pipeline="fused"))
    g = usp.Simulation(w).set_particles(pos, vel, pid)
    if R:
        g.set_tuning(fused_R=R)
    g.step(3)
    assert g.info()["counters"][5] == 0
    assert g.info()["counters"][4] >= 2 * 0.99 * len(pid)        # every particle relaxed, twice so far
    N = g.sample()[15]
    P = by_pid(g.particles())
    assert np.array_equal(P["pid"], np.arange(len(pid), dtype=np.uint32))
    assert np.array_equal(np.bincount(P["cell"], minlength=len(N)), N.astype(np.int64))
    if w["grid"]["dim"] == 1:   # FP32 rounding of the particles and of each cell's factors
        assert np.all(np.abs(P["vel"].sum(0) - vel.sum(0)) < 2e-6 * np.abs(vel).sum())
        assert abs((P["vel"] ** 2).sum() - (vel ** 2).sum()) < 1e-5 * (vel ** 2).sum()
    g.close()
    return P


def _differing_cells(usp, w, counts, R, R_ref, seed):
    st = _state(w, counts, seed)
    a, b = _stepped(usp, w, st, R), _stepped(usp, w, st, R_ref)
    bad = np.abs(a["vel"] - b["vel"]).max(1) > 1e-4 * VSCALE
    return set(b["cell"][bad].tolist())


@pytest.mark.parametrize("R", [4, 12])
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("reach", [0.02, 1.0])
def test_fused_cell_sizes(usp, dim, R, reach):
    """Cells at the edges of tiles, staging and register capacity: a warp
    per cell (4) and a block of eight warps (12) against a block of four (8);
    reach 1: most particles leave their cell."""
    # (1-D is periodic: up and down again, since a cell of 16 beside one of 1500
    # that empties into it asks for more spill entries than there are)
    counts = EDGES + EDGES[::-1] if dim == 1 else EDGES
    w = _domain(dim, len(counts), int(np.mean(counts)), reach)
    sets = [_differing_cells(usp, w, counts, R, 8, seed) for seed in (5, 6)]
    assert max(map(len, sets)) <= 3 and not sets[0] & sets[1], sets


@pytest.mark.parametrize("ppc_ref", [100, 450])
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("reach", [0.02, 1.0])
def test_fused_warp_per_cell_staging(usp, dim, ppc_ref, reach):
    """The warp form with four blocks per SM (100 particles per cell meant) and
    with three and more staging (450): cells at the edges of either area and in
    several chunks, against blocks of four warps."""
    counts = EDGES + [575, 577, 639, 640, 641, 704, 735, 736, 737, 800, 900]
    if dim == 1:
        counts = counts + counts[::-1]
    w = _domain(dim, len(counts), int(np.mean(counts)), reach)
    w["params"]["ppc_ref"] = ppc_ref
    sets = [_differing_cells(usp, w, counts, 4, 8, seed) for seed in (14, 15)]
    assert max(map(len, sets)) <= 3 and not sets[0] & sets[1], sets


@pytest.mark.parametrize("ablation", [{"selection": "fixed_count"}, {"mode": "spesbgk", "es_sampler": "gallis_torczynski"},
                                      {"selection": "fixed_count", "mode": "spesbgk", "es_sampler": "gallis_torczynski"}])
@pytest.mark.parametrize("ppc_ref", [360, 500])
@pytest.mark.parametrize("dim", [1, 2])
def test_fused_ablations_warp_per_cell(usp, dim, ppc_ref, ablation):
    """The ablations with a warp per cell (four and three blocks per SM)
    against blocks of four warps, at one collision time, so that the fixed count
    takes a part of each cell; cells of several chunks and with spill-list
    entries among them."""
    counts = EDGES + EDGES[::-1] if dim == 1 else EDGES
    n = len(counts)
    for reach in (0.02, 1.0):
        if dim == 1:
            w = W.homogeneous_column(ny=n, ppc=360, Kn=reach, dt_over_tauc=1.0, precision="fp32")
        else:
            w = W.cavity(n=math.isqrt(n), ppc=360, Kn=reach / math.isqrt(n), dt_over_tauc=1.0)
        w["params"].update(ablation, pipeline="fused", ppc_ref=ppc_ref)
        bad = []
        for seed in (16, 17):
            st = _state(w, counts, seed)
            P = []
            for R in (4, 8):
                g = usp.Simulation(w).set_particles(*st).set_tuning(fused_R=R).step(3)
                assert g.info()["counters"][5] == 0 and 0 < g.info()["counters"][4] < 2 * len(st[2])
                N = g.sample()[15]
                P.append(by_pid(g.particles()))
                assert np.array_equal(P[-1]["pid"], np.arange(len(st[2]), dtype=np.uint32))
                assert np.array_equal(np.bincount(P[-1]["cell"], minlength=n), N.astype(np.int64))
                g.close()
            d = np.abs(P[0]["vel"] - P[1]["vel"]).max(1) > 1e-4 * VSCALE
            bad.append(set(P[1]["cell"][d].tolist()))
        assert max(map(len, bad)) <= 3 and not bad[0] & bad[1], (reach, bad)


@pytest.mark.parametrize("R", [4, 12])
def test_fused_cells_with_long_spill_lists(usp, R):
    """Cells of 16 and 1500 particles side by side at reach 1: hundreds go to
    the spill list for one cell.  All of them count in the cell's moments and go
    on with it."""
    counts = EDGES
    w = _domain(1, len(counts), int(np.mean(counts)), 1.0)
    g = usp.Simulation(dict(w, params=dict(w["params"], pipeline="fused"))).set_particles(*_state(w, counts, 5))
    g.set_tuning(fused_R=R).step(1)
    assert g.info()["counters"][5] == 0 and g.info()["counters"][6] > 128
    g.close()
    sets = [_differing_cells(usp, w, counts, R, 8, seed) for seed in (5, 6)]
    assert max(map(len, sets)) <= 3 and not sets[0] & sets[1], sets


@pytest.mark.parametrize("selection", ["bernoulli", "fixed_count"])
@pytest.mark.parametrize("R", [4, 8, 12])
@pytest.mark.parametrize("dim", [1, 2])
def test_fused_counting_plane_in_every_form(usp, dim, R, selection):
    """Net flow through a plane in closed walls: the particles at or above it
    after each step less those before."""
    w = W.couette(ny=30, ppc=80, dt_over_tauc=3.0) if dim == 1 else W.cavity(n=12, ppc=40, Kn=0.05)
    w = W.with_precision(w, "fp32")
    w["params"].update(pipeline="fused", selection=selection, flux_axis=2, flux_pos=0.37 * w["grid"]["hi"][1])
    g = usp.Simulation(w).init_particles().set_tuning(fused_R=R)
    plane = np.float32(w["params"]["flux_pos"])

    def above():
        return int(np.sum(g.particles()["pos"][:, 1].astype(np.float32) >= plane))

    before, counted = above(), 0
    for _ in range(4):
        g.step(2)
        now = above()
        assert g.info()["counters"][7] - counted == now - before
        counted, before = g.info()["counters"][7], now
    assert g.info()["counters"][5] == 0


@pytest.mark.parametrize("ncells", [1, 8191, 8192, 8193])
def test_fused_layout_on_both_sides_of_the_one_kernel_limit(usp, ncells):
    w = _domain(1, ncells, 16, 0.02)
    sets = [_differing_cells(usp, w, [16] * ncells, 0, 8, seed) for seed in (7, 8)]
    assert max(map(len, sets)) <= 3 and not sets[0] & sets[1], sets


@pytest.mark.parametrize("selection", ["bernoulli", "fixed_count"])
@pytest.mark.parametrize("mode", ["usp", "spesbgk"])
def test_fp64_relaxation_chunks_match_oracle(usp, selection, mode):
    """Cells around the 512 particles whose draws are kept, and the 1024
    selection words that are staged."""
    counts = [2, 3, 127, 128, 129, 511, 512, 513, 1023, 1024, 1025, 1100]
    w = W.homogeneous_column(ny=len(counts), ppc=500, Kn=0.02, dt_over_tauc=1.5)
    w["params"].update(mode=mode, selection=selection)
    st = _state(w, counts, 9)
    g, o = usp.Simulation(w).set_particles(*st), oracle.OracleSim(w).set_particles(*st)
    for _ in range(2):
        g.step(1)
        o.step(1)
        assert_particles_close(g.particles(), o.particles(), VSCALE, 1e-6, rtol=1e-11)
        assert np.array_equal(g.params()[:, 15], o.params()[:, 15])


def test_weighted_relaxation_of_large_cells_matches_oracle(usp):
    """One cell below and one above the 2048 selection words that are kept."""
    counts = [700, 2040, 2300, 2500]
    w = W.homogeneous_column(ny=4, ppc=2000, Kn=0.02, dt_over_tauc=1.5, mode="fixed", fixed_pne=0.5)
    w["params"].update(weighted=1, capacity_factor=8.0)
    st = _state(w, counts, 10)
    g, o = usp.Simulation(w).set_particles(*st), oracle.OracleSim(w).set_particles(*st)
    for _ in range(2):
        g.step(1)
        o.step(1)
        assert_particles_close(g.particles(), o.particles(), VSCALE, 1e-6, rtol=1e-10)


@pytest.mark.parametrize("dim", [1, 2])
def test_fp64_cells_at_faces_match_oracle(usp, dim):
    """Particles at rest on cell faces and a few units in the last place to
    either side: the cell found with the reciprocal is the divided one.
    (Of odd cell counts, so that faces are rounded.)"""
    n = 77
    w = W.cavity(n=n, ppc=9, precision="fp64") if dim == 2 else W.couette(ny=n, ppc=9, precision="fp64")
    L = w["grid"]["hi"][1]
    face = np.arange(1, n) * (L / n)
    y = np.concatenate([face] + [face + s * k * np.spacing(face) for s in (1, -1) for k in (1, 2, 3)])
    rng = np.random.default_rng(11)
    pos = np.stack([rng.permutation(y) if dim == 2 else np.zeros(len(y)), y], 1)
    vel = np.zeros((len(y), 3))
    pid = np.arange(len(y), dtype=np.uint32)
    g, o = usp.Simulation(w).set_particles(pos, vel, pid), oracle.OracleSim(w).set_particles(pos, vel, pid)
    g.step(1)
    o.step(1)
    P, Q = by_pid(g.particles()), by_pid(o.particles())
    assert np.array_equal(P["cell"], Q["cell"]) and np.array_equal(P["pos"][:, 1], Q["pos"][:, 1])


@pytest.mark.parametrize("pipeline", ["plain", "fused"])
def test_steps_after_a_reload_are_those_of_a_new_handle(usp, pipeline):
    """The captured step is kept over a load into the same storage."""
    w = W.couette(ny=40, ppc=60, precision="fp64" if pipeline == "plain" else "fp32")
    w["params"]["pipeline"] = pipeline
    a, b = _state(w, [60] * 40, 12), _state(w, [30] * 20 + [80] * 20, 13)
    g = usp.Simulation(w).set_particles(*a)
    g.step(3)
    g.set_particles(*b)
    h = usp.Simulation(w).set_particles(*b)
    g.step(1)
    h.step(1)
    dy = w["grid"]["hi"][1] / 40
    assert_particles_close(g.particles(), h.particles(), VSCALE, dy, rtol=1e-12 if pipeline == "plain" else 1e-4,
                           check_cells=False)
    assert np.array_equal(g.sample()[15], h.sample()[15])


def test_fp64_normals_against_extended_precision(usp):
    """The initial velocities are sqrt(theta) z with z of two Box-Muller
    pairs.  Against extended precision, z is off by a few units in the last
    place: root 1, logarithm 0.3 (half of 0.6), sine or cosine 1.2, the two
    products 0.5 each, sqrt(theta) 0.5: 4."""
    w = W.homogeneous_box(ppc=200_000)
    seed = 0x1234ABCD
    g = usp.Simulation(w).init_particles(seed=seed)
    P = by_pid(g.particles())
    n = len(P["pid"])
    assert n > 100_000
    ctr = np.zeros((n, 4), np.uint32)
    ctr[:, 0], ctr[:, 3] = P["pid"], 1
    v = usp.debug_philox(ctr, (seed, 0)).astype(np.int64)
    F = np.longdouble
    theta = F(w["regions"][0]["T"]) * F(1.380649e-23) / F(w["gas"]["mass"])
    pi = F("3.14159265358979323846264338327950288")

    def pair(a, b):
        u = (a.astype(F) + F(0.5)) / F(2) ** 32
        r = np.sqrt(-2 * np.where(u > 0.5, np.log1p(u - 1), np.log(u)))
        t = 2 * b + 1                                  # units of pi 2^-32
        q = (t + (1 << 30)) >> 31                      # nearest quarter turn
        d = (t - (q << 31)).astype(F) * (pi / F(2) ** 32)
        s, c = np.sin(d), np.cos(d)
        return r * np.choose(q & 3, [c, -s, -c, s]), r * np.choose(q & 3, [s, c, -s, -c])

    z0, z1 = pair(v[:, 0], v[:, 1])
    z2, _ = pair(v[:, 2], v[:, 3])
    for k, z in enumerate((z0, z1, z2)):
        ref = np.sqrt(theta) * z
        err = np.abs(P["vel"][:, k].astype(F) - ref) / np.spacing(np.abs(ref).astype(np.float64))
        # (theta's own rounding: two operations, half of it through the root)
        assert err.max() <= 5.0, (k, err.max())
