"""Particle windows of the tile kernel: rows copied 16 bytes at a time or value by
value (x1 extents that are or aren't multiples of 16 bytes), windows larger than the
grid, tiles shrunk on small grids, several tiles sharing nodes across the periodic
seams.  Full steps with depositing particles against the oracle: 1e-12 in FP64, 5e-6
next to FP32 fields (the bars of the parity tests)."""
import numpy as np
import pytest

from oracle import oracle as orc
from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu

NAMES6 = ("e1", "e2", "e3", "b1", "b2", "b3")


@pytest.mark.parametrize("n", [(5, 3), (33, 9), (64, 16), (66, 20), (130, 37), (260, 70),
                               (6, 3, 2), (17, 9, 5), (40, 20, 12), (34, 18, 18)])
@pytest.mark.parametrize("precision, tol", [("fp64", 1e-12), ("mixed", 5e-6)])
def test_windows_equal_the_oracle(n, precision, tol):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    g = orc.Grid(n, dx, inputs.DT, cE, cB)
    sim = P.Simulation(n, dx, inputs.DT, cE, cB, precision=precision, pusher="boris")
    F = orc.Fields(g)
    for nm, a in zip(NAMES6, inputs.random_fields(g.shape, amp=0.5, seed=7)):
        getattr(F, nm)[...] = a
        sim.load_field(nm, a)
    Ps = inputs.random_particles(n, dx, 1500, umax=2.0, seed=8)
    sim.load_particles(Ps.x, Ps.u, Ps.w)
    Po = orc.Particles(Ps.x, Ps.u, Ps.w)
    orc.step(g, F, Po, nsteps=3)
    sim.step(3)
    for nm in NAMES6:
        ref = getattr(F, nm)
        assert np.abs(sim.read_field(nm) - ref).max() <= tol * np.abs(ref).max(), nm
    x, u, _ = sim.read_particles()
    for c in range(3):
        assert np.abs(u[c] - Po.u[c]).max() <= tol * np.abs(Po.u[c]).max(), c
    for d in range(len(n)):
        L = g.length[d]
        assert np.abs((x[d] - Po.x[d] + L / 2) % L - L / 2).max() <= tol * L, d
    sim.close()


@pytest.mark.parametrize("n", [(3, 2), (65, 9), (256, 40), (5, 3, 2), (40, 9, 6)])
@pytest.mark.parametrize("count", [1, 5, 256, 257])
@pytest.mark.parametrize("pusher", ["boris", "hc"])
def test_few_particles_equal_the_oracle(n, count, pusher):
    # up to 256 particles next to FP64 fields take a warp each, from 257 on tiles
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.25, 0.3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    dt = 0.25 * inputs.DX1
    g = orc.Grid(n, dx, dt, cE, cB)
    sim = P.Simulation(n, dx, dt, cE, cB, precision="fp64", pusher=pusher)
    F = orc.Fields(g)
    for nm, a in zip(NAMES6, inputs.random_fields(g.shape, amp=0.5, seed=17)):
        getattr(F, nm)[...] = a
        sim.load_field(nm, a)
    Ps = inputs.random_particles(n, dx, count, umax=2.0, seed=18)
    sim.load_particles(Ps.x, Ps.u, Ps.w)
    Po = orc.Particles(Ps.x, Ps.u, Ps.w)
    orc.step(g, F, Po, nsteps=25, pusher=pusher)
    sim.step(25)
    for nm in NAMES6:
        ref = getattr(F, nm)
        assert np.abs(sim.read_field(nm) - ref).max() <= 1e-12 * max(np.abs(ref).max(), 1.0), nm
    x, u, _ = sim.read_particles()
    for c in range(3):
        assert np.abs(u[c] - Po.u[c]).max() <= 1e-11 * np.abs(Po.u[c]).max(), c   # 25 chained pushes
    for d in range(len(n)):
        L = g.length[d]
        assert np.abs((x[d] - Po.x[d] + L / 2) % L - L / 2).max() <= 1e-12 * L, d
    sim.close()


@pytest.mark.parametrize("n", [(64, 32), (70, 33), (40, 20, 12)])
@pytest.mark.parametrize("precision, tol", [("fp64", 1e-12), ("mixed", 5e-6), ("compensated", 5e-6)])
@pytest.mark.parametrize("count", [1024, 1025, 9000])
def test_crowded_tiles_equal_the_oracle(n, precision, tol, count):
    # nearly all particles in a few cells: their tiles are shared by several CTAs (from
    # 1025 particles on), whose windows are added up, step after step
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    g = orc.Grid(n, dx, inputs.DT, cE, cB)
    sim = P.Simulation(n, dx, inputs.DT, cE, cB, precision=precision, pusher="boris")
    F = orc.Fields(g)
    for nm, a in zip(NAMES6, inputs.random_fields(g.shape, amp=0.5, seed=27)):
        getattr(F, nm)[...] = a
        sim.load_field(nm, a)
    Ps = inputs.random_particles(n, dx, count, umax=2.0, seed=28)
    for d in range(len(n)):   # the crowd: cells 6 .. 10 of each axis
        Ps.x[d][: count - 20] = (6 + 4 * Ps.x[d][: count - 20] / (n[d] * dx[d])) * dx[d]
    Ps.w[:] = -1e-4 * np.linspace(0.2, 1.0, count)
    sim.load_particles(Ps.x, Ps.u, Ps.w)
    Po = orc.Particles(Ps.x, Ps.u, Ps.w)
    for steps in (1, 3):
        orc.step(g, F, Po, nsteps=steps)
        sim.step(steps)
        for nm in NAMES6:
            ref = getattr(F, nm)
            assert np.abs(sim.read_field(nm) - ref).max() <= tol * max(np.abs(ref).max(), 0.5), nm
        x, u, _ = sim.read_particles()
        for c in range(3):
            assert np.abs(u[c] - Po.u[c]).max() <= tol * np.abs(Po.u[c]).max(), c
    sim.close()
