"""Particles in the last place below the box's end, nextafter(n dx, 0): on these grids
x (1/dx) rounds to n, a cell past the last one.  They are pushed, moved and deposited as
any other, next to particles at x = 0 and elsewhere: against the oracle, FP64 1e-12,
mixed 5e-6 (the bars of the parity tests); more than 256 particles, so that they take
tiles, several along the axis (n = 104) or one (n = 13)."""
import numpy as np
import pytest

from oracle import oracle as orc
from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu

NAMES6 = ("e1", "e2", "e3", "b1", "b2", "b3")


@pytest.mark.parametrize("n", [(104, 13, 16), (16, 104, 13), (13, 17, 104), (104, 26), (40, 104)])
@pytest.mark.parametrize("precision, tol", [("fp64", 1e-12), ("mixed", 5e-6), ("compensated", 5e-6)])
def test_last_place_below_the_box_end(n, precision, tol):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    g = orc.Grid(n, dx, inputs.DT, cE, cB)
    sim = P.Simulation(n, dx, inputs.DT, cE, cB, precision=precision, pusher="boris")
    F = orc.Fields(g)
    for nm, a in zip(NAMES6, inputs.random_fields(g.shape, amp=0.5, seed=37)):
        getattr(F, nm)[...] = a
        sim.load_field(nm, a)
    Ps = inputs.random_particles(n, dx, 600, umax=0.5, seed=38)
    at_end = 0
    for d in range(len(n)):
        last = np.nextafter(n[d] * dx[d], 0.0)
        if np.floor(last * (1.0 / dx[d])) == n[d]:
            at_end += 1
            Ps.x[d][100 * d:100 * d + 60] = last
            Ps.x[d][100 * d + 60:100 * d + 80] = 0.0
            Ps.u[d][100 * d:100 * d + 20] = 0.0     # stay near the end
    assert at_end > 0
    sim.load_particles(Ps.x, Ps.u, Ps.w)
    Po = orc.Particles(Ps.x, Ps.u, Ps.w)
    for steps in (1, 4):
        orc.step(g, F, Po, nsteps=steps)
        sim.step(steps)
        for nm in NAMES6:
            ref = getattr(F, nm)
            assert np.abs(sim.read_field(nm) - ref).max() <= tol * max(np.abs(ref).max(), 0.5), nm
        x, u, _ = sim.read_particles()
        for c in range(3):
            assert np.abs(u[c] - Po.u[c]).max() <= tol * np.abs(Po.u[c]).max(), c
        for d in range(len(n)):
            L = g.length[d]
            assert np.abs((x[d] - Po.x[d] + L / 2) % L - L / 2).max() <= tol * L, d
    sim.close()
