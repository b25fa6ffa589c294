"""Ensembles with few particles (a warp each) and with many (32 to a warp), on runs
narrower than the stencil's ghost columns, ragged ones and ones of a few rows, with
particles next to every edge: each run against the oracle at 1e-12 (FP64)."""
import numpy as np
import pytest

from oracle import oracle as orc
from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [(20, 6), (71, 3), (130, 17)]


@pytest.mark.parametrize("per_run", [7, 170, 171, 400])   # 21, 510 | 513, 1200 particles
@pytest.mark.parametrize("pusher", ["boris", "hc"])
@pytest.mark.parametrize("depositing", [False, True])
def test_particles_of_an_ensemble(per_run, pusher, depositing):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    dx, dt, steps = (inputs.DX1, inputs.DX2), inputs.DT, 3
    ens = P.Ensemble([s[0] for s in SIZES], [s[1] for s in SIZES], dx, dt, cE, cB, precision="fp64",
                     pusher=pusher)
    lasers, parts = [], []
    for r, (a, b) in enumerate(SIZES):
        L = 0.5 * a * dx[0]
        lasers.append(P.pic_laser(2.0 + r, 1.0, 0.3 * r, L, L + 2 * dx[0], 3.0, b * dx[1] / 2, 0.0))
        ps = inputs.random_particles((a, b), dx, per_run, umax=1.5, seed=40 + r)
        edge = 1e-9 * np.array([1.0, 0.0])   # the box corners
        ps.x[0][:2], ps.x[1][:2] = edge, edge[::-1]
        ps.x[0][2], ps.x[1][2] = a * dx[0] * (1 - 1e-12), b * dx[1] * (1 - 1e-12)
        if not depositing:
            ps.w[:] = 0.0
        parts.append(ps)
    ens.load_lasers(lasers)
    ens.load_particles([per_run] * len(SIZES), [np.concatenate([p.x[d] for p in parts]) for d in range(2)],
                       [np.concatenate([p.u[c] for p in parts]) for c in range(3)],
                       np.concatenate([p.w for p in parts]))
    ens.set_steps([steps] * len(SIZES))
    ens.run()
    x, u, _ = ens.read_particles()
    for r, (size, las, ps) in enumerate(zip(SIZES, lasers, parts)):
        g = orc.Grid(size, dx, dt, cE, cB)
        F = orc.Fields(g)
        orc.laser_load(g, F, a0=las.a0, k0=1.0, phase=las.phase, Lenv=las.L_env, x_front=las.x_front,
                       w0=las.w0, x2c=las.x2c)
        Po = orc.Particles(ps.x, ps.u, ps.w)
        orc.step(g, F, Po, nsteps=steps, pusher=pusher)
        q = slice(r * per_run, (r + 1) * per_run)
        for c in range(3):
            assert np.abs(u[c][q] - Po.u[c]).max() <= 1e-12 * max(np.abs(Po.u[c]).max(), 1.0), (r, c)
        for d in range(2):
            Ld = g.length[d]
            assert np.abs((x[d][q] - Po.x[d] + Ld / 2) % Ld - Ld / 2).max() <= 1e-12 * Ld, (r, d)
        for nm in ("e1", "e2", "e3", "b1", "b2", "b3"):
            ref = getattr(F, nm)
            scale = max(np.abs(ref).max(), 1e-3)
            assert np.abs(ens.read_field(r, nm) - ref).max() <= 1e-12 * scale, (r, nm)
    ens.close()
