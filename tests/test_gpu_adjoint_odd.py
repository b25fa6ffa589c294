"""The laser-energy adjoint on grids with an odd number of cells, where the states of a
segment kept one after another don't all fall on 16-byte boundaries by themselves: the
three forms of the reverse pass agree (1e-10, as on even grids), and value and gradients
meet central differences of the CPU oracle (1e-12 and 1e-6, the bars of the even grid),
with test electrons and with a depositing plasma."""
import numpy as np
import pytest

from oracle import oracle as orc
from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu

DX1, DX2, DT = inputs.DX1, inputs.DX2, inputs.DT


@pytest.mark.parametrize("pusher", ["boris", "analytic"])
@pytest.mark.parametrize("M, n", [(16, (301, 63)), (8, (67, 33))])
def test_adjoint_forms_agree(pusher, M, n):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(M, 0.5, 0.3 if M == 16 else 0.4)
    g = inputs.rng(5)
    k = 8
    x = np.array([n[0] * (0.5 + 0.2 * g.random(k)) * DX1, g.random(k) * n[1] * DX2])
    las = P.pic_laser(2.0, 1.0, 0.4, 0.4 * n[0] * DX1, 0.5 * n[0] * DX1, 6.0, n[1] * DX2 / 2, 0.0)
    got = []
    for rep in (1, 90, 1200):      # 8 (n <= cells/256), 720, 9600 (> 8192)
        sim = P.Simulation(n, (DX1, DX2), DT, cE, cB, precision="fp64", pusher=pusher)
        xs = np.tile(x, (1, rep)).reshape(-1)
        got.append(P.pic_adjoint_laser_energy(sim.ctx, las, xs, np.zeros(3 * k * rep), 60, 25))
        sim.close()
    for a in got[1:]:
        assert np.abs(np.array(a) - np.array(got[0])).max() <= 1e-10 * np.abs(np.array(got[0])).max()


@pytest.mark.parametrize("pusher, plasma", [("boris", False), ("analytic", False), ("boris", True)])
def test_gradient_matches_oracle_differences(pusher, plasma):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    n, nsteps = (127, 17), 90
    laser = dict(a0=2.0, k0=1.0, phase=0.3, Lenv=6 * np.pi, x_front=100 * DX1, w0=4.0, x2c=8 * DX2, x3c=0.0)
    if plasma:
        Pl = inputs.plasma(n, (DX1, DX2), 2, (96, 123), density=0.05, uth=0.0, seed=41)
        xs, w = Pl.x, Pl.w
    else:
        xs = [np.array([104, 106.5, 109, 111.2, 113, 114.7]) * DX1, np.array([6.1, 7.3, 8.0, 8.6, 9.4, 10.2]) * DX2]
        w = np.zeros(6)
    las = P.pic_laser(2.0, 1.0, 0.3, laser["Lenv"], laser["x_front"], laser["w0"], laser["x2c"], 0.0)
    sim = P.Simulation(n, (DX1, DX2), DT, cE, cB, precision="fp64", pusher=pusher)
    if plasma:
        J, ga, gp = P.pic_adjoint_laser_energy_w(sim.ctx, las, np.concatenate(xs), np.zeros(3 * w.size), w, nsteps, 40)
    else:
        J, ga, gp = P.pic_adjoint_laser_energy(sim.ctx, las, np.concatenate(xs), np.zeros(3 * w.size), nsteps, 40)
    sim.close()

    def energy(**kw):
        g = orc.Grid(n, (DX1, DX2), DT, cE, cB)
        F = orc.Fields(g)
        orc.laser_load(g, F, **{**laser, **kw})
        Po = orc.Particles(xs, [np.zeros(w.size)] * 3, w)
        orc.step(g, F, Po, pusher=pusher, nsteps=nsteps)
        return float(np.mean(np.sqrt(1 + Po.u[0] ** 2 + Po.u[1] ** 2 + Po.u[2] ** 2) - 1))

    J0 = energy()
    assert abs(J - J0) <= 1e-12 * abs(J0)
    fd_a = (energy(a0=2.0002) - energy(a0=1.9998)) / 4e-4
    fd_p = (energy(phase=0.3001) - energy(phase=0.2999)) / 2e-4
    assert abs(ga - fd_a) <= 1e-6 * abs(fd_a), (ga, fd_a)
    assert abs(gp - fd_p) <= 1e-6 * max(abs(fd_p), abs(fd_a)), (gp, fd_p)
