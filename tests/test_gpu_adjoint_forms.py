"""The reverse pass of the laser-energy adjoint in its three forms -- few particles (a
warp each, the time-centred B's curl by atomics around the particle), more (a warp
each, the curl by grid passes) and many (a thread each) -- on the same electrons
repeated: the objective is a mean over electrons, so value and gradients agree to the
rounding of the sums, 200 steps of FP64 (1e-10)."""
import numpy as np
import pytest

from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pusher", ["boris", "analytic"])
@pytest.mark.parametrize("M, n", [(16, (300, 70)), (8, (301, 64))])
def test_adjoint_forms_agree(pusher, M, n):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(M, 0.5, 0.3 if M == 16 else 0.4)
    dx = (inputs.DX1, inputs.DX2)
    g = inputs.rng(5)
    k = 24
    x = np.array([(150 + 60 * g.random(k)) * dx[0], g.random(k) * n[1] * dx[1]])
    las = P.pic_laser(2.0, 1.0, 0.4, 120 * dx[0], 150 * dx[0], 6.0, n[1] * dx[1] / 2, 0.0)
    got = []
    for rep in (1, 30, 400):      # 24 (n <= cells/256), 720, 9600 (> 8192)
        sim = P.Simulation(n, dx, inputs.DT, cE, cB, precision="fp64", pusher=pusher)
        xs = np.tile(x, (1, rep)).reshape(-1)
        got.append(P.pic_adjoint_laser_energy(sim.ctx, las, xs, np.zeros(3 * k * rep), 60, 25))
        sim.close()
    for a in got[1:]:
        assert np.abs(np.array(a) - np.array(got[0])).max() <= 1e-10 * np.abs(np.array(got[0])).max()
