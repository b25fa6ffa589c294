"""Momenta beyond FP32 arithmetic next to FP32 fields: an infinite or NaN momentum, or
one whose gamma^2 leaves FP32, is reported at the next sync and the particle stays
where it was; a momentum of 1e10 is pushed and moves at the speed of light."""
import numpy as np
import pytest

from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sim(n, pusher, u1, weight):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    sim = P.Simulation(n, dx, inputs.DT, cE, cB, precision="mixed", pusher=pusher)
    shape = tuple(reversed(n))
    for nm in ("e2", "b3"):
        sim.load_field(nm, np.full(shape, 0.5))
    x = np.array([[0.4 * n[d] * dx[d]] * 3 for d in range(len(n))])
    u = np.zeros((3, 3))
    u[0, 1] = u1
    sim.load_particles(list(x), list(u), np.full(3, weight))
    return P, sim, x, dx


@pytest.mark.parametrize("n", [(64, 16), (32, 16, 16)])
@pytest.mark.parametrize("pusher", ["boris", "analytic", "hc"])
@pytest.mark.parametrize("u1", [np.inf, -np.inf, np.nan, 1e39])
def test_non_finite_momentum_is_reported(n, pusher, u1):
    P, sim, x, dx = _sim(n, pusher, u1, -1e-6)
    sim.step(1)
    with pytest.raises(P.PicError, match="non-finite|proper-time|moved"):
        sim.sync()
    xr, ur, _ = sim.read_particles()
    for d in range(len(n)):
        assert xr[d][1] == x[d][1]
        assert np.isfinite(xr[d]).all()
    assert np.isfinite(sim.read_field("e1")).all()   # and deposited nothing
    sim.close()


@pytest.mark.parametrize("n", [(64, 16), (32, 16, 16)])
@pytest.mark.parametrize("pusher", ["boris", "analytic", "hc"])
@pytest.mark.parametrize("u1", [3e8, 1e10, 1e18])
def test_large_momentum_is_pushed(n, pusher, u1):
    P, sim, x, dx = _sim(n, pusher, u1, 0.0)
    sim.step(3)
    sim.sync()
    xr, ur, _ = sim.read_particles()
    assert abs(xr[0][1] - x[0][1] - 3 * inputs.DT) <= 1e-12 * x[0][1]
    assert abs(ur[0][1] - u1) <= 1e-8 * u1
    sim.close()
