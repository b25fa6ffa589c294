"""An infinite or NaN particle weight next to FP64 fields shows in the fields after the
step (the current around that particle is not a number), with tiles (more than 256
particles) and without; particles of another tile deposit as ever."""
import numpy as np
import pytest

from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(96, 48), (48, 24, 24)])
@pytest.mark.parametrize("count", [40, 300, 3000])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_weight_shows(n, count, bad):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    g = inputs.rng(3)
    x = [g.random(count) * 0.4 * n[d] * dx[d] for d in range(len(n))]
    for d in range(len(n)):
        x[d][0] = 0.8 * n[d] * dx[d]           # alone in its part of the box
    u = [g.normal(0.0, 0.5, count) for _ in range(3)]
    got = []
    for first in (-1e-4, bad):
        w = np.full(count, -1e-4)
        w[0] = first
        sim = P.Simulation(n, dx, inputs.DT, cE, cB, precision="fp64")
        sim.load_particles(x, u, w)
        sim.step(1)
        got.append([sim.read_field(f) for f in ("e1", "e2", "e3")])
        sim.close()
    k = tuple(int(0.8 * n[d]) for d in reversed(range(len(n))))
    low = tuple(slice(2, int(0.4 * n[d]) - 2) for d in reversed(range(len(n))))
    for a, b in zip(*got):
        assert np.isfinite(a).all()
        assert not np.isfinite(b[k])
        assert np.isfinite(b[low]).all() and np.abs(a[low] - b[low]).max() <= 1e-15
