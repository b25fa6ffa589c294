"""The laser-energy adjoint counts each step twice in the context's steps_done, forward
and for the reverse pass, whatever the segments are."""
import numpy as np
import pytest

from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("steps, every", [(20, 100), (20, 20), (21, 5), (1, 1)])
def test_steps_done(steps, every):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3)
    sim = P.Simulation((64, 16), (inputs.DX1, inputs.DX2), inputs.DT, cE, cB, precision="fp64")
    sim.step(3)
    las = P.pic_laser(2.0, 1.0, 0.0, 20 * inputs.DX1, 40 * inputs.DX1, 0.0, 0.0, 0.0)
    x = np.array([45 * inputs.DX1, 5 * inputs.DX2])
    P.pic_adjoint_laser_energy(sim.ctx, las, x, np.zeros(3), steps, every)
    assert sim.info().steps_done == 3 + 2 * steps
    sim.close()
