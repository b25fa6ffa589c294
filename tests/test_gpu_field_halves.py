"""The field step as a Faraday and an Ampere row pass (the default with particles, and
in vacuum on all but large 2D FP32 grids) against the fused kernel on CTA tiles: the
same bits, on rows shorter than a segment and than the stencil, ragged rows (partial
16-byte groups at both ends), single rows and planes, and stencils of every unrolled
length; with particles, against the oracle in the other parity tests."""
import numpy as np
import pytest

from oracle.gen_tables import load as load_table
from paper_2004_03754_gb300 import inputs

pytestmark = pytest.mark.gpu

NAMES6 = ("e1", "e2", "e3", "b1", "b2", "b3")


@pytest.mark.parametrize("n", [(1, 1), (3, 2), (7, 1), (34, 5), (129, 3), (1030, 4), (2051, 3), (2048, 600),
                               (5, 3, 2), (66, 4, 1), (131, 6, 5), (512, 5, 4)])
@pytest.mark.parametrize("precision", ["mixed", "fp64", "compensated"])
@pytest.mark.parametrize("M", [5, 16, 20])
def test_field_passes_equal_the_fused_kernel(n, precision, M):
    from paper_2004_03754_gb300 import pic as P
    cE, cB = load_table(16, 0.5, 0.3) if M == 16 else inputs.random_coeffs(M, seed=3)
    dx = (inputs.DX1, inputs.DX2, inputs.DX2)[:len(n)]
    dt = 0.25 * inputs.DX1
    out = []
    for fused in (False, True):
        sim = P.Simulation(n, dx, dt, cE, cB, precision=precision)
        if fused:
            sim.set_field_tile(64, 4, 2 if len(n) == 3 else 1, staging=1)
        for nm, a in zip(NAMES6, inputs.random_fields(sim.shape, amp=0.5, seed=11)):
            sim.load_field(nm, a)
        sim.step(3)
        out.append([sim.read_field(nm) for nm in NAMES6])
        sim.close()
    for nm, a, b in zip(NAMES6, *out):
        assert np.array_equal(a, b), nm
