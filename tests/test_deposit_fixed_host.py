"""The integer form of the FP64 current deposit (csrc/particle_core.cuh, deposit_fixed)
against its FP64 form, compiled by nvcc and run on the host: moves that stay on and
cross the nearest node, no move, moves of one part in 1e12, positions on the node and
half-node boundaries, weights far below the tile's largest, windows of few and of many
particles.  CPU only."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2004_03754_gb300", "csrc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("dfix") / "deposit_fixed_check_host")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                           "--expt-relaxed-constexpr", "-diag-suppress", "128", "-I", CSRC,
                           "-I", os.path.join(ROOT, "include"), "-o", exe,
                           os.path.join(HERE, "native", "deposit_fixed_check_host.cu")])
    return exe


@pytest.mark.parametrize("ndim", [2, 3])
@pytest.mark.parametrize("limb", [21, 17, 8])
def test_integer_deposit_equals_the_fp64_one(harness, tmp_path, ndim, limb):
    rng = np.random.Generator(np.random.PCG64(11))
    eps = 2.0 ** -53
    cases = []
    fs = [0.0, 0.5, 0.5 - eps, 1 - eps, 0.25, 1e-9]
    ds = [0.0, 1e-12, -1e-12, 0.5, -0.5, 0.3, -0.9, 1 - eps, -(1 - eps), 1e-300]
    for f in fs:
        for d in ds:
            cases.append((1.0, 1.0, 0.3, [f] * 3, [d] * 3))
    for _ in range(300):
        w = 10.0 ** rng.uniform(-12, 0) * rng.choice([-1, 1])
        cases.append((1.0, w, rng.uniform(-1, 1), rng.random(3), rng.uniform(-1, 1, 3)))
        cases.append((3e-3, 3e-3 * rng.random(), 1e-6 * rng.uniform(-1, 1), rng.random(3),
                      10.0 ** rng.uniform(-9, 0) * rng.uniform(-1, 1, 3)))
    cases.append((1.0, 5e-324, 0.1, rng.random(3), rng.uniform(-1, 1, 3)))
    fin, fout = tmp_path / "in.bin", tmp_path / "out.bin"
    with open(fin, "wb") as h:
        h.write(struct.pack("<i", len(cases)))
        for bound, w, v3, f, d in cases:
            h.write(struct.pack("<2i", ndim, limb))
            h.write(struct.pack("<3d", bound, w, v3))
            for a in range(3):
                h.write(struct.pack("<3d", f[a], d[a], (2.0, 8.0, 8.0)[a]))
    subprocess.check_call([harness, str(fin), str(fout)])
    got = np.fromfile(fout, dtype="<f8").reshape(len(cases), 2)
    for (bound, w, v3, f, d), (worst, _) in zip(cases, got):
        # the FP64 form's shapes carry 2^-54 each, their differences and running sums a few
        # of them, times |w| dx/dt <= 8 |w| (and |w v3|); plus half a unit of the window,
        # 2^-(19 - log2(bound) rounded + 2 limb)
        unit = 2.0 ** -(19 - np.floor(np.log2(bound)) + 2 * limb)
        assert worst <= 8 * abs(w) * 8 * 2.0 ** -53 + unit, (bound, w, v3, f, d, worst)
