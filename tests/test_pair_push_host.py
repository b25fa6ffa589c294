"""The momentum advance of particles in FP32 fields (csrc/pair_push.cuh: FP32
pairs, added to the FP64 state) and the series form of the analytic push
(csrc/analytic_series.cuh), compiled for the host, against the oracle's pushers:
zero, weak, strong (past the series: the FP64 form) and null fields, from rest to
gamma = 1e4.  CPU only."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

from oracle import oracle as orc

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2004_03754_gb300", "csrc")
DT = 0.0981747704


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("pair") / "pair_push_check_host")
    subprocess.check_call([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-Wno-unknown-pragmas",
                           "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", exe,
                           os.path.join(HERE, "native", "pair_push_check_host.cpp")])
    return exe


def _cases():
    rng = np.random.Generator(np.random.PCG64(23))
    out = [(np.zeros(6), np.zeros(3)), (np.zeros(6), np.array([3.0, -1e-7, 1e-30])),
           (np.array([0, 1e-25, 0, 0, 0, 1e-25]), np.zeros(3)),
           (np.array([0, 1e-25, 0, 0, 0, 1e-25]), np.array([1e-20, 0, 0]))]
    for scale in (1e-6, 0.1, 1.0, 30.0, 300.0):
        for um in (0.0, 1.0, 1e4):
            for _ in range(8):
                out.append((rng.uniform(-scale, scale, 6), um * rng.uniform(-1, 1, 3)))
    for E in (0.5, 5.0, 50.0, 500.0):    # plane waves: |E| = |B|, E.B = 0
        out.append((np.array([0.0, E, 0.0, 0.0, 0.0, E]), np.array([20.0, 1.0, -0.5])))
        out.append((np.array([0.0, E, 0.0, 0.0, 0.0, E]), np.zeros(3)))
    return [(eb.astype(np.float32).astype(np.float64), u) for eb, u in out]


# a pair operation is good to a few 2^-47 of its operands and a push chains about
# thirty: 30 * 4 * 2^-47 = 8.5e-13; FP64: 1e-13 as the form it stands for
@pytest.mark.parametrize("kind, tol", [(0, 8.5e-13), (1, 8.5e-13), (2, 8.5e-13), (3, 1e-13)],
                         ids=["boris", "analytic", "hc", "series"])
def test_pair_pushers_equal_the_oracle(harness, tmp_path, kind, tol):
    cases = _cases()
    fin, fout = tmp_path / "in.bin", tmp_path / "out.bin"
    with open(fin, "wb") as f:
        f.write(struct.pack("<i", len(cases)))
        for eb, u in cases:
            f.write(struct.pack("<i", kind))
            f.write(np.concatenate([[-1.0, DT], eb, u]).astype("<f8").tobytes())
    subprocess.check_call([harness, str(fin), str(fout)])
    got = np.fromfile(fout, dtype="<f8").reshape(len(cases), 7)
    for (eb, u), g in zip(cases, got):
        assert g[6] == 1.0
        ref = {0: orc.boris, 2: orc.hc}[kind](-1.0, DT, eb, u) if kind in (0, 2) else orc.analytic(-1.0, DT, eb, u)[0]
        scale = max(np.abs(ref).max(), np.abs(u).max(), DT * np.abs(eb).max())
        assert np.abs(g[:3] - ref).max() <= tol * scale, (kind, eb, u, g[:3], ref)
        if kind < 3:
            gam = np.sqrt(1.0 + ref @ ref)
            assert np.abs(g[3:6] - DT * ref / gam).max() <= tol * DT * max(scale / gam, np.abs(ref / gam).max())
