"""The push of particles in FP32 fields (csrc/pair_push.cuh) outside the ordinary: momenta
and fields that are infinite, NaN or too large for FP32 arithmetic, against the FP64
push it stands for.  Where that moves the particle, this one moves it alike (2^-40);
where it gives no finite move or does not converge, neither does this one, so that the
caller latches the particle.  CPU only."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2004_03754_gb300", "csrc")
DT = 0.0981747704


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("range") / "push_range_check_host")
    subprocess.check_call([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-Wno-unknown-pragmas",
                           "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", exe,
                           os.path.join(HERE, "native", "push_range_check_host.cpp")])
    return exe


def _cases():
    rng = np.random.Generator(np.random.PCG64(31))
    eb0, u0 = np.array([0.1, 1.0, 0.2, 0.3, 0.1, 1.0]), np.array([0.4, -0.3, 1.0])
    out = []
    for v in (np.inf, -np.inf, np.nan, 1e39, -1e39, 1e20, 1e19, -1e15, 1e12, 5e9, 1e9, 1e7):
        for d in range(3):
            u = u0.copy()
            u[d] = v
            out.append((eb0, u))
        out.append((np.zeros(6), np.array([v, -0.3 * v, 1.0])))
    for v in (np.inf, -np.inf, np.nan, 3e38, 1e30, 1e20, 1e12, 1e10, 1e9, 1e7, 1e5):
        for c in range(6):
            eb = eb0.copy()
            eb[c] = v
            out.append((eb, u0))
    for e in range(8, 40):   # across the line between the two forms
        out.append((rng.uniform(-1, 1, 6), 2.0 ** e * rng.uniform(-1, 1, 3)))
        out.append((2.0 ** e * rng.uniform(-1, 1, 6), rng.uniform(-1, 1, 3)))
    with np.errstate(over="ignore"):
        return [(eb.astype(np.float32).astype(np.float64), u) for eb, u in out]


@pytest.mark.parametrize("kind", [0, 1, 2], ids=["boris", "analytic", "hc"])
@pytest.mark.parametrize("qm", [-1.0, 1e-3, -40.0])
def test_range_of_the_push(harness, tmp_path, kind, qm):
    cases = _cases()
    fin, fout = tmp_path / "in.bin", tmp_path / "out.bin"
    with open(fin, "wb") as f:
        f.write(struct.pack("<i", len(cases)))
        for eb, u in cases:
            f.write(struct.pack("<i", kind))
            f.write(np.concatenate([[qm, DT], eb, u]).astype("<f8").tobytes())
    subprocess.check_call([harness, str(fin), str(fout)])
    got = np.fromfile(fout, dtype="<f8").reshape(len(cases), 2, 8)
    moved = latched = 0
    for (eb, u), (g, r) in zip(cases, got):
        if r[7] == 1.0 and np.isfinite(r[:7]).all():
            moved += 1
            assert g[7] == 1.0 and np.isfinite(g).all(), (eb, u, g, r)
            scale = max(np.abs(r[:3]).max(), np.abs(u).max(), abs(qm) * DT * np.abs(eb).max())
            assert np.abs(g[:3] - r[:3]).max() <= 2.0 ** -40 * scale, (eb, u, g, r)
            gam = np.sqrt(1.0 + r[:3] @ r[:3])
            assert np.abs(g[3:6] - r[3:6]).max() <= 2.0 ** -40 * DT * max(scale / gam, 1.0), (eb, u, g, r)
        else:
            latched += 1
            assert g[7] == 0.0 or not np.isfinite(g[6]), (eb, u, g, r)
    assert moved > 60 and latched > 20
