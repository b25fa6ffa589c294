"""The push of particles in FP32 fields (csrc/pair_push.cuh) is no further from 64 bits
than the FP64 push with one Newton step per reciprocal: errors of both against long
double over electrons carried by pulses of a0 = 1 to 100 with plasma fields, at rest and
at gamma up to several hundred (root mean square and 99th percentile of u and of the
move, with 2 % for the sample).  CPU only."""
import math
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2004_03754_gb300", "csrc")
N = 1 << 15


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("long double is FP64 here")
    exe = str(tmp_path_factory.mktemp("err") / "push_error_check_host")
    subprocess.check_call([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-Wno-unknown-pragmas",
                           "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-o", exe,
                           os.path.join(HERE, "native", "push_error_check_host.cpp")])
    return exe


def _electrons(r):
    """dt, fields and momenta of N electrons after 0 to 120 steps in a pulse."""
    rng = np.random.Generator(np.random.PCG64(5))
    dt = r * 2 * math.pi / 32
    a0 = np.exp(rng.uniform(0, math.log(100), N))
    ph, L = rng.uniform(0, 2 * math.pi, N), 20 * math.pi
    noise = rng.normal(0, 1, (6, N)) * np.where(rng.random(N) < 0.5, 0.01, 0.1) * np.sqrt(a0)
    u = rng.normal(0, 1, (3, N)) * np.where(rng.random(N) < 0.7, 0.001, 0.0)
    last, x = rng.integers(0, 120, N), np.zeros(N)
    ahead = np.where(ph < 1, 5, 30)

    def fields(t):
        p = t - x + ahead
        F = noise * np.cos(0.3 * x + 0.1 * t)
        w = a0 * np.where((p > 0) & (p < L), np.sin(math.pi * p / L) ** 2, 0) * np.cos(p + ph)
        F[1] += w
        F[5] += w
        return F

    for k in range(120):
        F = fields(np.minimum(k, last) * dt)
        m = u - 0.5 * dt * F[:3]
        t = -0.5 * dt * F[3:] / np.sqrt(1 + (m * m).sum(0))
        un = m + np.cross(m + np.cross(m, t, axis=0), 2 * t / (1 + (t * t).sum(0)), axis=0) - 0.5 * dt * F[:3]
        go = k < last
        u = np.where(go, un, u)
        x = np.where(go, x + dt * u[0] / np.sqrt(1 + (u * u).sum(0)), x)
    return dt, fields(last * dt).astype(np.float32).astype(np.float64), u


def _run(harness, tmp_path, kind, dt, F, u):
    rec = np.empty(N, dtype=[("kind", "<i4"), ("v", "<f8", 11)])
    rec["kind"] = kind
    rec["v"] = np.concatenate([np.full((1, N), -1.0), np.full((1, N), dt), F, u]).T
    fin, fout = tmp_path / "in.bin", tmp_path / "out.bin"
    with open(fin, "wb") as f:
        f.write(struct.pack("<i", N))
        f.write(rec.tobytes())
    subprocess.check_call([harness, str(fin), str(fout)])
    return np.fromfile(fout, dtype="<f8").reshape(N, 4)


@pytest.mark.parametrize("r", [0.5, 0.25])
@pytest.mark.parametrize("kind", [0, 1, 2], ids=["boris", "analytic", "hc"])
def test_error_is_no_larger(harness, tmp_path, kind, r):
    dt, F, u = _electrons(r)
    e = _run(harness, tmp_path, kind, dt, F, u)
    for mine, fp64 in ((e[:, 0], e[:, 1]), (e[:, 2], e[:, 3])):
        assert np.sqrt(np.mean(mine ** 2)) <= 1.02 * np.sqrt(np.mean(fp64 ** 2))
        assert np.quantile(mine, 0.99) <= 1.02 * np.quantile(fp64, 0.99)
        assert np.median(mine) <= 1.02 * np.median(fp64)


@pytest.mark.parametrize("cold", [True, False])
@pytest.mark.parametrize("kind", [0, 1, 2], ids=["boris", "analytic", "hc"])
def test_error_in_the_pairs_range(harness, tmp_path, kind, cold):
    # across the lines past which the FP64 push takes over: |s|^2 (E^2 + B^2) to 2^-6, weak
    # and strong shares of E and B, electrons at rest (|u| error against their new u, so
    # the fields' share is as large as it gets) and hot ones
    rng = np.random.Generator(np.random.PCG64(6))
    dt = 2 * math.pi / 64
    u = np.zeros((3, N)) if cold else rng.normal(0, 1, (3, N)) * 10.0 ** rng.uniform(-3, 3, N)
    gam = np.sqrt(1 + (u * u).sum(0))
    F = rng.normal(0, 1, (6, N))
    F[:3] *= 10.0 ** rng.uniform(-4, 0, N)
    F *= gam / dt * 2.0 ** rng.uniform(-8, -3, N) / np.sqrt((F * F).sum(0))
    e = _run(harness, tmp_path, kind, dt, F.astype(np.float32).astype(np.float64), u)
    for q in (0.5, 0.99, 0.999):
        # (a rest of rounding of the pairs, 2^-48 of a change of u of up to a tenth)
        assert np.quantile(e[:, 0], q) <= max(1.02 * np.quantile(e[:, 1], q), 2.0 ** -48 / 10 * 5), q
        assert np.quantile(e[:, 2], q) <= 1.02 * np.quantile(e[:, 3], q), q
