"""Field states kept one after another for the laser-energy adjoint: the row passes load
and store 16 bytes at a time, so every component of every state starts on a 16-byte
boundary for odd cell counts too, and arrays that don't are refused.  CPU only (no
launch)."""
import os
import shutil
import subprocess

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
    exe = str(tmp_path_factory.mktemp("states") / "field_states_check_host")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O0", "-std=c++17",
                           "--expt-relaxed-constexpr", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                           "-o", exe, os.path.join(HERE, "native", "field_states_check_host.cu")])
    return exe


@pytest.mark.parametrize("cells", [1, 2, 31, 32, 33, 67 * 33, 301 * 45, 301 * 64])
def test_states_start_on_16_bytes(harness, cells):
    off, room, refused = (int(v) for v in subprocess.check_output([harness, str(cells)]).split())
    assert off == 0
    assert 0 <= room < 32
    assert refused == 1
