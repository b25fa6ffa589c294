"""Which particle tiles are shared by several CTAs (csrc/common.cuh, share_line): none of
a uniform plasma whose tiles fill the SMs, every one where there are fewer tiles than
SMs, and a sheet's tile beside ordinary ones.  CPU only."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def line(tmp_path_factory):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc"
                                    if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("line") / "share_line_check_host")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O1", "-std=c++17",
                           "--expt-relaxed-constexpr", "-I",
                           os.path.join(ROOT, "paper_2004_03754_gb300", "csrc"), "-I",
                           os.path.join(ROOT, "include"), "-o", exe,
                           os.path.join(HERE, "native", "share_line_check_host.cu")])

    def call(particles, occupied):
        chunk = max(1024, -(-particles // 608))
        out = subprocess.run([exe], input=f"{particles} {occupied} {chunk}", capture_output=True, text=True)
        return int(out.stdout), chunk
    return call


@pytest.mark.parametrize("tiles, per_tile", [(230, 2048), (256, 2048), (384, 2048), (512, 2048), (512, 4096),
                                             (600, 1100), (740, 2048), (6000, 4096), (250, 1 << 16)])
def test_uniform_plasma_is_not_split(line, tiles, per_tile):
    got, chunk = line(tiles * per_tile, tiles)
    assert got >= per_tile and got >= chunk
    # a tile of twice the others is split unless it stays under a share's smallest size
    got, _ = line((tiles + 1) * per_tile, tiles)
    assert got < 2 * per_tile or got == max(1024, -(-(tiles + 1) * per_tile // 608))


@pytest.mark.parametrize("tiles, per_tile", [(1, 5000), (50, 8400), (64, 4096), (128, 4096), (150, 1 << 16)])
def test_few_tiles_are_split(line, tiles, per_tile):
    got, chunk = line(tiles * per_tile, tiles)
    assert chunk <= got < per_tile


def test_small_counts(line):
    assert line(0, 0)[0] == 1024
    assert line(1024, 1)[0] == 1024
    assert line(1500, 1)[0] == 1024
