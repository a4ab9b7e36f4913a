"""The built-in tile rule over the whole documented range (grids of 8 to 1024 points per axis, both kernel
precisions): its own choice is always a tile that the autotuner's candidates hold, that is one within the
kernels' thread bound and shared memory.  Host code only."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_2602_17950_gb300 import build
    build.build()
    exe = str(tmp_path_factory.mktemp("tiles") / "tile_rule_check")
    subprocess.run([build._nvcc(), *build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    os.path.join(HERE, "native", "tile_rule_check.cu"), build.LIB,
                    "-Xlinker", "-rpath=" + os.path.dirname(build.LIB), "-o", exe], check=True)
    return exe


# batches on both sides of the rule's thresholds (176, 304 and 1216 blocks), odd ones among them
BATCHES = ["1", "2", "3", "7", "8", "16", "40", "64", "255", "1000"]


@pytest.mark.parametrize("dim,most,batches", [(2, 20, BATCHES), (3, 24, BATCHES[:6]), (3, 30, ["1", "2"])])
def test_the_rule_picks_tiles_the_kernels_run(program, dim, most, batches):
    r = subprocess.run([program, str(dim), str(most), *batches], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout.split()[-4]) >= 1000
