"""What the plan tuner times (fei_candidates.cuh, compiled for the host): the
grid that an untuned plan runs is among the candidates of every kernel, and
first among those of its variant, so that tuning cannot lose it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CC, TC, SF = 0, 1, 2


@pytest.fixture(scope="module")
def candidates(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("candidates") / "candidates")
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1310_1194_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "candidates_host.cu"), "-o", exe], check=True, capture_output=True)

    def run(kind, ntc=0, sf_too=0):
        out = subprocess.run([exe], input=f"{kind} {ntc} {sf_too}\n", capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in pair.split(":")) for pair in out.split()]

    return run


def test_default_grid_is_a_candidate(candidates):
    assert candidates(CC) == [(0, 0)] + [(0, 152 * k) for k in (2, 4, 8, 16)]
    assert candidates(SF) == [(0, 0), (0, 152)]
    assert candidates(TC, 3) == [(0, 0), (1, 0), (2, 0)]
    # FEI_AUTO at p >= 3: the sum-factorised kernel is variant ntc
    assert candidates(TC, 2, 1) == [(0, 0), (1, 0), (2, 0), (2, 152)]
