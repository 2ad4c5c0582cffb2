"""kkt_residual keeps the partial maxima of its pass in the Krylov basis: four
doubles per block, and up to one block per slice of 32 rows. The basis must
hold them for every size and restart length that the options allow (compiled
here with g++)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_08656_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

SOURCE = """
#include "kernels.cuh"
#include <cstdio>
int main()
{
    for (int restart = 1; restart <= 3; ++restart)
        for (int n = 1; n <= 4096; ++n) {
            const int64_t slices = (n + 31) / 32, have = kktgb::krylov_doubles(n, restart);
            if (have < 4 * slices || have < (int64_t)n * (restart + 1)) {
                std::printf("n = %d, restart = %d: %lld doubles\\n", n, restart, (long long)have);
                return 1;
            }
        }
    return 0;
}
"""


def test_partial_maxima_fit_the_krylov_basis(tmp_path):
    if shutil.which("g++") is None or not os.path.isdir(CUDA_INC):
        pytest.skip("g++ or the CUDA headers not available")
    (tmp_path / "t.cpp").write_text(SOURCE)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", CSRC, "-I", CUDA_INC, str(tmp_path / "t.cpp"), "-o", exe],
                   check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
