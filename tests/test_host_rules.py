"""Host-only checks of the rules by which the library cuts its work: compiled from the kernels' own header, run on the CPU."""
import os
import subprocess

from paper_2405_04304_b200 import build

_TILING = r"""
#include "umma_tail.cuh"
#include <cstdio>
using disco::VerifyTiling;
int main() {
    const int grids[] = {1, 2, 148}, vs[] = {1, 300, 32000, 151936}, ds[] = {8, 768, 2040, 2048, 6144};
    for (int grid : grids)
        for (int R = 1; R <= 128 * 2 * grid + 129; R += R < 1000 ? 1 : 127) {
            const bool want = R <= 128 * 2 * grid;
            if (VerifyTiling::possible(R, grid) != want) return std::printf("possible(%d, %d)\n", R, grid), 1;
            if (!want) continue;
            for (int V : vs)
                for (int d : ds) {
                    const VerifyTiling t = VerifyTiling::make(R, V, d, grid);
                    const bool rows = t.groups * t.GS * 128 >= R && t.groups * t.CN <= grid && t.CN >= 1 && (t.GS == 1 || t.GS == 2);
                    const bool cols = (long long)t.CN * t.TPC * t.TR >= V && t.TR >= 1 && t.TRN >= t.TR && t.TRN <= 256 && t.TRN % 16 == 0;
                    if (!rows || !cols) return std::printf("R %d V %d d %d grid %d\n", R, V, d, grid), 1;
                }
        }
    return 0;
}
"""


def test_verification_tiling_covers_everything_with_the_ctas_there_are(tmp_path):
    src, exe = tmp_path / "tiling.cu", tmp_path / "tiling"
    src.write_text(_TILING)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", build.CSRC, "-I", include, "-o", str(exe),
                    str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, (run.returncode, run.stdout)
