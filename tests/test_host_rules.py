"""Host-only checks of the rules by which the library cuts its work: compiled from the kernels' own header, run on the CPU."""
import os
import subprocess

from paper_2405_04304_b200 import build

_TILING = r"""
#include "umma_tail.cuh"
#include <cstdio>
using disco::VerifyTiling;
int main() {
    // head, rows: whether pairs of CTAs were measured to be the faster form
    struct { int V, d, R; bool pairs; } measured[] = {
        {32000, 2048, 251, true}, {32000, 5120, 650, true}, {32000, 1024, 2432, true}, {32000, 2048, 1520, false}, {49152, 1024, 428, false},
        {8000, 1024, 512, false}, {8000, 1024, 2432, false}, {32000, 5120, 300, false}, {4000, 5120, 1520, true}, {32000, 5120, 1520, false},
        {4000, 1024, 650, false}, {32000, 768, 650, false}, {32000, 5120, 128, false},
        // (sizes at which the GPU tests check pairs)
        {300, 1032, 129, true}, {300, 1032, 256, true}, {2500, 2056, 500, true}, {20000, 1032, 180, true}, {400, 2056, 1160, true},
        {700, 2056, 1409, true}, {9000, 1032, 1409, true}, {4000, 4104, 1409, true}};
    for (auto& m : measured)
        if (VerifyTiling::in_pairs(m.R, m.V, m.d, 148) != m.pairs) return std::printf("pairs: %d x %d, %d\\n", m.V, m.d, m.R), 1;
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
                    // pairs of CTAs: what the kernel derives from a count in device memory
                    const bool pairs = (R + 511) / 512 <= grid / 2;
                    if (VerifyTiling::pairs_possible(R, grid) != pairs) return std::printf("pairs_possible(%d, %d)\n", R, grid), 1;
                    if (!pairs) continue;
                    const VerifyTiling u = VerifyTiling::make_pairs(R, V, d, grid);
                    const bool u_rows = u.groups * u.GS * 256 >= R && 2 * u.groups * u.CN <= grid && u.CN >= 1 && (u.GS == 1 || u.GS == 2);
                    const bool u_cols = (long long)u.CN * u.TPC * u.TR >= V && u.TR >= 1 && u.TRN >= u.TR && u.TRN <= 256 && u.TRN % 16 == 0;
                    if (!u_rows || !u_cols) return std::printf("pairs: R %d V %d d %d grid %d\n", R, V, d, grid), 1;
                }
        }
    return 0;
}
"""


def _run(tmp_path, source):
    src, exe = tmp_path / "rules.cu", tmp_path / "rules"
    src.write_text(source)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include")
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", build.CSRC, "-I", include, "-o", str(exe),
                    str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, (run.returncode, run.stdout)


def test_verification_tiling_covers_everything_with_the_ctas_there_are(tmp_path):
    _run(tmp_path, _TILING)


_DRAFT = r"""
#include "draft_rules.cuh"
#include <cstdio>
using disco::DraftTiling;
int main() {
    // head, tiles of rows, logits kept, statistics only: whether pairs of CTAs were measured to be the faster form
    struct { int V, d, MT; bool kept, stats, pairs; } measured[] = {
        {32000, 2048, 5, false, false, false}, {49152, 4096, 7, false, false, false}, {32000, 5120, 5, true, false, true},
        {32000, 5120, 3, true, true, false}, {32000, 768, 8, true, false, false}, {17000, 1024, 8, true, true, false},
        {32000, 1536, 8, true, false, true}, {5000, 2048, 2, true, false, false}, {5000, 2048, 8, false, false, false},
        {32000, 2048, 2, false, false, true}, {32000, 2048, 4, false, false, true}, {17000, 2048, 4, true, true, true},
        // (sizes at which the GPU tests check pairs)
        {8000, 2048, 2, true, false, true}, {8003, 2048, 4, true, false, true}, {12300, 2048, 5, true, false, true},
        {300, 2048, 8, true, false, true}};
    for (auto& m : measured)
        if (disco::draft_in_pairs(m.V, m.d, m.MT, m.kept, m.stats, 148) != m.pairs) return std::printf("pairs: %d x %d, %d\\n", m.V, m.d, m.MT), 1;
    if (disco::draft_in_pairs(32000, 5120, 148, true, false, 147) || disco::draft_in_pairs(32000, 5120, 1, true, false, 148)) return 1;
    // steps to a launch: as many as there is scratch for, in even shares, and never more rows than have a shared bound
    for (int B : {1, 2, 3, 8, 12, 64, 100, 128, 130, 200, 256})
        for (int d : {64, 256, 768, 1024})
            for (int V : {1, 4000, 32000, 49152})
                for (int S = 1; S <= 40; ++S)
                    for (int most = 1; most <= 16; ++most) {
                        const int k = disco::draft_steps_per_launch(V, d, B, S, most, 148);
                        const int launches = (S + k - 1) / k;
                        if (k < 1 || k > most || k > S || (launches > 1 && (S + launches - 1) / launches != k) ||
                            (k > 1 && 148 / ((k * B + 127) / 128) < 10))
                            return std::printf("steps: %d x %d, B %d, %d, most %d: %d\\n", V, d, B, S, most, k), 1;
                    }
    // one sequence's ten steps fit a launch; narrow heads of many sequences, whose rows cost an epilogue each, do not gain by sixteen
    if (disco::draft_steps_per_launch(32000, 768, 1, 10, 10, 148) != 10 || disco::draft_steps_per_launch(32000, 256, 130, 16, 16, 148) > 8) return 1;
    const int grids[] = {1, 2, 16, 148}, ds[] = {8, 320, 328, 768, 5120}, rows[] = {1, 33, 40, 64, 100, 128, 129, 256, 257, 640, 1000};
    for (int sms : grids)
        for (int V = 1; V < 80000; V += V < 300 || (V > 34000 && V < 38200) ? 1 : 97)
            for (int R : rows) {
                if ((R + 127) / 128 > sms) continue;
                for (int d : ds)
                    for (int kind = 0; kind < 4; ++kind) {
                        const bool kept = kind & 1, pair = (kind & 2) && R > 128 && (((R + 127) / 128 + 1) & ~1) <= sms;
                        const DraftTiling t = DraftTiling::make(V, d, R, kept, pair, sms);
                        const bool covered = t.MT * 128 >= R && t.CN >= 1 && t.TPC >= 1 && t.TR >= 1 && (long long)t.CN * t.TPC * t.TR >= V;
                        const bool fits = t.MT * t.CN + t.finishers <= sms && t.TRN >= t.TR && t.TRN % 16 == 0 && t.TRN <= 256 &&
                                          (!pair || t.MT % 2 == 0) && (!kept || t.TR % 4 == 0) && (t.finishers == 0 || R <= 128);
                        // one tile of rows: one wide vocabulary tile and nobody to finish the rows is the worst of both
                        const bool lame = R <= 128 && t.TRN > 128 && t.TPC == 1 && t.finishers == 0 && d > 320;
                        if (!covered || !fits || (lame && sms > 16))
                            return std::printf("V %d d %d R %d kept %d pair %d sms %d\n", V, d, R, kept, pair, sms), 1;
                    }
            }
    return 0;
}
"""


def test_draft_tiling_covers_everything_with_the_ctas_there_are(tmp_path):
    _run(tmp_path, _DRAFT)
