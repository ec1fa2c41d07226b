"""Tile rule of the CTA-pair kernel (host code): tiles cover every position, pooled positions are neighbouring lanes, accumulators fit
tensor memory and stages fit shared memory, also where the last MMA rows of a tile run past its box."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "idf_pair_tiles.h"
using namespace idf;
int main() {
    long long n = 0;
    for (int pooled = 0; pooled <= 1; ++pooled)
        for (int S : {1, 2, 5, 64, 130, 1024, 4096})
            for (int Wout : {1, 2, 7, 14, 28, 39, 56, 57, 64, 112, 126, 127, 128, 129, 157, 224, 500})
                for (int Cout : {32, 64, 96, 128, 256, 512})
                    for (int Kh : {1, 2, 3, 5, 9})
                        for (int kx = 0; kx < 2; ++kx)
                            for (int swb : {64, 128})
                                for (int n_kb : {1, 2, 4})
                                    for (int rows : {1, 3, 7, 56, 2000}) {
                                        const int Kw = Wout == 1 || kx ? 1 : Kh;
                                        if (Wout == 1 && pooled) continue;
                                        const PairTiles t = pair_tiles(S, Wout, Cout, Kh, Kw, swb, n_kb, rows, pooled);
                                        if (!t.ok) continue;
                                        ++n;
                                        const int live = t.R < Kh ? t.R : Kh;
                                        const size_t b_stage = t.b_tile * Kw, used = 1024 + t.n_a * t.a_bytes + t.n_b * b_stage;
                                        bool ok = t.BX * t.n_xt >= Wout && t.BX * (t.n_xt - 1) < Wout && (t.BS - 1) * t.BXP + t.BX <= 128 && t.BXP >= t.BX + Kw - 1 &&
                                                  t.BXP <= 256 && t.BS <= 256 && t.n_mt == t.n_xt * ((S + t.BS - 1) / t.BS) &&
                                                  (!pooled || (t.BX % 2 == 0 && t.BXP % 2 == 0 && t.R % 2 == 0)) &&
                                                  Cout % t.N == 0 && t.N % 32 == 0 && t.N <= 256 && t.R >= 1 && t.R <= PAIR_MAX_R && t.R * t.N <= 512 &&
                                                  t.n_a >= 3 && t.n_a <= PAIR_MAX_A && t.n_b >= live + 1 && t.n_b <= PAIR_MAX_B && used <= PAIR_SMEM &&
                                                  t.a_box <= t.a_bytes && t.a_bytes % 1024 == 0 && t.b_tile % 1024 == 0 && t.b_tile >= (size_t)t.N / 2 * swb &&
                                                  (size_t)(128 + Kw) * swb <= t.a_bytes + t.n_b * b_stage &&
                                                  t.clusters >= 1 && t.clusters <= PAIR_CLUSTERS && t.units >= t.clusters &&
                                                  t.n_u * t.row_step >= rows && t.units == (long long)((t.n_mt + 1) / 2) * (Cout / t.N) * t.n_u;
                                        if (!ok) { printf("S %d W %d Cout %d Kh %d Kw %d swb %d kb %d rows %d pooled %d: BX %d BXP %d BS %d N %d R %d a %d b %d\n", S, Wout, Cout, Kh, Kw, swb, n_kb, rows, pooled, t.BX, t.BXP, t.BS, t.N, t.R, t.n_a, t.n_b); return 1; }
                                    }
    printf("%lld rules\n", n);
    return n > 10000 ? 0 : 1;
}
"""


def test_tiles_fit(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1804_10727_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
