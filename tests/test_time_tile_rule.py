"""Tile rule of the 1D kernel (host code): the 32-byte stores of its epilogue start on 32-byte boundaries for every channel count,
row count and stream count, and slices, shares and shared memory come out whole."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "idf_time_tiles.h"
using namespace idf;
int main() {
    long long n = 0, wide = 0;
    for (int dtype = 1; dtype <= 2; ++dtype)
        for (int Cout = 16; Cout <= 1024; Cout += 16)
            for (long long S : {1, 7, 48, 130, 300, 800, 4000})
                for (int n_rows : {1, 16, 17, 32, 33, 48, 49, 64, 65, 200, 4096})
                    for (int Kh : {1, 3, 9})
                        for (int stride = 1; stride <= 2 && stride <= Kh; ++stride)
                            for (int row : {32, 64, 128, 512}) {
                                const int swb = row < 128 ? row : 128;
                                const TimeTiles t = time_tiles(dtype, S, n_rows, Cout, Kh, stride, swb, row / swb);
                                ++n; wide += t.wide;
                                const int nc = t.N / t.cparts;
                                bool ok = t.N % 16 == 0 && Cout % t.N == 0 && nc % 16 == 0 && nc * t.cparts == t.N && t.MT >= 1 && t.MT * t.cparts <= 4 &&
                                          t.n_w >= 3 - 2 * t.resident && t.window <= 256 && 1024 + 2 * t.a_bytes + t.n_w * t.w_bytes <= TIME_SMEM;
                                for (int n0 = 0; n0 < Cout; n0 += t.N)
                                    for (int part = 0; part < t.cparts; ++part)
                                        for (int c = part * nc; c < (part + 1) * nc; c += 32) {
                                            const bool two = c + 16 < (part + 1) * nc;
                                            const long long at = (long long)Cout * 3 + n0 + c;      // a row's start is a multiple of Cout
                                            if (!t.wide) continue;
                                            if (dtype == 2) ok = ok && (!two || at % 32 == 0);       // int8: 32 outputs in one store
                                            else ok = ok && at * 2 % 32 == 0;                        // bf16, fp32: 16 or 8 outputs
                                        }
                                if (!ok) { printf("dtype %d Cout %d S %lld rows %d Kh %d stride %d row %d: N %d cparts %d wide %d\n", dtype, Cout, S, n_rows, Kh, stride, row, t.N, t.cparts, t.wide); return 1; }
                            }
    printf("%lld rules, %lld wide\n", n, wide);
    return 0;
}
"""


def test_every_wide_store_is_aligned(tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1804_10727_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
