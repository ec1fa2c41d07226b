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


POOL_PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include <vector>
#include "idf_pair_tiles.h"
using namespace idf;
struct Args { int units, n_u, R, row_step, row_lo, row_hi, Kh, base_ty, n_in; };
int main() {
    // launches of a 3x3 layer with padding and a pool: every output row belongs to one item; of pairs split over launches, the items that
    // take the first row out of the pool state and that park one there
    long long apart = 0, launches = 0;
    for (int S : {1, 3, 64})
        for (int Wout : {40, 56, 112, 131})
            for (int o_begin : {0, 1, 35})
                for (int rows : {1, 2, 3, 6, 7, 8, 35, 36, 37}) {
                    const int r0 = o_begin ? o_begin + 1 : 0, r1 = r0 + rows, done_end = r1 - 1, o_end = r1 + 1, o0 = o_begin & ~1;
                    if (done_end < o_begin) continue;
                    const PairTiles t = pair_tiles(S, Wout, 128, 3, 3, 128, 2, o_end - o0, 1);
                    if (!t.ok) { printf("no tiles\n"); return 1; }
                    const Args a{(int)t.units, t.n_u, t.R, 2, o_begin - o0, o_end - o0, 3, r0 + 1 - o0, r1 - r0};
                    const int cols = (int)(t.units / t.n_u), done = done_end - o0;
                    std::vector<int> seen(cols * a.row_hi, 0), taker(cols, -1), parker(cols, -1);
                    int item = 0;
                    for (int c = 0; c < t.clusters; ++c) {
                        PairWalk w;
                        for (bool more = w.start(a, c, t.clusters); more; more = w.next(a), ++item)
                            for (int j = w.j_lo; j < w.nr; ++j) {
                                const int row = w.row0 + j;
                                seen[w.col * a.row_hi + row]++;
                                if (row >= done) continue;
                                if ((row & 1) && row - 1 < a.row_lo) taker[w.col] = c;
                                if (!(row & 1) && row + 1 >= done) parker[w.col] = c;
                            }
                    }
                    ++launches;
                    const bool both = pair_pool_state_both(o_begin, done_end, 1);
                    for (int k = 0; k < cols; ++k) {
                        for (int row = a.row_lo; row < a.row_hi; ++row)
                            if (seen[k * a.row_hi + row] != 1) { printf("row %d of column %d: %d items\n", row, k, seen[k * a.row_hi + row]); return 1; }
                        if (both != (taker[k] >= 0 && parker[k] >= 0)) { printf("S %d W %d rows [%d, %d): taken by %d, parked by %d, rule %d\n", S, Wout, o_begin, done_end, taker[k], parker[k], both); return 1; }
                        apart += both && taker[k] != parker[k];
                    }
                }
    printf("%lld launches, %lld columns with the two in different clusters\n", launches, apart);
    return apart > 0 && !pair_pool_state_both(1, 7, 0) ? 0 : 1;
}
"""

DRAIN_PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "idf_pair_tiles.h"
using namespace idf;
int main() {
    // a ring of n stages after t uses, one of its stages (or none) not yet given back; a barrier is the number of its completed phases,
    // and a wait for a parity passes where the phase of that parity is the one before the current
    for (int n = 1; n <= PAIR_MAX_B; ++n)
        for (int t = 0; t <= 3 * n; ++t)
            for (int late = -1; late < n && late < t; ++late) {
                std::vector<unsigned> done(n, 0);
                int stage = 0;
                unsigned ph = 1;
                for (int k = 0; k < t; ++k) {
                    done[stage]++;
                    if (++stage == n) { stage = 0; ph ^= 1u; }
                }
                if (late >= 0) done[late]--;
                const bool over = pair_drain(stage, ph, n, [&](int s, unsigned parity) { return (done[s] & 1u) != parity; });
                if (over != (late < 0)) { printf("%d stages, %d uses, stage %d late: over %d\n", n, t, late, over); return 1; }
            }
    return 0;
}
"""

GIVE_UP_PROGRAM = r"""
#include <cstdio>
#include "idf_pair_tiles.h"
using namespace idf;
int main() {
    // barriers of one arrival; issuer k's instructions finish at its look number p, the other issuers' at look q
    for (int k = 0; k < PAIR_MMA_WARPS; ++k)
        for (int p = 0; p <= 6; ++p)
            for (int q = 0; q <= 6; ++q) {
                unsigned phases[PAIR_MMA_WARPS] = {};
                int looks = 0, mine = -1, theirs[PAIR_MMA_WARPS];
                for (int o = 0; o < PAIR_MMA_WARPS; ++o)                      // the barriers the others commit to
                    if (o != k) pair_give_up(o, [&](int b) { theirs[o] = b; }, [](int) { return true; });
                pair_give_up(k, [&](int b) { mine = b; }, [&](int b) {
                    if (looks == p) phases[mine]++;
                    for (int o = 0; o < PAIR_MMA_WARPS; ++o)
                        if (o != k && looks == q) phases[theirs[o]]++;
                    ++looks;
                    return (phases[b] & 1u) == 1u;
                });
                if (looks != p + 1) { printf("issuer %d done at %d, the other at %d: left at %d\n", k, p, q, looks - 1); return 1; }
            }
    return 0;
}
"""


def run(program, tmp_path):
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(program)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1804_10727_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_tiles_fit(tmp_path):
    run(PROGRAM, tmp_path)


def test_launches_that_take_and_park_a_pool_row_are_known(tmp_path):
    """Nothing orders the clusters: where one may read the pool state's words that another writes, the launch must read a copy."""
    run(POOL_PROGRAM, tmp_path)


def test_closing_waits_cover_every_stage_in_use(tmp_path):
    """No CTA leaves before the arrivals on its barriers are in, also where fewer stages were used than there are."""
    run(DRAIN_PROGRAM, tmp_path)


def test_issuers_that_give_up_wait_for_their_own_instructions(tmp_path):
    run(GIVE_UP_PROGRAM, tmp_path)
