// Tile sizes of the CTA-pair kernel (idf_kernels_pair.cu), chosen per launch, and the order in which its clusters take the work.  No CUDA
// headers: the parts that the kernel runs compile as plain host code too.
#pragma once
#include <cstddef>

#ifdef __CUDACC__
#define IDF_ANYWHERE __host__ __device__ __forceinline__
#else
#define IDF_ANYWHERE inline
#endif

namespace idf {

constexpr int PAIR_MAX_A = 8, PAIR_MAX_B = 24, PAIR_MAX_R = 8;     // stages of input rows and of tap rows, rows of a work item
constexpr int PAIR_TMEM = 512;                                     // columns of tensor memory
constexpr int PAIR_MMA_WARPS = 2;                                  // issuing warps: each issues for every other accumulator
constexpr int PAIR_CLUSTERS = 74;                                  // two SMs each
constexpr double PAIR_ROW_CLK = 800, PAIR_ITEM_CLK = 600;          // cycles from one input row to the next with little to do in it, and between items
constexpr size_t PAIR_SMEM = 230400;                               // dynamic shared memory per CTA (227 KB less the static part)

struct PairTiles {
    int ok;
    int BX, BXP, BS, n_xt, n_mt;     // an M tile: BS streams x BX positions of a row (BXP with the halo of the kx taps)
    int N, R, n_a, n_b;              // channels and rows of a work item, stages
    size_t a_box, a_bytes, b_tile;   // input row tile (bytes copied, bytes of a stage), half a weight tile (a stage: Kw of them)
    int row_step, n_u, clusters;
    long long units;
};

// rows: visited output rows, counted from the even one at or below the first where rows are pooled
inline PairTiles pair_tiles(int S, int Wout, int Cout, int Kh, int Kw, int swb, int n_kb, int rows, int pooled)
{
    PairTiles best{};
    if (rows < 1 || S < 1) return best;
    // positions: as few tiles of 128 lanes as possible
    PairTiles g{};
    for (int n_xt = (Wout + 127) / 128, last = n_xt + 4; n_xt <= last && n_xt <= Wout; ++n_xt) {
        int BX = (Wout + n_xt - 1) / n_xt;
        if (pooled) BX += BX & 1;                                   // the two positions of a pooled one are neighbouring lanes
        int BXP = BX + Kw - 1;
        if (pooled) BXP += BXP & 1;
        if (BX > 128 || BXP > 256) continue;
        int BS = 1 + (128 - BX) / BXP;
        if (BS > S) BS = S;
        const long long n_mt = (long long)((Wout + BX - 1) / BX) * ((S + BS - 1) / BS);
        if (n_mt > 0x3fffffff || (g.n_mt && n_mt >= g.n_mt)) continue;
        g.BX = BX; g.BXP = BXP; g.BS = BS; g.n_xt = (Wout + BX - 1) / BX; g.n_mt = (int)n_mt;
    }
    if (!g.n_mt) return best;
    g.a_box = (size_t)g.BXP * g.BS * swb;
    g.a_bytes = (g.a_box + 1023) / 1024 * 1024;
    g.row_step = pooled ? 2 : 1;
    g.n_u = (rows + g.row_step - 1) / g.row_step;
    double best_t = 0;
    for (int N = 256; N >= 32; N /= 2) {
        if (Cout % N) continue;
        for (int R = g.row_step; R <= PAIR_MAX_R && R * N <= PAIR_TMEM; R += g.row_step) {
            PairTiles t = g;
            t.N = N; t.R = R;
            t.b_tile = ((size_t)(N / 2) * swb + 1023) / 1024 * 1024;
            const int live = R < Kh ? R : Kh;                       // tap rows that one input row takes
            const size_t room = PAIR_SMEM - 1024, b_stage = t.b_tile * Kw;
            const int least = live + 1;
            if (least > PAIR_MAX_B || least * b_stage + 3 * t.a_bytes > room) continue;
            t.n_a = (int)((room - least * b_stage) / t.a_bytes);
            if (t.n_a > 6) t.n_a = 6;
            t.n_b = (int)((room - t.n_a * t.a_bytes) / b_stage);
            if (t.n_b > live + 6) t.n_b = live + 6;
            if (t.n_b > PAIR_MAX_B) t.n_b = PAIR_MAX_B;
            // (the last MMA rows of a tile run past its box into the next stage, the last stage's into the weights)
            if ((size_t)(128 + Kw) * swb > t.a_bytes + t.n_b * b_stage) continue;
            const long long cols = (long long)((t.n_mt + 1) / 2) * (Cout / N);
            t.units = cols * t.n_u;
            if (t.units > 0x3fffffff) continue;
            const int per = R / t.row_step;
            const long long items = cols * ((t.n_u + per - 1) / per);
            t.clusters = items < PAIR_CLUSTERS ? (int)items : PAIR_CLUSTERS;
            // Cycles of an item: input row by input row, MMAs (N / 2 a K step, or what its operands take out of shared memory) or the hand-over
            // between rows; its input must come out of the L2 meanwhile; and its accumulators be emitted.
            const int full = R < rows ? R : rows;
            const double sect = (double)Kw * (swb / 32) * (N / 2 > 32 + N / 8 ? N / 2 : 32 + N / 8);
            double mma = 0;
            for (int i = 0; i < full + Kh - 1; ++i) {
                const int hi = i < full - 1 ? i : full - 1, lo = i - Kh + 1 > 0 ? i - Kh + 1 : 0;
                const double clk = (hi - lo + 1) * sect;
                mma += n_kb * (clk > PAIR_ROW_CLK ? clk : PAIR_ROW_CLK);
            }
            const double bytes = (double)(full + Kh - 1) * n_kb * t.a_box + (double)Kh * Kw * n_kb * t.b_tile;
            const double emit = full * (400.0 + 6.0 * N);
            double item = mma > bytes / 40 ? mma : bytes / 40;
            if (emit > item) item = emit;
            item += PAIR_ITEM_CLK;
            const long long most = (t.units + t.clusters - 1) / t.clusters;              // units of the busiest cluster
            const double time = item * ((double)most * t.row_step / full) + 400.0 + 6.0 * N + bytes / 100;
            if (!best.ok || time < best_t) { best = t; best.ok = 1; best_t = time; }
        }
    }
    return best;
}

// The work items of a cluster: an even share of all units, cut into items of at most R rows of one column of work.  Args: PairArgs, or what
// a test has in its place.
struct PairWalk {
    int u, u_end;
    int col, row0, nr;           // column of work, first row, rows
    int j_lo, i_lo, i_hi;        // first accumulator in use; i in [i_lo, i_hi]: the input rows the block holds (input row row0 + i - base_ty)
    static IDF_ANYWHERE int least(int x, int y) { return x < y ? x : y; }
    static IDF_ANYWHERE int most(int x, int y) { return x > y ? x : y; }
    template <class Args>
    IDF_ANYWHERE bool start(const Args& a, unsigned c, unsigned n)      // cluster c of n
    {
        u = (int)((long long)a.units * c / n);
        u_end = (int)((long long)a.units * (c + 1) / n);
        return next(a);
    }
    template <class Args>
    IDF_ANYWHERE bool next(const Args& a)
    {
        if (u >= u_end) return false;
        col = u / a.n_u;
        const int r = u - col * a.n_u, rem = least(u_end - u, a.n_u - r), per = a.R / a.row_step;
        const int pieces = (rem + per - 1) / per, take = (rem + pieces - 1) / pieces;
        row0 = r * a.row_step;
        nr = least(take * a.row_step, a.row_hi - row0);
        u += take;
        j_lo = most(a.row_lo - row0, 0);
        i_lo = most(j_lo, a.base_ty - row0);
        i_hi = least(nr + a.Kh - 2, a.n_in - 1 + a.base_ty - row0);
        return true;
    }
    // input rows of accumulator j; none at all: the row has nothing to add
    IDF_ANYWHERE int first_row(int j) const { return most(i_lo, j); }
    template <class Args>
    IDF_ANYWHERE int last_row(const Args& a, int j) const { return least(i_hi, j + a.Kh - 1); }
    template <class Args>
    IDF_ANYWHERE bool has_taps(const Args& a, int j) const { return first_row(j) <= last_row(a, j); }
};

// A producer's last waits: every stage of its ring of n is free again, `stage` and its parity `ph` being those of the next use.  All n are looked
// at however many were used (a stage that never was passes at once: the phase before a barrier's first counts as over).
template <class Wait>
IDF_ANYWHERE bool pair_drain(int stage, unsigned ph, int n, Wait wait)
{
    for (int k = 0; k < n; ++k) {
        if (!wait(stage, ph)) return false;
        if (++stage == n) { stage = 0; ph ^= 1u; }
    }
    return true;
}

// What an issuing warp does that gives up: all it has issued is committed to a barrier of its own (of one arrival: a shared one would tell it of
// the other warp's instructions, and turn twice) and has a bounded time to finish.
template <class Commit, class Over>
IDF_ANYWHERE void pair_give_up(int issuer, Commit commit, Over over)
{
    commit(issuer);
    for (int i = 0; i < 4096 && !over(issuer); ++i) {}
}

// Whether a launch with the max-pool folded in both takes the x-pooled first row of a pair out of the pool layer's state (it begins with the
// pair's second row) and parks another one there (it ends with a first row).  The two pairs are different work items, mostly of different
// clusters, and nothing orders them: such a launch takes the row from a copy.
inline bool pair_pool_state_both(long long o_begin, long long done_end, int pool_keep)
{
    return pool_keep && (o_begin & 1) && (done_end & 1) && done_end > o_begin;
}

}  // namespace idf
