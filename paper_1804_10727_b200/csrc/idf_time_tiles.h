// Tile sizes of the 1D kernel (idf_kernels_time.cu), chosen per launch.  Plain host code: no CUDA headers.
#pragma once
#include <cstddef>

namespace idf {

constexpr int TIME_SB = 8, TIME_TM = 16;     // streams and output rows of an M tile
constexpr int TIME_MAX_W = 40;               // weight tiles in shared memory
constexpr size_t TIME_SMEM = 226304;         // dynamic shared memory per CTA (227 KB less the static part)

struct TimeTiles {
    int N, MT, cparts;           // outputs per channel slice, M tiles per work item, epilogue groups per M tile
    int n_w, resident, window;   // weight tiles in shared memory, 1: all of them, input rows of an item
    size_t a_bytes, w_bytes;     // of one K block of a window, of one weight tile
    int wide;                    // every run of 32 outputs that a thread stores starts on a 32-byte boundary of the row
};

// 128 outputs per MMA run at the pipe's full rate and four M tiles amortise a weight tile; where a launch has too few
// items for the SMs, channel slices are narrowed (the weights are what a lone CTA waits for).  Up to 64 rows are one item per
// stream group whatever its size: rows taken from the ring and rows parked in it then meet in one CTA.
inline TimeTiles time_tiles(int dtype, long long S, int n_rows, int Cout, int Kh, int stride, int swb, int n_kb)
{
    TimeTiles t{};
    int N = Cout;
    while (N > 128) N = N % 32 == 0 ? N / 2 : 16;
    if (Cout % N != 0 || N % 16 != 0) N = 16;
    const long long n_g = (S + TIME_SB - 1) / TIME_SB, big_items = n_g * ((n_rows + 63) / 64);
    while (N > 32 && N % 32 == 0 && big_items * (Cout / N) < 100) N /= 2;
    int MT = (n_rows + TIME_TM - 1) / TIME_TM;
    if (MT > 4) MT = 4;
    t.w_bytes = ((size_t)N * swb + 1023) / 1024 * 1024;
    auto window = [&](int mt) { return (mt * TIME_TM - 1) * stride + Kh; };
    auto a_bytes = [&](int mt) { return ((size_t)window(mt) * TIME_SB * swb + 1023) / 1024 * 1024; };
    while (MT > 1 && (window(MT) > 256 || 1024 + 2 * a_bytes(MT) + 3 * t.w_bytes > TIME_SMEM)) --MT;
    const int n_tiles = Kh * n_kb;
    int n_w = (int)((TIME_SMEM - 1024 - 2 * a_bytes(MT)) / t.w_bytes);
    if (n_w > TIME_MAX_W) n_w = TIME_MAX_W;
    t.resident = n_w >= n_tiles;
    t.n_w = t.resident ? n_tiles : (n_w > 8 ? 8 : n_w);
    t.N = N; t.MT = MT; t.window = window(MT); t.a_bytes = a_bytes(MT);
    t.cparts = MT == 1 ? 4 : (MT == 2 ? 2 : 1);
    while (t.cparts > 1 && (N % (16 * t.cparts)) != 0) t.cparts /= 2;
    // A thread's runs start at the multiples of 32 from the start of its group's share of the slice.  16 outputs of bf16 or fp32 are
    // 32 bytes whatever the slice; of int8 they are 16, and slices of 48 or 112 outputs (Cout 96, 224) start between.
    t.wide = dtype == 1 || (Cout % 32 == 0 && N % 32 == 0 && (N / t.cparts) % 32 == 0);
    return t;
}

}  // namespace idf
