// Eager (anytime) emission: the paper's literal rule, one segment at a time.
//
// Every unit keeps its state c (Eq. 2) and the activation it last announced.  After a segment has
// been applied, a unit whose activation f(c) differs from the announced one sends the difference
// dh = h(t) - h(t-1) to the layer above (Eq. 3), which adds w * dh to its own states (Eq. 4) and
// re-evaluates in turn (Eq. 5 and the sentence after it), layer by layer, within the same push.  So
// the net's output is available - and converges - while the input still arrives (Section
// "Experimental verification").  Units announce partial sums here, so a layer keeps every row that
// present or future input can still reach: the rows of the input cone, not just ceil(Kh/stride).
//
// Per layer three rings of `cap` rows (slot = row mod cap), 32-bit words (fp32 / int32):
//   c  the state variable,  h  the announced activation,  d  the change announced in this push.
// A push of one segment touches, in every layer, exactly the rows whose receptive field contains
// that segment; the host works the row intervals out and launches one kernel per layer.
//
// Two sets of kernels: plain ones (a thread per unit, any shape and type), and a tiled one for nets whose layers
// eager_tiled_words accepts and for which it is the faster (eager_tiled_pays), which keeps no h ring for conv layers and
// passes d on in the activation type.
#include "../../include/idf.h"
#include "idf_internal.h"

namespace idf {

namespace {

__device__ __forceinline__ float eager_act(float c, float b, int relu, int, int round_bf16)
{
    float v = c + b;
    if (relu && v < 0.f) v = 0.f;
    if (round_bf16) v = __bfloat162float(__float2bfloat16_rn(v));
    return v;
}
__device__ __forceinline__ int eager_act(int c, int b, int relu, int shift, int)
{
    int v = c + b;
    if (relu && v < 0) v = 0;
    if (shift > 0) v = (v + (1 << (shift - 1))) >> shift;
    const int lo = relu ? 0 : -127;
    return v < lo ? lo : (v > 127 ? 127 : v);
}
__device__ __forceinline__ float w_val(float w) { return w; }
__device__ __forceinline__ int w_val(int8_t w) { return (int)w; }

// one count per warp instead of one atomic per thread
__device__ __forceinline__ void count_events(unsigned long long* counter, bool nonzero)
{
    const unsigned m = __ballot_sync(__activemask(), nonzero);
    if (counter && m && (threadIdx.x & 31) == (__ffs(m) - 1)) atomicAdd(counter, (unsigned long long)__popc(m));
}

__device__ __forceinline__ void write_out(const EagerArgs& a, long long o, int s, int x, int co, float h)
{
    const long long i = (long long)s * a.out_stream_stride + o * a.out_row_stride + (long long)x * a.Cout + co;
    if (IDF_OK_AT(a.status, i, a.out_elems)) ((float*)a.out)[i] = h;
}
__device__ __forceinline__ void write_out(const EagerArgs& a, long long o, int s, int x, int co, int h)
{
    const long long i = (long long)s * a.out_stream_stride + o * a.out_row_stride + (long long)x * a.Cout + co;
    if (IDF_OK_AT(a.status, i, a.out_elems)) ((int8_t*)a.out)[i] = (int8_t)h;
}

// The pushed segment as the input layer's announcement: input units start at 0, so dh = x (paragraph after Eq. 3).
template <typename TI, typename TS>
__global__ void __launch_bounds__(256) eager_input_kernel(const TI* __restrict__ in, TS* __restrict__ d, long long n,
                                                          unsigned long long* events)
{
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < (n + 31) / 32 * 32;
         i += (long long)gridDim.x * blockDim.x) {
        TS v = 0;
        if (i < n) {
            if constexpr (sizeof(TI) == 2) v = (TS)__bfloat162float(in[i]);
            else v = (TS)in[i];
            d[i] = v;
        }
        count_events(events, v != (TS)0);
    }
}

// Conv layer: rows [o_lo, o_hi] take up the changes of rows [in_lo, in_hi] of the layer below (Eq. 4, zero
// changes skipped), re-evaluate, and announce their own change (Eq. 3).  One thread per unit.
template <typename TS, typename TW>
__global__ void __launch_bounds__(256) eager_conv_kernel(EagerArgs a)
{
    const TS* __restrict__ din = (const TS*)a.din;
    const TW* __restrict__ w = (const TW*)a.w;
    const TS* __restrict__ bias = (const TS*)a.bias;
    TS* cr = (TS*)a.c;
    TS* hr = (TS*)a.h;
    TS* dr = (TS*)a.d;
    const long long row_elems = (long long)a.Wout * a.Cout;
    const long long n = (a.o_hi - a.o_lo + 1) * a.S * row_elems;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < (n + 31) / 32 * 32;
         idx += (long long)gridDim.x * blockDim.x) {
        bool emitted = false;
        if (idx < n) {
            const int co = (int)(idx % a.Cout);
            long long t = idx / a.Cout;
            const int x = (int)(t % a.Wout);
            t /= a.Wout;
            const int s = (int)(t % a.S);
            const long long o = a.o_lo + t / a.S;
            TS acc = 0;
            if (a.in_lo <= a.in_hi)
                for (int ky = 0; ky < a.Kh; ++ky) {
                    const long long i = o * a.stride - a.pad + ky;
                    if (i < a.in_lo || i > a.in_hi) continue;
                    const TS* drow = din + ((i % a.cap_in) * a.S + s) * (long long)a.Win * a.Cin;
                    if (!IDF_OK_AT(a.status, (drow - din) + (long long)a.Win * a.Cin - 1, a.in_elems)) continue;
                    for (int kx = 0; kx < a.Kw; ++kx) {
                        const int ix = x * a.stride_x - a.pad_x + kx;
                        if (ix < 0 || ix >= a.Win) continue;
                        const TS* dp = drow + (long long)ix * a.Cin;
                        const TW* wp = w + ((long long)(ky * a.Kw + kx) * a.Cin) * a.Cout + co;
                        for (int ci = 0; ci < a.Cin; ++ci) {
                            const TS dv = dp[ci];
                            if (dv != (TS)0) acc += w_val(wp[(long long)ci * a.Cout]) * dv;     // only non-zero events cost work
                        }
                    }
                }
            const long long e = (((o % a.cap) * a.S + s) * a.Wout + x) * (long long)a.Cout + co;
            if (!IDF_OK_AT(a.status, e, a.ring_elems)) continue;
            const bool fresh = o >= a.o_new;                        // first touch: the slot still holds an older row
            const TS cn = (fresh ? (TS)0 : cr[e]) + acc;
            const TS hold = fresh ? (TS)0 : hr[e];
            const TS hn = o >= a.o_cut ? (TS)0 : eager_act(cn, bias ? bias[co] : (TS)0, a.relu, a.shift, a.round_bf16);
            cr[e] = cn;
            hr[e] = hn;
            dr[e] = hn - hold;
            emitted = hn != hold;
            if (a.out) write_out(a, o, s, x, co, hn);
        }
        count_events(a.events, emitted);
    }
}

// Max-pool unit: it holds its four current inputs (the announced activations of the layer below, 0 for units
// that have not announced anything yet) and announces max_new - max_old.
template <typename TS>
__global__ void __launch_bounds__(256) eager_pool_kernel(EagerArgs a)
{
    const TS* __restrict__ hin = (const TS*)a.hin;
    TS* hr = (TS*)a.h;
    TS* dr = (TS*)a.d;
    const int px = a.Win == 1 ? 1 : 2;
    const long long row_elems = (long long)a.Wout * a.Cout;
    const long long n = (a.o_hi - a.o_lo + 1) * a.S * row_elems;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < (n + 31) / 32 * 32;
         idx += (long long)gridDim.x * blockDim.x) {
        bool emitted = false;
        if (idx < n) {
            const int c = (int)(idx % a.Cout);
            long long t = idx / a.Cout;
            const int x = (int)(t % a.Wout);
            t /= a.Wout;
            const int s = (int)(t % a.S);
            const long long o = a.o_lo + t / a.S;
            TS m = 0;
            bool have = false;
            for (int dy = 0; dy < 2; ++dy) {
                const long long i = 2 * o + dy;
                for (int dx = 0; dx < px; ++dx) {
                    TS v = 0;                                          // a unit that has announced nothing stands at 0
                    const long long hi_at = (((i % a.cap_in) * a.S + s) * a.Win + (px * x + dx)) * (long long)a.Cin + c;
                    if (i <= a.in_hi && IDF_OK_AT(a.status, hi_at, a.in_elems)) v = hin[hi_at];
                    m = have ? (v > m ? v : m) : v;
                    have = true;
                }
            }
            const long long e = (((o % a.cap) * a.S + s) * a.Wout + x) * (long long)a.Cout + c;
            if (!IDF_OK_AT(a.status, e, a.ring_elems)) continue;
            const TS hold = o >= a.o_new ? (TS)0 : hr[e];
            const TS hn = o >= a.o_cut ? (TS)0 : m;
            hr[e] = hn;
            dr[e] = hn - hold;
            emitted = hn != hold;
            if (a.out) write_out(a, o, s, x, c, hn);
        }
        count_events(a.events, emitted);
    }
}

// ---- tiled kernel ---------------------------------------------------------------------------------------------------
// A block owns G streams and takes the segment through n consecutive layers (all of them where their weights fit shared memory
// together: no other block touches its streams, so a block-wide barrier is all there is between layers).  Per layer the changed
// rows below come into shared memory once, as [row][stream][channel group][x] words; a warp then takes an (output row, run of 32
// positions, NC channels) at a time, its lanes the positions: per tap and channel group one conflict-free load of the change, one
// broadcast load of NC weights, NC multiply-adds (dp4a on four channels for int nets).  A unit's old activation is f(c + b) of the
// state it reads anyway.  Bound by shared-memory and multiply-add instructions.  Measured, 512 streams of 28x28 int8 (conv 1->16->32,
// pool, 32->32), one row per push: 195 us per push with a thread per unit (global loads and a zero test per multiply-add, an atomic
// per warp for the event counts, a launch per layer), 64 us tiled with a launch per layer, 48 us in one launch,
// 39 us with the changes handed on in shared memory and int activations compared as bytes.  (Warp-level int8 matrix products instead of
// dp4a: slower, 51 us.)
constexpr int EAGER_THREADS = 512;
constexpr int EAGER_NC = 8;

template <int NC> __device__ __forceinline__ void ld_words(const void* p, uint32_t* v)
{
#pragma unroll
    for (int j = 0; j < NC / 4; ++j) {
        const uint4 q = ((const uint4*)p)[j];
        v[4 * j] = q.x; v[4 * j + 1] = q.y; v[4 * j + 2] = q.z; v[4 * j + 3] = q.w;
    }
}
template <int NC> __device__ __forceinline__ void st_words(void* p, const uint32_t* v)
{
#pragma unroll
    for (int j = 0; j < NC / 4; ++j) ((uint4*)p)[j] = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
}
template <int NC> __device__ __forceinline__ void st_values(void* base, long long at, const float* v)
{
    float* p = (float*)base + at;
    if (((uintptr_t)p & 15) == 0) st_words<NC>(p, (const uint32_t*)v);
    else {
#pragma unroll
        for (int j = 0; j < NC; ++j) p[j] = v[j];
    }
}
template <int NC> __device__ __forceinline__ void st_bytes(int8_t* p, const uint32_t* v)
{
    if (((uintptr_t)p & 3) == 0) {
#pragma unroll
        for (int j = 0; j < NC / 4; ++j) ((uint32_t*)p)[j] = v[j];
    } else {
#pragma unroll
        for (int j = 0; j < NC; ++j) p[j] = (int8_t)(v[j >> 2] >> (8 * (j & 3)));
    }
}
__device__ __forceinline__ float as_ts(float, uint32_t v) { return __uint_as_float(v); }
__device__ __forceinline__ int as_ts(int, uint32_t v) { return (int)v; }

// n / d by one multiplication (n below 2^16, d below 2^16: 0xffffffff / d + 1 is exact there)
struct FastDiv {
    uint32_t m;
    int d;
    __device__ __forceinline__ explicit FastDiv(int div) : m(0xffffffffu / (uint32_t)div + 1u), d(div) {}
    __device__ __forceinline__ int div(int n, int& rem) const
    {
        const int q = d == 1 ? n : (int)__umulhi((uint32_t)n, m);
        rem = n - q * d;
        return q;
    }
};
// A unit's NC changes (int nets: as words of four int8) on their way to the layer above: its d ring, or its changed rows in
// shared memory, word (row_g * groups + group) * W + x.
template <int NC>
__device__ __forceinline__ void pass_changes(int mode, uint32_t* dn, int row_g, int C, int co, int W, int x, void* dring, long long e, const float* d)
{
    if (mode == EO_WORDS) {
#pragma unroll
        for (int j = 0; j < NC; ++j) dn[(row_g * C + co + j) * W + x] = __float_as_uint(d[j]);
    } else if (mode == EO_RING) {
        st_values<NC>(dring, e, d);
    }
}
template <int NC>
__device__ __forceinline__ void pass_changes(int mode, uint32_t* dn, int row_g, int C, int co, int W, int x, void* dring, long long e, const uint32_t* d)
{
    if (mode == EO_QUADS) {
#pragma unroll
        for (int j = 0; j < NC / 4; ++j) dn[(row_g * (C >> 2) + (co >> 2) + j) * W + x] = d[j];
    } else if (mode == EO_WORDS) {
#pragma unroll
        for (int j = 0; j < NC; ++j) dn[(row_g * C + co + j) * W + x] = (uint32_t)(int)(int8_t)(d[j >> 2] >> (8 * (j & 3)));
    } else if (mode == EO_RING) {
        st_bytes<NC>((int8_t*)dring + e, d);
    }
}
// h = f(c + b) of NC int units as bytes, and the bytes of h_new - h_old (both in 0..127: with bit 7 set first, and put right after,
// no borrow crosses a byte)
template <int NC>
__device__ __forceinline__ void act_bytes(const uint32_t* c, const int* bias, int rnd, int shift, uint32_t* h)
{
#pragma unroll
    for (int q = 0; q < NC / 4; ++q) {
        int t[4];
        uint32_t hi2, neg;
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = ((int)c[4 * q + j] + (bias ? bias[4 * q + j] : 0) + rnd) >> shift;
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi2) : "r"(t[3]), "r"(t[2]));
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(h[q]) : "r"(t[1]), "r"(t[0]), "r"(hi2));
        asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(neg) : "r"(h[q]));              // ReLU: 0xff where a byte is negative
        h[q] &= ~neg;
    }
}
__device__ __forceinline__ uint32_t sub_bytes(uint32_t x, uint32_t y) { return ((x | 0x80808080u) - y) ^ 0x80808080u; }
__device__ __forceinline__ unsigned int count_bytes(uint32_t x) { return __popc((((x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | x) & 0x80808080u); }

// (What the loops need of the arguments is copied out first: they lie in parameter space behind a runtime layer index, where every
// use would be a load of its own.)
template <typename TS, int NC, bool QUADS>
__device__ __forceinline__ void eager_conv_units(const EagerArgs& a, const uint32_t* sw, const uint32_t* sd, int G, int s0, int Gn, int mode, uint32_t* dn, unsigned int& n_out)
{
    constexpr bool INT = (TS)0.5f == (TS)0;
    const int tid = threadIdx.x, lane = tid & 31;
    const int CQ = QUADS ? a.Cin >> 2 : a.Cin, Win = a.Win, Wout = a.Wout, Cout = a.Cout, Kw = a.Kw, stride = a.stride, stride_x = a.stride_x, pad_x = a.pad_x;
    const int relu = a.relu, shift = a.shift, round_bf16 = a.round_bf16, rnd = shift > 0 ? 1 << (shift - 1) : 0;
    const int n_pos = Gn * Wout, n_rows = (int)(a.o_hi - a.o_lo + 1);
    const FastDiv by_oct(Cout / NC), by_run((n_pos + 31) >> 5), by_w(Wout);
    const int n_units = n_rows * by_run.d * by_oct.d;
    const int tap0 = (int)(a.in_lo - (a.o_lo * stride - a.pad)), n_in = (int)(a.in_hi - a.in_lo + 1), Kh = a.Kh;    // row o_lo reaches changed row 0 through tap tap0
    const int slot0 = (int)(a.o_lo % a.cap), cap = a.cap;
    const int new_rel = (int)min(a.o_new - a.o_lo, (long long)n_rows), cut_rel = (int)min(a.o_cut - a.o_lo, (long long)n_rows);
    const long long row_elems = (long long)a.S * Wout * Cout;
    uint32_t* cring = (uint32_t*)a.c + (long long)s0 * Wout * Cout;
    void* dring = a.d;
    const TS* __restrict__ bias = (const TS*)a.bias;
    const bool last = a.out != nullptr;
    for (int u = tid >> 5; u < n_units; u += blockDim.x >> 5) {
        int oct, run, x;
        const int orel = by_run.div(by_oct.div(u, oct), run);
        const int pos = run * 32 + lane, co = oct * NC;
        const bool live = pos < n_pos;
        const int g = by_w.div(live ? pos : 0, x);
        int slot = slot0 + orel;                                                // (a cone has at most `cap` rows)
        if (slot >= cap) slot -= cap;
        const long long e = slot * row_elems + pos * Cout + co;                 // from the block's first stream
        const bool ok = live && IDF_OK_AT(a.status, e + (long long)s0 * Wout * Cout, a.ring_elems - (NC - 1));
        const bool fresh = orel >= new_rel;                                     // first touch: the slot still holds an older row
        uint32_t cw[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) cw[j] = 0u;
        if (ok && !fresh) ld_words<NC>(cring + e, cw);                          // (in flight during the sum)
        TS acc[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) acc[j] = 0;
        // changed rows below that this row reaches: taps first ... first + n_in - 1, as far as they are taps
        const int first = tap0 - orel * stride;
        const int ky0 = max(0, first), ky1 = min(Kh, first + n_in);
        const int ix0 = x * stride_x - pad_x;
        for (int ky = ky0; ky < ky1; ++ky) {
            const uint32_t* drow = sd + ((ky - first) * G + g) * CQ * Win;
            const uint32_t* wp = sw + ky * Kw * CQ * Cout + co;
            for (int kx = 0; kx < Kw; ++kx) {
                const bool in = (unsigned)(ix0 + kx) < (unsigned)Win;
                const uint32_t* dp = drow + (in ? ix0 + kx : 0);
#pragma unroll 4
                for (int c = 0; c < CQ; ++c, dp += Win, wp += Cout) {
                    uint32_t v = *dp;
                    if (!in) v = 0u;
                    uint32_t wv[NC];
                    ld_words<NC>(wp, wv);
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        if constexpr (QUADS) acc[j] = __dp4a((int)v, (int)wv[j], acc[j]);
                        else acc[j] += as_ts(TS(0), wv[j]) * as_ts(TS(0), v);
                    }
                }
            }
        }
        if (!ok) continue;
        const long long ring_at = e + (long long)s0 * Wout * Cout;
        const long long out_at = last ? (long long)(s0 + g) * a.out_stream_stride + (a.o_lo + orel) * a.out_row_stride + (long long)x * Cout + co : 0;
        const bool emit = last && IDF_OK_AT(a.status, out_at, a.out_elems - (NC - 1));
        if constexpr (INT) {
            const int* b = bias ? (const int*)bias + co : nullptr;
            uint32_t h_old[NC / 4], h_new[NC / 4], d[NC / 4];
            act_bytes<NC>(cw, b, rnd, shift, h_old);
#pragma unroll
            for (int j = 0; j < NC; ++j) cw[j] += (uint32_t)acc[j];
            act_bytes<NC>(cw, b, rnd, shift, h_new);
#pragma unroll
            for (int j = 0; j < NC / 4; ++j) {
                if (orel >= cut_rel) h_new[j] = 0u;
                d[j] = sub_bytes(h_new[j], fresh ? 0u : h_old[j]);
                n_out += count_bytes(d[j]);
            }
            st_words<NC>(cring + e, cw);
            pass_changes<NC>(mode, dn, orel * G + g, Cout, co, Wout, x, dring, ring_at, d);
            if (emit) st_bytes<NC>((int8_t*)a.out + out_at, h_new);
        } else {
            float d[NC], h[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                const float b = bias ? (float)bias[co + j] : 0.f, c_old = __uint_as_float(cw[j]), c_new = c_old + (float)acc[j];
                const float h_old = fresh ? 0.f : eager_act(c_old, b, relu, shift, round_bf16);
                h[j] = orel >= cut_rel ? 0.f : eager_act(c_new, b, relu, shift, round_bf16);
                d[j] = h[j] - h_old;
                n_out += d[j] != 0.f;
                cw[j] = __float_as_uint(c_new);
            }
            st_words<NC>(cring + e, cw);
            pass_changes<NC>(mode, dn, orel * G + g, Cout, co, Wout, x, dring, ring_at, d);
            if (emit) st_values<NC>(a.out, out_at, h);
        }
    }
}

template <typename TS, int NC>
__device__ __forceinline__ void eager_pool_units(const EagerArgs& a, int G, int s0, int Gn, int mode, uint32_t* dn, unsigned int& n_out)
{
    constexpr bool INT = (TS)0.5f == (TS)0;
    const int px = a.Win == 1 ? 1 : 2, Win = a.Win, C = a.Cout, Wout = a.Wout, S = a.S;
    const FastDiv by_oct(C / NC), by_w(Wout), by_g(Gn);
    const int n_rows = (int)(a.o_hi - a.o_lo + 1), n = n_rows * Gn * Wout * by_oct.d;
    const TS* __restrict__ bias = (const TS*)a.below_bias;
    const int of_conv = a.pool_of_conv, relu = a.below_relu, shift = a.below_shift, round_bf16 = a.below_round_bf16, rnd = shift > 0 ? 1 << (shift - 1) : 0;
    const int slot0 = (int)(a.o_lo % a.cap), cap = a.cap, slot_in0 = (int)((2 * a.o_lo) % a.cap_in), cap_in = a.cap_in;
    const int new_rel = (int)min(a.o_new - a.o_lo, (long long)n_rows), cut_rel = (int)min(a.o_cut - a.o_lo, (long long)n_rows);
    const int have_in = (int)min(a.in_hi + 1 - 2 * a.o_lo, 2LL * n_rows);        // rows below, from 2 * o_lo on, that have announced anything
    const uint32_t* hin = (const uint32_t*)a.hin;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        // (more than 2^16 items where rows are wide and channels many: by division there)
        int oct, x, sg;
        int t, t2, orel;
        if (n <= 65536) { t = by_oct.div(idx, oct); t2 = by_w.div(t, x); orel = by_g.div(t2, sg); }
        else { t = idx / by_oct.d; oct = idx - t * by_oct.d; t2 = t / Wout; x = t - t2 * Wout; orel = t2 / Gn; sg = t2 - orel * Gn; }
        const int co = oct * NC, s = s0 + sg;
        TS m[NC];
#pragma unroll
        for (int dy = 0; dy < 2; ++dy) {
            int slot = slot_in0 + 2 * orel + dy;
            while (slot >= cap_in) slot -= cap_in;
            for (int dx = 0; dx < px; ++dx) {
                const long long at = (((long long)slot * S + s) * Win + (px * x + dx)) * C + co;
                uint32_t w[NC];
#pragma unroll
                for (int j = 0; j < NC; ++j) w[j] = 0u;                         // a unit that has announced nothing stands at 0
                const bool have = 2 * orel + dy < have_in && IDF_OK_AT(a.status, at, a.in_elems - (NC - 1));
                if (have) ld_words<NC>(hin + at, w);
                // (int nets: f never falls when c rises, so the maximum is taken of the states and f applied to it once)
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    TS v = as_ts(TS(0), w[j]);
                    if (!INT && of_conv && have) v = eager_act(v, bias ? bias[co + j] : (TS)0, relu, shift, round_bf16);
                    if (INT && of_conv && !have) v = (TS)(-0x40000000);          // f of it is 0, whatever the bias
                    m[j] = dy + dx == 0 ? v : (v > m[j] ? v : m[j]);
                }
            }
        }
        int slot = slot0 + orel;
        if (slot >= cap) slot -= cap;
        const long long e = (((long long)slot * S + s) * Wout + x) * C + co;
        if (!IDF_OK_AT(a.status, e, a.ring_elems - (NC - 1))) continue;
        uint32_t hw[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) hw[j] = 0u;
        if (orel < new_rel) ld_words<NC>((const uint32_t*)a.h + e, hw);
        const long long out_at = a.out ? (long long)s * a.out_stream_stride + (a.o_lo + orel) * a.out_row_stride + (long long)x * C + co : 0;
        const bool emit = a.out && IDF_OK_AT(a.status, out_at, a.out_elems - (NC - 1));
        if constexpr (INT) {
            uint32_t h[NC / 4], h_old[NC / 4], d[NC / 4];
            act_bytes<NC>((const uint32_t*)m, of_conv && bias ? (const int*)bias + co : nullptr, of_conv ? rnd : 0, of_conv ? shift : 0, h);
            act_bytes<NC>(hw, nullptr, 0, 0, h_old);
            uint32_t hn[NC];
#pragma unroll
            for (int j = 0; j < NC / 4; ++j) {
                if (orel >= cut_rel) h[j] = 0u;
                d[j] = sub_bytes(h[j], h_old[j]);
                n_out += count_bytes(d[j]);
            }
#pragma unroll
            for (int j = 0; j < NC; ++j) hn[j] = (h[j >> 2] >> (8 * (j & 3))) & 0xffu;
            st_words<NC>((uint32_t*)a.h + e, hn);
            pass_changes<NC>(mode, dn, orel * G + sg, C, co, Wout, x, a.d, e, d);
            if (emit) st_bytes<NC>((int8_t*)a.out + out_at, h);
        } else {
            float d[NC], h[NC];
#pragma unroll
            for (int j = 0; j < NC; ++j) {
                h[j] = orel >= cut_rel ? 0.f : (float)m[j];
                d[j] = h[j] - __uint_as_float(hw[j]);
                n_out += d[j] != 0.f;
            }
            st_words<NC>((uint32_t*)a.h + e, (const uint32_t*)h);
            pass_changes<NC>(mode, dn, orel * G + sg, C, co, Wout, x, a.d, e, d);
            if (emit) st_values<NC>(a.out, out_at, h);
        }
    }
}

template <typename TS>
__global__ void __launch_bounds__(EAGER_THREADS, 2) eager_tiled_kernel(const __grid_constant__ EagerNetArgs net)
{
    constexpr bool INT = sizeof(TS) == sizeof(int) && (TS)0.5f == (TS)0;
    extern __shared__ __align__(16) uint32_t esm[];
    __shared__ unsigned int s_cnt[EAGER_MAX_LAYERS + 1];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31, G = net.G;
    if (tid <= EAGER_MAX_LAYERS) s_cnt[tid] = 0;
    // the weights do not depend on earlier kernels
    for (int l = 0; l < net.n; ++l) {
        const EagerArgs& a = net.layer[l];
        if (net.pool[l]) continue;
        const bool quads = INT && a.wq != nullptr;
        const int n_w = a.Kh * a.Kw * (quads ? a.Cin >> 2 : a.Cin) * a.Cout;
        uint32_t* sw = esm + net.w_at[l];
        const void* src = quads ? a.wq : a.w;
        for (int i = tid; i < n_w; i += blockDim.x) sw[i] = INT && !quads ? (uint32_t)(int)((const int8_t*)src)[i] : ((const uint32_t*)src)[i];
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int s0 = blockIdx.x * G, Gn = min(G, net.layer[0].S - s0);
    for (int l = 0; l < net.n; ++l) {
        const EagerArgs& a = net.layer[l];
        unsigned int n_in = 0, n_out = 0;
        const bool wide = a.Cout % EAGER_NC == 0;
        uint32_t *sd = esm + net.d_at[l & 1], *dn = esm + net.d_at[(l + 1) & 1];
        const int mode = net.d_ring ? EO_RING : (l + 1 == net.n || net.pool[l + 1] ? EO_NONE : (INT && net.layer[l + 1].wq ? EO_QUADS : EO_WORDS));
        __syncthreads();                                  // the layer below is done
        if (net.pool[l]) {
            if (wide) eager_pool_units<TS, EAGER_NC>(a, G, s0, Gn, mode, dn, n_out);
            else eager_pool_units<TS, 4>(a, G, s0, Gn, mode, dn, n_out);
        } else {
            const bool quads = INT && a.wq != nullptr;
            const int CQ = quads ? a.Cin >> 2 : a.Cin, row_elems = a.Win * a.Cin;
            const int rows = (int)(a.in_hi - a.in_lo + 1), Win = a.Win, elem = a.din_elem;      // changed rows below (may be none)
            const bool count = a.in_events != nullptr;
            const FastDiv by_c(CQ), by_w(Win);
            const int n = Gn * Win * CQ;
            // (within a launch the layer below has left its changes in place)
            for (int r = 0; r < (l == 0 ? rows : 0); ++r) {
                const long long first = (((a.in_lo + r) % a.cap_in) * a.S + s0) * (long long)row_elems;
                if (!IDF_OK_AT(a.status, first + (long long)Gn * row_elems - 1, a.in_elems)) continue;
                uint32_t* dst = sd + r * G * CQ * Win;
                const unsigned char* src = (const unsigned char*)a.din + first * (elem == E_I8 ? 1 : (elem == E_BF16 ? 2 : 4));
                const bool aligned = ((uintptr_t)src & 3) == 0;
                for (int i = tid; i < n; i += blockDim.x) {
                    int c, x;
                    const int g = by_w.div(by_c.div(i, c), x);
                    uint32_t v;
                    if (quads) {
                        const unsigned char* p = src + 4 * i;
                        v = aligned ? *(const uint32_t*)p : (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
                        if (count) n_in += __popc((((v & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v) & 0x80808080u);
                    } else {
                        if (elem == E_I8) v = (uint32_t)(int)((const int8_t*)src)[i];
                        else if (elem == E_BF16) v = __float_as_uint(__bfloat162float(((const __nv_bfloat16*)src)[i]));
                        else v = ((const uint32_t*)src)[i];
                        if (count) n_in += as_ts(TS(0), v) != TS(0);
                    }
                    dst[(g * CQ + c) * Win + x] = v;
                }
            }
            if (l == 0) __syncthreads();
            const uint32_t* sw = esm + net.w_at[l];
            if (quads) {
                if (wide) eager_conv_units<TS, EAGER_NC, INT>(a, sw, sd, G, s0, Gn, mode, dn, n_out);
                else eager_conv_units<TS, 4, INT>(a, sw, sd, G, s0, Gn, mode, dn, n_out);
            } else {
                if (wide) eager_conv_units<TS, EAGER_NC, false>(a, sw, sd, G, s0, Gn, mode, dn, n_out);
                else eager_conv_units<TS, 4, false>(a, sw, sd, G, s0, Gn, mode, dn, n_out);
            }
        }
        n_in = __reduce_add_sync(0xffffffffu, n_in);
        n_out = __reduce_add_sync(0xffffffffu, n_out);
        if (lane == 0 && a.in_events && n_in) atomicAdd(&s_cnt[EAGER_MAX_LAYERS], n_in);
        if (lane == 0 && a.events && n_out) atomicAdd(&s_cnt[l], n_out);
    }
    __syncthreads();
    if (tid < net.n && net.layer[tid].events && s_cnt[tid]) atomicAdd(net.layer[tid].events, (unsigned long long)s_cnt[tid]);
    if (tid == 0 && net.layer[0].in_events && s_cnt[EAGER_MAX_LAYERS]) atomicAdd(net.layer[0].in_events, (unsigned long long)s_cnt[EAGER_MAX_LAYERS]);
}

unsigned blocks_for(long long n)
{
    long long b = (n + 255) / 256;
    return (unsigned)(b < 1 ? 1 : (b > 148LL * 32 ? 148LL * 32 : b));
}

}  // namespace

cudaError_t launch_eager_input(const void* in, int in_elem, void* d, long long n, unsigned long long* events, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    switch (in_elem) {
        case E_F32: eager_input_kernel<float, float><<<blocks_for(n), 256, 0, st>>>((const float*)in, (float*)d, n, events); break;
        case E_BF16: eager_input_kernel<__nv_bfloat16, float><<<blocks_for(n), 256, 0, st>>>((const __nv_bfloat16*)in, (float*)d, n, events); break;
        case E_I8: eager_input_kernel<int8_t, int><<<blocks_for(n), 256, 0, st>>>((const int8_t*)in, (int*)d, n, events); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_eager_layer(const EagerArgs& a, int is_pool, int int_net, cudaStream_t st)
{
    if (a.o_hi < a.o_lo) return cudaSuccess;
    const long long n = (a.o_hi - a.o_lo + 1) * a.S * (long long)a.Wout * a.Cout;
    if (is_pool) {
        if (int_net) eager_pool_kernel<int><<<blocks_for(n), 256, 0, st>>>(a);
        else eager_pool_kernel<float><<<blocks_for(n), 256, 0, st>>>(a);
    } else {
        if (int_net) eager_conv_kernel<int, int8_t><<<blocks_for(n), 256, 0, st>>>(a);
        else eager_conv_kernel<float, float><<<blocks_for(n), 256, 0, st>>>(a);
    }
    return cudaGetLastError();
}

bool eager_tiled_words(int is_pool, int int_net, int Win, int Cin, int Cout, int Kh, int Kw, int rows_in, size_t* w, size_t* d)
{
    *w = *d = 0;
    if (Cout % 4 != 0) return false;
    if (is_pool) return true;
    const size_t cq = int_net && Cin % 4 == 0 ? Cin / 4 : Cin;
    *w = (size_t)Kh * Kw * cq * Cout;
    *d = (size_t)rows_in * cq * Win;
    return *w + 2 * *d <= EAGER_SMEM_WORDS;
}
// As few streams per block as still give every SM its two blocks (a narrow row fills a warp's lanes better with several streams).
int eager_tiled_group(int S, size_t w, size_t d, size_t limit_words)
{
    if (w + 2 * d > limit_words) return 0;               // (two sets of changed rows: a layer's and the next one's)
    int G = (S + 295) / 296;
    if (G > 8) G = 8;
    while (G > 1 && w + 2 * (size_t)G * d > limit_words) --G;
    return G;
}

cudaError_t launch_eager_tiled(const EagerNetArgs& a, int int_net, size_t smem_words, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = (debug_flags() & IDF_DEBUG_NO_PDL) ? 0 : 1;
    cfg.gridDim = dim3((unsigned)((a.layer[0].S + a.G - 1) / a.G));
    // a warp per unit of the layer that has most, at most sixteen
    int units = 4;
    for (int l = 0; l < a.n; ++l) {
        const EagerArgs& e = a.layer[l];
        const int nc = e.Cout % EAGER_NC == 0 ? EAGER_NC : 4, rows = (int)(e.o_hi - e.o_lo + 1);
        const int n = a.pool[l] ? (rows * a.G * e.Wout * (e.Cout / nc) + 31) / 32 : rows * ((a.G * e.Wout + 31) / 32) * (e.Cout / nc);
        units = units > n ? units : n;
    }
    cfg.blockDim = dim3((unsigned)(32 * (units > EAGER_THREADS / 32 ? EAGER_THREADS / 32 : units)));
    cfg.dynamicSmemBytes = smem_words * 4;
    typedef void (*Fn)(const EagerNetArgs);
    const Fn fn = int_net ? (Fn)eager_tiled_kernel<int> : (Fn)eager_tiled_kernel<float>;
    if (cfg.dynamicSmemBytes > 48 * 1024) {
        cudaError_t ce = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(EAGER_SMEM_WORDS * 4));
        if (ce != cudaSuccess) return ce;
    }
    cudaError_t ce = cudaLaunchKernelEx(&cfg, fn, a);
    return ce != cudaSuccess ? ce : cudaGetLastError();
}

}  // namespace idf
