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
// Two sets of kernels: plain ones (a thread per unit, any shape and type), and tiled ones for the shapes that
// eager_tiled_ok accepts, which keep no h ring for conv layers and pass d on in the activation type.
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
// per warp for the event counts, a launch per layer), 64 us tiled with a launch per layer, XX us in one launch.
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
template <int NC> __device__ __forceinline__ void st_values(void* base, long long at, int elem, const float* v)
{
    (void)elem;
    float* p = (float*)base + at;
    if (((uintptr_t)p & 15) == 0) st_words<NC>(p, (const uint32_t*)v);
    else {
#pragma unroll
        for (int j = 0; j < NC; ++j) p[j] = v[j];
    }
}
template <int NC> __device__ __forceinline__ void st_values(void* base, long long at, int elem, const int* v)
{
    if (elem != E_I8) { st_words<NC>((int*)base + at, (const uint32_t*)v); return; }
    int8_t* p = (int8_t*)base + at;
    if (((uintptr_t)p & 3) == 0) {
#pragma unroll
        for (int j = 0; j < NC / 4; ++j)
            ((uint32_t*)p)[j] = __byte_perm(__byte_perm(v[4 * j], v[4 * j + 1], 0x0040), __byte_perm(v[4 * j + 2], v[4 * j + 3], 0x0040), 0x5410);
    } else {
#pragma unroll
        for (int j = 0; j < NC; ++j) p[j] = (int8_t)v[j];
    }
}
__device__ __forceinline__ float as_ts(float, uint32_t v) { return __uint_as_float(v); }
__device__ __forceinline__ int as_ts(int, uint32_t v) { return (int)v; }

template <typename TS, int NC, bool QUADS>
__device__ __forceinline__ void eager_conv_units(const EagerArgs& a, const uint32_t* sw, const uint32_t* sd, int G, int s0, int Gn, unsigned int& n_out)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int CQ = QUADS ? a.Cin >> 2 : a.Cin;
    const int n_pw = (Gn * a.Wout + 31) >> 5, n_oct = a.Cout / NC;
    const int n_units = (int)(a.o_hi - a.o_lo + 1) * n_pw * n_oct;
    const TS* __restrict__ bias = (const TS*)a.bias;
    for (int u = tid >> 5; u < n_units; u += blockDim.x >> 5) {
        const int oct = u % n_oct, t = u / n_oct, pw = t % n_pw;
        const long long o = a.o_lo + t / n_pw;
        const int pos = pw * 32 + lane, co = oct * NC;
        const bool live = pos < Gn * a.Wout;
        const int g = live ? pos / a.Wout : 0, x = live ? pos - g * a.Wout : 0;
        TS acc[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) acc[j] = 0;
        // changed rows below that row o reaches: taps ky0 ... ky1
        const int first = (int)(a.in_lo - (o * a.stride - a.pad)), last = (int)(a.in_hi - (o * a.stride - a.pad));
        const int ky0 = max(0, first), ky1 = min(a.Kh - 1, last);
        for (int ky = ky0; ky <= ky1; ++ky) {
            const uint32_t* drow = sd + ((ky - first) * G + g) * CQ * a.Win;
            for (int kx = 0; kx < a.Kw; ++kx) {
                const int ix = x * a.stride_x - a.pad_x + kx;
                const bool in = (unsigned)ix < (unsigned)a.Win;
                const uint32_t* wp = sw + (ky * a.Kw + kx) * CQ * a.Cout + co;
                const uint32_t* dp = drow + (in ? ix : 0);
#pragma unroll 4
                for (int c = 0; c < CQ; ++c) {
                    uint32_t v = dp[c * a.Win];
                    if (!in) v = 0u;
                    uint32_t wv[NC];
                    ld_words<NC>(wp + c * a.Cout, wv);
#pragma unroll
                    for (int j = 0; j < NC; ++j) {
                        if constexpr (QUADS) acc[j] = __dp4a((int)v, (int)wv[j], acc[j]);
                        else acc[j] += as_ts(TS(0), wv[j]) * as_ts(TS(0), v);
                    }
                }
            }
        }
        const long long e = (((o % a.cap) * a.S + s0 + g) * a.Wout + x) * (long long)a.Cout + co;
        if (!live || !IDF_OK_AT(a.status, e, a.ring_elems - (NC - 1))) continue;
        const bool fresh = o >= a.o_new;                                        // first touch: the slot still holds an older row
        uint32_t cw[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) cw[j] = 0u;
        if (!fresh) ld_words<NC>((const uint32_t*)a.c + e, cw);
        TS d[NC], h[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            const TS b = bias ? bias[co + j] : (TS)0, c_old = as_ts(TS(0), cw[j]), c_new = c_old + acc[j];
            const TS h_old = fresh ? (TS)0 : eager_act(c_old, b, a.relu, a.shift, a.round_bf16);
            h[j] = o >= a.o_cut ? (TS)0 : eager_act(c_new, b, a.relu, a.shift, a.round_bf16);
            d[j] = h[j] - h_old;
            n_out += d[j] != (TS)0;
            cw[j] = *(const uint32_t*)&c_new;
        }
        st_words<NC>((uint32_t*)a.c + e, cw);
        st_values<NC>(a.d, e, a.d_elem, d);
        if (a.out) {
            const long long i = (long long)(s0 + g) * a.out_stream_stride + o * a.out_row_stride + (long long)x * a.Cout + co;
            if (IDF_OK_AT(a.status, i, a.out_elems - (NC - 1))) st_values<NC>(a.out, i, E_I8, h);
        }
    }
}

template <typename TS, int NC>
__device__ __forceinline__ void eager_pool_units(const EagerArgs& a, int s0, int Gn, unsigned int& n_out)
{
    const int px = a.Win == 1 ? 1 : 2, n_oct = a.Cout / NC;
    const int n = (int)(a.o_hi - a.o_lo + 1) * Gn * a.Wout * n_oct;
    const TS* __restrict__ bias = (const TS*)a.below_bias;
    for (int idx = threadIdx.x; idx < n; idx += blockDim.x) {
        const int co = (idx % n_oct) * NC, t = idx / n_oct, x = t % a.Wout, t2 = t / a.Wout, s = s0 + t2 % Gn;
        const long long o = a.o_lo + t2 / Gn;
        TS m[NC];
        for (int dy = 0; dy < 2; ++dy)
            for (int dx = 0; dx < px; ++dx) {
                const long long i = 2 * o + dy;
                const long long at = (((i % a.cap_in) * a.S + s) * a.Win + (px * x + dx)) * (long long)a.Cin + co;
                uint32_t w[NC];
#pragma unroll
                for (int j = 0; j < NC; ++j) w[j] = 0u;
                const bool have = i <= a.in_hi && IDF_OK_AT(a.status, at, a.in_elems - (NC - 1));
                if (have) ld_words<NC>((const uint32_t*)a.hin + at, w);
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    TS v = as_ts(TS(0), w[j]);                                  // a unit that has announced nothing stands at 0
                    if (have && a.pool_of_conv) v = eager_act(v, bias ? bias[co + j] : (TS)0, a.below_relu, a.below_shift, a.below_round_bf16);
                    m[j] = dy + dx == 0 ? v : (v > m[j] ? v : m[j]);
                }
            }
        const long long e = (((o % a.cap) * a.S + s) * a.Wout + x) * (long long)a.Cout + co;
        if (!IDF_OK_AT(a.status, e, a.ring_elems - (NC - 1))) continue;
        uint32_t hw[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) hw[j] = 0u;
        if (o < a.o_new) ld_words<NC>((const uint32_t*)a.h + e, hw);
        TS d[NC];
#pragma unroll
        for (int j = 0; j < NC; ++j) {
            if (o >= a.o_cut) m[j] = 0;
            d[j] = m[j] - as_ts(TS(0), hw[j]);
            n_out += d[j] != (TS)0;
        }
        st_words<NC>((uint32_t*)a.h + e, (const uint32_t*)m);
        st_values<NC>(a.d, e, a.d_elem, d);
        if (a.out) {
            const long long i = (long long)s * a.out_stream_stride + o * a.out_row_stride + (long long)x * a.Cout + co;
            if (IDF_OK_AT(a.status, i, a.out_elems - (NC - 1))) st_values<NC>(a.out, i, E_I8, m);
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
        for (int i = tid; i < n_w; i += blockDim.x)
            sw[i] = quads ? ((const uint32_t*)a.wq)[i] : (INT ? (uint32_t)(int)((const int8_t*)a.w)[i] : ((const uint32_t*)a.w)[i]);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int s0 = blockIdx.x * G, Gn = min(G, net.layer[0].S - s0);
    uint32_t* sd = esm + net.d_at;
    for (int l = 0; l < net.n; ++l) {
        const EagerArgs& a = net.layer[l];
        unsigned int n_in = 0, n_out = 0;
        const bool wide = a.Cout % EAGER_NC == 0;
        __syncthreads();                                  // the layer below is done (and its changed rows in shared memory are used up)
        if (net.pool[l]) {
            if (wide) eager_pool_units<TS, EAGER_NC>(a, s0, Gn, n_out);
            else eager_pool_units<TS, 4>(a, s0, Gn, n_out);
        } else {
            const bool quads = INT && a.wq != nullptr;
            const int CQ = quads ? a.Cin >> 2 : a.Cin, row_elems = a.Win * a.Cin;
            const int rows = (int)(a.in_hi - a.in_lo + 1);                      // changed rows below (may be none)
            for (int r = 0; r < rows; ++r) {
                const long long first = (((a.in_lo + r) % a.cap_in) * a.S + s0) * (long long)row_elems;
                if (!IDF_OK_AT(a.status, first + (long long)Gn * row_elems - 1, a.in_elems)) continue;
                uint32_t* dst = sd + r * G * CQ * a.Win;
                for (int i = tid; i < Gn * a.Win * CQ; i += blockDim.x) {
                    const int c = i % CQ, t = i / CQ, x = t % a.Win, g = t / a.Win;
                    uint32_t v;
                    if (quads) {
                        const unsigned char* p = (const unsigned char*)a.din + first + 4LL * i;
                        v = ((uintptr_t)p & 3) == 0 ? *(const uint32_t*)p : (uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16) | ((uint32_t)p[3] << 24);
                        if (a.in_events) n_in += __popc((((v & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v) & 0x80808080u);
                    } else {
                        if (a.din_elem == E_I8) v = (uint32_t)(int)((const int8_t*)a.din)[first + i];
                        else if (a.din_elem == E_BF16) v = __float_as_uint(__bfloat162float(((const __nv_bfloat16*)a.din)[first + i]));
                        else v = ((const uint32_t*)a.din)[first + i];
                        if (a.in_events) n_in += as_ts(TS(0), v) != TS(0);
                    }
                    dst[(g * CQ + c) * a.Win + x] = v;
                }
            }
            __syncthreads();
            const uint32_t* sw = esm + net.w_at[l];
            if (quads) {
                if (wide) eager_conv_units<TS, EAGER_NC, INT>(a, sw, sd, G, s0, Gn, n_out);
                else eager_conv_units<TS, 4, INT>(a, sw, sd, G, s0, Gn, n_out);
            } else {
                if (wide) eager_conv_units<TS, EAGER_NC, false>(a, sw, sd, G, s0, Gn, n_out);
                else eager_conv_units<TS, 4, false>(a, sw, sd, G, s0, Gn, n_out);
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
    return *w + *d <= EAGER_SMEM_WORDS;
}
// As few streams per block as still give every SM its two blocks (a narrow row fills a warp's lanes better with several streams).
int eager_tiled_group(int S, size_t w, size_t d, size_t limit_words)
{
    if (w + d > limit_words) return 0;
    int G = (S + 295) / 296;
    if (G > 8) G = 8;
    while (G > 1 && w + (size_t)G * d > limit_words) --G;
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
