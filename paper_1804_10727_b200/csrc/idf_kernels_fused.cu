// Depth-first over ALL layers in one launch, with every layer's rolling state on chip.
//
// The paper pushes each arriving segment through the whole net before the next one is looked at, and
// keeps only the partial activations that present or future input can still influence (Section
// "Asynchronous incremental updates", first paragraph; Discussion: "activation subset buffers").  For
// nets whose per-stream state is small this kernel does exactly that on one SM: a CTA owns a group of
// streams, loads their rings (and pooling rows) into shared memory, and then takes the pushed
// segments one at a time: the segment's events update the first layer's ring rows (Eq. 4), a row
// that is complete is finalised (Eq. 2-3) into a shared-memory row buffer, which is the next layer's
// input at once, and so on up to the output row, which is the only thing written to global memory
// besides the state at the end of the launch.  Between layers nothing leaves the SM.
//
// State in global memory has the layout of the per-layer kernels (rings [slot][stream][x][c] of
// 32-bit words without the bias, pooling rows [stream][x][c] in the layer's element type), so a
// stream may be advanced by this kernel and by the per-layer kernels in turn.
//
// Rows travel between layers in shared memory as fp32 values (float nets; bf16 layers hold
// bf16-representable values) or int8 (int nets, four channels to a word for dp4a).  Row bookkeeping
// (which ring slots a row reaches, which row it completes) is kept in small counters that step from
// row to row: no division in the loop over segments.
#include "idf_internal.h"

namespace idf {

namespace {

template <typename TS> struct RowOf;
template <> struct RowOf<float> { typedef float T; typedef float W; };
template <> struct RowOf<int> { typedef int8_t T; typedef int8_t W; };

__device__ __forceinline__ float fused_act(float c, float b, int relu, int, int round_bf16)
{
    float v = c + b;
    if (relu && v < 0.f) v = 0.f;
    if (round_bf16) v = __bfloat162float(__float2bfloat16_rn(v));
    return v;
}
__device__ __forceinline__ int8_t fused_act(int c, int b, int relu, int shift, int)
{
    int v = c + b;
    if (relu && v < 0) v = 0;
    if (shift > 0) v = (v + (1 << (shift - 1))) >> shift;
    const int lo = relu ? 0 : -127;
    return (int8_t)(v < lo ? lo : (v > 127 ? 127 : v));
}

template <typename TR>
__device__ __forceinline__ TR load_elem(const void* p, long long i, int elem)
{
    if (elem == E_F32) return (TR)((const float*)p)[i];
    if (elem == E_BF16) return (TR)__bfloat162float(((const __nv_bfloat16*)p)[i]);
    return (TR)((const int8_t*)p)[i];
}
template <typename TR>
__device__ __forceinline__ void store_elem(void* p, long long i, int elem, TR v)
{
    if (elem == E_F32) ((float*)p)[i] = (float)v;
    else if (elem == E_BF16) ((__nv_bfloat16*)p)[i] = __float2bfloat16_rn((float)v);
    else ((int8_t*)p)[i] = (int8_t)v;
}

template <int B>
__device__ __forceinline__ void copy_async(void* dst, const void* src)
{
    if (B == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// progress of one layer inside the launch (the same in every thread)
struct LayerClock {
    int ph;        // conv: (rows received + pad) mod stride = the first tap ky of the next input row; pool: rows received mod 2
    int hi_slot;   // conv: ring slot of the newest row the next input row reaches
    int hi_sat;    // conv: index of that newest row, saturated (only "how many older rows exist" matters)
    int phf;       // conv: (rows received + pad - (Kh-1)) mod stride: 0 when the next input row completes a row
    int tf_neg;    // conv: input rows still to come before the first row can complete
    int done_slot; // conv: ring slot of the oldest open row (the next to complete)
};

constexpr int FUSED_TAPS = 3;      // rows one input row reaches in the fast loops (ceil(Kh/stride) <= 3); more take the plain loop

// n / d and the remainder by one multiplication (m = 0xffffffff / d + 1, from the host; n below 2^16)
__device__ __forceinline__ int div_by(int n, int d, unsigned int m, int& rem)
{
    const int q = d == 1 ? n : (int)__umulhi((unsigned int)n, m);
    rem = n - q * d;
    return q;
}

// Layer i takes the row `in` ([G][Win][Cin]) as its next input row.  Returns true if it completed a row, which then
// stands in the layer's row buffer.  (A push of one segment is one chain of dependent steps through all layers, so what counts is
// the latency of a step: the layer's numbers are fetched together at its start - they lie in parameter space behind a runtime index,
// where each use would be a load of its own in the chain - nothing is divided, and no load hides behind a branch.)
template <typename TS>
__device__ __forceinline__ bool fused_feed(const FusedArgs& a, int i, const typename RowOf<TS>::T* in, unsigned char* smem, LayerClock& k, int G,
                           unsigned long long* ev_local)
{
    typedef typename RowOf<TS>::T TR;
    typedef typename RowOf<TS>::W TW;
    const FusedLayer& L = a.layer[i];
    const int kind = L.kind, count = L.count_events, Win = L.Win, Wout = L.Wout, Cin = L.Cin, Cout = L.Cout, Kh = L.Kh, Kw = L.Kw, stride = L.stride;
    const int stride_x = L.stride_x, pad_x = L.pad_x, relu = L.relu, shift = L.shift, round_bf16 = L.round_bf16, ring_rows = L.ring_rows;
    const unsigned int m_cout = L.m_cout, m_wout = L.m_wout;
    const long long bias_off = L.bias_off, wq_off = L.wq_off, w_off = L.w_off;
    const int b_soff = L.b_soff, w_soff = L.w_soff;
    TR* rowbuf = (TR*)(smem + L.rowbuf_soff);
    TS* ring = (TS*)(smem + L.state_soff);
    LayerClock c = k;
    if (count) {
        // the layer's input events: the non-zero components of the row (Eq. 3)
        unsigned n = 0;
        for (int e = threadIdx.x; e < G * Win * Cin; e += blockDim.x) n += in[e] != (TR)0;
        n = __reduce_add_sync(0xffffffffu, n);
        if ((threadIdx.x & 31) == 0 && n) atomicAdd(&ev_local[i], (unsigned long long)n);
    }
    const int row_elems = Wout * Cout, n_elems = G * row_elems;
    const bool small = n_elems <= 65535;
    auto split = [&](int e, int& co, int& x) {                   // element -> (stream, x, channel)
        if (small) { const int t = div_by(e, Cout, m_cout, co); return div_by(t, Wout, m_wout, x); }
        const int t = e / Cout;
        co = e - t * Cout;
        const int g = t / Wout;
        x = t - g * Wout;
        return g;
    };
    if (kind == 1) {
        // 2x2 max-pool fold: the x-pooled first row of a pair waits in the pool state
        TR* st = (TR*)ring;
        const int px = Win == 1 ? 1 : 2;
        const bool second = c.ph != 0;
        for (int e = threadIdx.x; e < n_elems; e += blockDim.x) {
            int co, x;
            const int g = split(e, co, x);
            const TR* p = in + ((g * Win + px * x) * Cin + co);
            TR m = p[0];
            if (px == 2) { const TR v = p[Cin]; m = v > m ? v : m; }
            if (second) { const TR f = st[e]; rowbuf[e] = f > m ? f : m; }
            else st[e] = m;
        }
        __syncthreads();
        k.ph = c.ph ^ 1;
        return second;
    }
    // conv: Eq. 4 for every event of the row, tap by tap, then Eq. 2-3 for the row this input row completes
    const TS* bias = bias_off < 0 ? nullptr : b_soff >= 0 ? (const TS*)(smem + b_soff) : (const TS*)((const unsigned char*)a.weights + bias_off);
    // taps ky = ph, ph + s, ... < Kh; tap j reaches the row j below the newest one (if that many rows exist)
    int nt = 0;
    for (int ky = c.ph; ky < Kh; ky += stride) ++nt;
    if (nt > c.hi_sat + 1) nt = c.hi_sat + 1;
    const bool completes = c.phf == 0 && c.tf_neg == 0;      // ... and the oldest row reached then has its last tap
    // The newest row begins with its tap 0, in a slot that may hold what an earlier row left (the per-layer kernels do not clear the
    // slots they empty): it starts from 0.  (Rows begun by input row 0 with a later tap find slots as the reset left them.)
    const bool begins = c.ph == 0;
    const int Cq = Cin >> 2;
    const bool quads = (Cin & 3) == 0 && !count && wq_off >= 0;
    if (nt <= FUSED_TAPS && (quads || Cin <= 4)) {
        // Four input channels at a time (dp4a / four FMAs), or one by one for up to four; the input fetched once for all taps.  Taps
        // beyond nt repeat the last one's loads and are dropped at the end: a branch per tap would put every load's latency in the chain.
        const int tap_q = stride * Kw * Cq * Cout, tap_w = stride * Kw * Cin * Cout;      // from tap j to tap j + 1
        int at_q[FUSED_TAPS], at_w[FUSED_TAPS];
#pragma unroll
        for (int j = 0; j < FUSED_TAPS; ++j) {
            const int jj = j < nt ? j : nt - 1;
            at_q[j] = jj * tap_q;
            at_w[j] = jj * tap_w;
        }
        // (inlined once for weights in shared memory and once for weights in global memory)
        auto run = [&](const int* wq, const TW* w, const TS* bias) {
            for (int e = threadIdx.x; e < n_elems; e += blockDim.x) {
                int co, x;
                const int g = split(e, co, x);
                // the ring words these taps reach, in flight during the sum
                int at[FUSED_TAPS];
                TS old[FUSED_TAPS], acc[FUSED_TAPS];
#pragma unroll
                for (int j = 0; j < FUSED_TAPS; ++j) {
                    int slot = c.hi_slot - (j < nt ? j : nt - 1);
                    if (slot < 0) slot += ring_rows;
                    at[j] = (slot * G + g) * row_elems + x * Cout + co;
                    old[j] = ring[at[j]];
                    if (j == 0 && begins) old[j] = 0;
                    acc[j] = 0;
                }
                const TS b = bias ? bias[co] : (TS)0;
                for (int kx = 0; kx < Kw; ++kx) {
                    const int ix = x * stride_x - pad_x + kx;
                    if ((unsigned)ix >= (unsigned)Win) continue;
                    const TR* ip = in + (g * Win + ix) * Cin;
                    if (!quads) {
                        const TW* wp = w + (c.ph * Kw + kx) * Cin * Cout + co;
                        for (int ci = 0; ci < Cin; ++ci, wp += Cout) {
                            const TS v = (TS)ip[ci];
#pragma unroll
                            for (int j = 0; j < FUSED_TAPS; ++j) acc[j] += (TS)wp[at_w[j]] * v;
                        }
                        continue;
                    }
#pragma unroll 2
                    for (int c4 = 0; c4 < Cq; ++c4) {
                        if constexpr (sizeof(TR) == 1) {
                            const int v = ((const int*)ip)[c4];
                            const int* wp = wq + ((c.ph * Kw + kx) * Cq + c4) * Cout + co;
#pragma unroll
                            for (int j = 0; j < FUSED_TAPS; ++j) acc[j] = __dp4a(v, wp[at_q[j]], acc[j]);
                        } else {
                            const float4 v = ((const float4*)ip)[c4];
                            const TW* wp = w + ((c.ph * Kw + kx) * Cin + 4 * c4) * Cout + co;
#pragma unroll
                            for (int j = 0; j < FUSED_TAPS; ++j) {
                                const TW* wj = wp + at_w[j];
                                acc[j] += wj[0] * v.x; acc[j] += wj[Cout] * v.y;
                                acc[j] += wj[2 * Cout] * v.z; acc[j] += wj[3 * Cout] * v.w;
                            }
                        }
                    }
                }
                TS done = 0;
#pragma unroll
                for (int j = 0; j < FUSED_TAPS; ++j) {
                    const TS s = old[j] + acc[j];
                    const bool frees = completes && j == nt - 1;               // (left zero: the event scatter starts its rows from the ring)
                    if (j < nt) ring[at[j]] = frees ? (TS)0 : s;
                    if (j == nt - 1) done = s;
                }
                if (completes) rowbuf[e] = fused_act(done, b, relu, shift, round_bf16);
            }
        };
        const TS* gbias = bias_off < 0 ? nullptr : (const TS*)((const unsigned char*)a.weights + bias_off);
        if (w_soff >= 0) run((const int*)(smem + w_soff), (const TW*)(smem + w_soff), b_soff >= 0 ? (const TS*)(smem + b_soff) : gbias);
        else run((const int*)((const unsigned char*)a.weights + wq_off), (const TW*)a.weights + w_off, gbias);
    } else {
        const TW* w = w_soff >= 0 ? (const TW*)(smem + w_soff) : (const TW*)a.weights + w_off;
        for (int e = threadIdx.x; e < n_elems; e += blockDim.x) {
            int co, x;
            const int g = split(e, co, x);
            int slot = c.hi_slot;
            for (int j = 0; j < nt; ++j) {
                const int ky = c.ph + j * stride;
                TS acc = 0;
                for (int kx = 0; kx < Kw; ++kx) {
                    const int ix = x * stride_x - pad_x + kx;
                    if (ix < 0 || ix >= Win) continue;
                    const TR* ip = in + (g * Win + ix) * Cin;
                    const TW* wp = w + ((ky * Kw + kx) * Cin) * Cout + co;
                    for (int ci = 0; ci < Cin; ++ci) {
                        const TS v = (TS)ip[ci];
                        if (v != (TS)0) acc += (TS)wp[ci * Cout] * v;         // zero components send no event
                    }
                }
                TS* cp = ring + (slot * G + g) * row_elems + x * Cout + co;
                if (--slot < 0) slot += ring_rows;
                const TS s = (j == 0 && begins ? (TS)0 : *cp) + acc;
                if (completes && j == nt - 1) {
                    rowbuf[e] = fused_act(s, bias ? bias[co] : (TS)0, relu, shift, round_bf16);
                    *cp = 0;
                } else {
                    *cp = s;
                }
            }
        }
    }
    __syncthreads();
    // the clock moves on to the next input row
    if (++c.ph == stride) {
        c.ph = 0;
        if (++c.hi_slot == ring_rows) c.hi_slot = 0;
        if (c.hi_sat < (1 << 20)) ++c.hi_sat;
    }
    if (c.tf_neg > 0) --c.tf_neg;
    else if (++c.phf == stride) c.phf = 0;
    if (completes && ++c.done_slot == ring_rows) c.done_slot = 0;
    k = c;
    return completes;
}

// The row `cur` goes up through the layers from `first` on; the net's output row is written out.  (Inlined, with one call of
// fused_feed: behind a call the arguments would be read through a generic pointer, which costs a trip to the cache per field.)
template <typename TS>
__device__ __forceinline__ void fused_cascade(const FusedArgs& a, int first, const typename RowOf<TS>::T* cur, unsigned char* smem, LayerClock* clk, int G, int g0,
                                              int& out_row, unsigned long long* ev_local)
{
    typedef typename RowOf<TS>::T TR;
    for (int n = first; n < a.n_layers; ++n) {
        if (!fused_feed<TS>(a, n, cur, smem, clk[n], G, ev_local)) return;
        cur = (const TR*)(smem + a.layer[n].rowbuf_soff);
    }
    // a finished row of the last layer
    const FusedLayer& Z = a.layer[a.n_layers - 1];
    const int row_elems = Z.Wout * Z.Cout, out_elem = a.out_elem;
    const long long cap = a.out_cap;
    void* out = a.out;
    for (int g = 0; g < G; ++g)
        for (int q = threadIdx.x; q < row_elems; q += blockDim.x) {
            const long long at = ((long long)(g0 + g) * cap + out_row) * row_elems + q;
            if (IDF_OK_AT(a.status, at, (long long)a.S * cap * row_elems)) store_elem<TR>(out, at, out_elem, cur[g * row_elems + q]);
        }
    out_row += 1;
    __syncthreads();
}

template <typename TS>
__global__ void __launch_bounds__(512) depth_first_kernel(const __grid_constant__ FusedArgs a)
{
    typedef typename RowOf<TS>::T TR;
    extern __shared__ __align__(16) unsigned char fsmem[];
    __shared__ unsigned long long ev_local[FUSED_MAX_LAYERS];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int g0 = blockIdx.x * a.G;
    const int G = min(a.G, a.S - g0);
    LayerClock clk[FUSED_MAX_LAYERS];
    for (int i = 0; i < a.n_layers; ++i) {
        const FusedLayer& L = a.layer[i];
        clk[i].ph = L.ph0; clk[i].hi_slot = L.hi_slot0; clk[i].hi_sat = L.hi_sat0; clk[i].phf = L.phf0; clk[i].tf_neg = L.tf_neg0;
        clk[i].done_slot = L.done_slot0;
    }
    int out_row = a.out_row0;
    if (threadIdx.x < FUSED_MAX_LAYERS) ev_local[threadIdx.x] = 0;
    // parameters come on chip while the previous kernel of the stream still runs: they do not depend on it
    for (int i = 0; i < a.n_layers; ++i) {
        const FusedLayer& L = a.layer[i];
        const int w_soff = L.w_soff, b_soff = L.b_soff, n_w = (L.w_bytes + 15) >> 4, n_b = L.Cout;      // (every region starts on a 256-byte boundary)
        const unsigned char *src = (const unsigned char*)a.weights + L.w_src, *bsrc = (const unsigned char*)a.weights + L.bias_off;
        if (w_soff >= 0)
            for (int e = threadIdx.x; e < n_w; e += blockDim.x) copy_async<16>(fsmem + w_soff + 16 * e, src + 16 * e);
        if (b_soff >= 0)
            for (int e = threadIdx.x; e < n_b; e += blockDim.x) copy_async<4>(fsmem + b_soff + 4 * e, bsrc + 4 * e);
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ---- the group's rolling state and the first segment come on chip.  Asynchronous copies for everything that needs no
    // conversion: a launch for a single segment then pays the latency of one load, not of one per layer
    for (int i = 0; i < a.n_layers; ++i) {
        const FusedLayer& L = a.layer[i];
        const int row_elems = L.Wout * L.Cout, rows = L.kind == 0 ? L.ring_rows : 1, n = G * row_elems, soff = L.state_soff, elem = L.out_elem;
        const bool words = L.kind == 0 || elem == E_F32;
        const unsigned char* src = (const unsigned char*)L.state;
        for (int slot = 0; slot < rows; ++slot) {
            const long long first = ((long long)slot * a.S + g0) * row_elems;
            for (int q = threadIdx.x; q < n; q += blockDim.x) {
                if (!IDF_OK_AT(a.status, first + q, (long long)rows * a.S * row_elems)) continue;
                if (words) copy_async<4>(fsmem + soff + 4 * (slot * n + q), src + 4 * (first + q));
                else ((TR*)(fsmem + soff))[q] = load_elem<TR>(src, first + q, elem);
            }
        }
    }
    TR* inrow = (TR*)(fsmem + a.in_soff);
    const int in_elems = a.in_w * a.in_c;
    if (a.n_seg > 0)
        for (int e = threadIdx.x; e < G * in_elems; e += blockDim.x) {
            const long long at = (long long)g0 * in_elems + e;
            if (IDF_OK_AT(a.status, at, (long long)a.n_seg * a.S * in_elems)) inrow[e] = load_elem<TR>(a.in, at, a.in_elem);
        }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    // ---- segments, one at a time, each through every layer it can reach
    for (int seg = 0; seg < a.n_seg; ++seg) {
        if (seg > 0) {
            for (int e = threadIdx.x; e < G * in_elems; e += blockDim.x) {
                const long long at = ((long long)seg * a.S + g0) * in_elems + e;
                if (IDF_OK_AT(a.status, at, (long long)a.n_seg * a.S * in_elems)) inrow[e] = load_elem<TR>(a.in, at, a.in_elem);
            }
            __syncthreads();
        }
        fused_cascade<TS>(a, 0, inrow, fsmem, clk, G, g0, out_row, ev_local);
    }
    // ---- end of input: rows that wait only for bottom zero padding are complete as they stand, in depth order
    // (how many each layer has is a matter of row counts: worked out by the host for the rows the layer will have received)
    if (a.flush) {
        for (int i = 0; i < a.n_layers; ++i) {
            const FusedLayer& L = a.layer[i];
            if (L.kind != 0) continue;                   // (an unpaired pooling row is dropped)
            const int row_elems = L.Wout * L.Cout;
            const TS* bias = L.bias_off < 0 ? nullptr : L.b_soff >= 0 ? (const TS*)(fsmem + L.b_soff) : (const TS*)((const unsigned char*)a.weights + L.bias_off);
            for (int n = 0; n < L.n_flush; ++n) {
                TS* ring = (TS*)(fsmem + L.state_soff);
                TR* rowbuf = (TR*)(fsmem + L.rowbuf_soff);
                for (int e = threadIdx.x; e < G * row_elems; e += blockDim.x) {
                    const int g = e / row_elems, q2 = e - g * row_elems;
                    TS* cp = ring + (clk[i].done_slot * G + g) * row_elems + q2;
                    rowbuf[e] = fused_act(*cp, bias ? bias[q2 % L.Cout] : (TS)0, L.relu, L.shift, L.round_bf16);
                    *cp = 0;
                }
                __syncthreads();
                if (++clk[i].done_slot == L.ring_rows) clk[i].done_slot = 0;
                fused_cascade<TS>(a, i + 1, rowbuf, fsmem, clk, G, g0, out_row, ev_local);
            }
        }
    }
    // ---- the state goes back
    for (int i = 0; i < a.n_layers; ++i) {
        const FusedLayer& L = a.layer[i];
        const int row_elems = L.Wout * L.Cout, rows = L.kind == 0 ? L.ring_rows : 1, n = G * row_elems, soff = L.state_soff, elem = L.out_elem, kind = L.kind;
        void* dst = L.state;
        for (int slot = 0; slot < rows; ++slot) {
            const long long first = ((long long)slot * a.S + g0) * row_elems;
            for (int q = threadIdx.x; q < n; q += blockDim.x) {
                if (!IDF_OK_AT(a.status, first + q, (long long)rows * a.S * row_elems)) continue;
                if (kind == 0) ((TS*)dst)[first + q] = ((const TS*)(fsmem + soff))[slot * n + q];
                else store_elem<TR>(dst, first + q, elem, ((const TR*)(fsmem + soff))[q]);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < a.n_layers && ev_local[threadIdx.x] && a.counters) atomicAdd(a.counters + threadIdx.x, ev_local[threadIdx.x]);
}

}  // namespace

cudaError_t launch_depth_first(const FusedArgs& a, int int_net, int threads, size_t smem_bytes, cudaStream_t st)
{
    if (a.S <= 0 || (a.n_seg <= 0 && !a.flush)) return cudaSuccess;
    const unsigned grid = (unsigned)((a.S + a.G - 1) / a.G);
    auto kf = int_net ? depth_first_kernel<int> : depth_first_kernel<float>;
    static bool attr_set[2][64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[int_net ? 1 : 0][dev]) {
        cudaError_t e = cudaFuncSetAttribute(kf, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FUSED_SMEM_LIMIT);
        if (e != cudaSuccess) return e;
        attr_set[int_net ? 1 : 0][dev] = true;
    }
    return launch_pdl(kf, grid, (unsigned)threads, smem_bytes, st, a);
}

}  // namespace idf
