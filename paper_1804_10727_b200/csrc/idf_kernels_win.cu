// Window kernel: thin layers (few input channels, the raw input of a net) on the tensor cores.
//
// A thin layer has so little arithmetic per output that it is bound by the bytes it writes, as long as every other
// role keeps out of the way.  What costs in the usual im2col form is that an output position owns a row of the A
// operand: Kh*Kw*Cin values gathered one by one, and an accumulator row of only Cout columns.  Here a row of A is a
// WINDOW: the input one stream needs for P neighbouring outputs (P positions of a row, or P rows of a 1D signal).
// Per tap row ky that is ONE contiguous run of (P - 1)*stride + Kw positions, copied word by word (funnel shift for
// its alignment); the weights are laid out once as the banded matrix
//     B[(p, co)][(ky, e)] = w[co][ky][kx][ci]   for e = (p*stride + kx)*Cin + ci, zero elsewhere,
// so one MMA of N = P*Cout columns (at most 256) yields all P outputs of 128 windows, and the P*Cout results of a
// window are contiguous in the emitted row.  The zeros in B cost tensor time the layer has plenty of (2 -> 32 channels,
// 3x3: 256 cycles per 1024 positions); K = Kh runs padded to words, at most 128 bytes.
//
// Roles: warps 0-7   two sets of four builder warps, taking steps in turn (a step = 128 windows of one output row),
//                    the input of a set's next step in flight while the other set's is built;
//        warp 8      MMA issuer, two accumulator sets of 256 TMEM columns;
//        warps 9-20  three epilogue groups that take a step's columns in turn, 32 at a time: f(c + b), rounding or
//                    requantisation, 32 bytes per thread and instruction straight into the output row.
// Steps that exchange rows with the ring (begun by an earlier block, or left open by this one) are the same MMAs with
// the missing input rows as zeros; the epilogue then adds what the ring holds and parks what stays open.  Where two
// such rows can meet in one ring slot, those of a tile are one work item and a slot's words belong to one thread, which
// takes the rows in order, or the carried rows are read from a copy of the ring.  A freed slot is left zero where the event scatter shares the ring.  All else are independent work items, dealt round robin to one
// CTA per SM.  Layers that report their input events (Eq. 3: non-zero components) count them while the runs pass by.
//
// Measured on B200, against the kernels that served these layers before (event scatter on CUDA cores; one im2col row per
// output; x-unfold pass + row ring): 2 -> 32 channels int8, 2048 streams of 256-wide rows, 256 rows 5.46 -> 1.75 ms;
// 1 -> 16 int8, 4096 28x28 images 0.287 -> 0.033 ms; 1 -> 32 bf16 1D, 1024 streams of 16000 samples 0.54 -> 0.16 ms;
// 3 -> 64 bf16, 64 streams of 224-wide rows, 112 rows 0.094 -> 0.071 ms.
#include "../../include/idf.h"
#include "idf_ptx.h"

#include <cstring>

namespace idf {

namespace {

constexpr int WIN_BUILD_SETS = 2;
constexpr int WIN_MMA_WARP = 4 * WIN_BUILD_SETS;
constexpr int WIN_EPI_GROUPS = 3;
constexpr int WIN_THREADS = 32 * (WIN_MMA_WARP + 1 + 4 * WIN_EPI_GROUPS);
constexpr int WIN_STAGES = 4;
constexpr int WIN_MAX_WORDS = 32;            // 32-bit words of a window row (128 bytes)

struct WinArgs {
    const void* in;              // input rows of the block: [n_in][S][Win][Cin]
    const void* bias;
    void* ring;
    const void* ring_in;         // where the rows begun by earlier blocks are read: the ring, or a copy of it
    void* out;
    unsigned int* status;
    unsigned long long* events;  // count the non-zero input components here (int8 layers), or nullptr
    long long out_row_stride, out_stream_stride;   // in elements
    long long out_row_first;     // row index of visited row 0 in the output buffer
    int n_in, n_rows, done_rel, base_ty, carried;      // input rows, visited output rows, emitted ones; tap ky of visited row o reads
                                 // input row o*stride + ky - base_ty; carried: rows with o*stride < base_ty were begun by an earlier block
    int ring_slot0, ring_rows;   // ring slot of visited row 0
    int S, Win, Wout, Cin, Cout, Kh, Kw, stride, stride_x, pad_x, relu, shift, out_elem;
    int P, nxw, ncol, n_tiles;   // outputs per window, windows per row, windows per output row of all streams, tiles of 128
    int run_words;               // words of a tap row's run
    int swb, ksteps, N;
    int out_wide;                // output rows are whole 32-byte groups per 32 columns, 32-byte aligned
    unsigned int inv_c16;        // q * inv_c16 >> 16 = q / (Cout / 16) for q < 16
    // steps (2D: output rows, 1D: runs of P output rows): [e0_end, e1_begin) exchange nothing with the ring.  `ordered`: two
    // visited rows share a ring slot, so the other steps ([0, e0_end) and [e1_begin, n_steps)) of a tile are one work item;
    // all else are independent work items of R steps
    int n_steps, e0_end, e1_begin, R, ordered, n_items;
    int clear;                   // leave the slots of emitted rows zero (the scatter kernel starts its rows from what the ring holds)
    int parts, part_cols;        // a work item is all N columns of its windows (1 part), or one of `parts` runs of part_cols
    long long in_elems, out_elems, ring_elems;
};

// byte i of a word is non-zero -> bit 7 of byte i
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t x) { return (((x & 0x7f7f7f7fu) + 0x7f7f7f7fu) | x) & 0x80808080u; }
// bytes [lo, 4 - hi) of a word (shl / shr by 32 give 0)
__device__ __forceinline__ uint32_t byte_mask(int lo, int hi)
{
    lo = lo < 0 ? 0 : (lo > 4 ? 4 : lo);
    hi = hi < 0 ? 0 : (hi > 4 ? 4 : hi);
    uint32_t a, b;
    asm("shl.b32 %0, %1, %2;" : "=r"(a) : "r"(0xffffffffu), "r"(8 * lo));
    asm("shr.u32 %0, %1, %2;" : "=r"(b) : "r"(0xffffffffu), "r"(8 * hi));
    return a & b;
}
__device__ __forceinline__ void st_shared16(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
// Walks the steps this CTA takes.  A work item is a tile of 128 windows and the steps [a0, a0 + na), then from b0 on (n in all).
struct WinWalk {
    int it, i, n, a0, na, b0, tile, part;
    __device__ __forceinline__ void open(const WinArgs& a)
    {
        i = 0;
        if (it >= a.n_items) { n = 0; return; }
        int grp = it / a.n_tiles;
        tile = it - grp * a.n_tiles;
        part = 0;
        if (a.parts > 1) {
            const int g = grp / a.parts;
            part = grp - g * a.parts;
            grp = g;
        }
        if (a.ordered && grp == 0) {
            a0 = 0; na = a.e0_end; b0 = a.e1_begin; n = a.e0_end + (a.n_steps - a.e1_begin);
        } else {
            a0 = a.ordered ? a.e0_end + (grp - 1) * a.R : grp * a.R;
            na = min(a.R, (a.ordered ? a.e1_begin : a.n_steps) - a0);
            b0 = 0; n = na;
        }
    }
    __device__ __forceinline__ void start(const WinArgs& a) { it = blockIdx.x; open(a); }
    __device__ __forceinline__ bool at_end(const WinArgs& a) const { return it >= a.n_items; }
    __device__ __forceinline__ int step() const { return i < na ? a0 + i : b0 + (i - na); }
    // on to the next step; true if that is another work item
    __device__ __forceinline__ bool next(const WinArgs& a)
    {
        if (++i < n) return false;
        it += gridDim.x;
        open(a);
        return true;
    }
};

// A window is one row of A for all its outputs: an infinity or a NaN in it meets the zeros of B and turns the sums of outputs that do
// not read it into NaN - in all Cout columns, so a look at the first of 16 finds them.  Such 16 columns (k-th of the window; bf16 layers) are
// worked out here instead, one by one, from the output's own taps: added to what the ring holds, parked or emitted.  A call, by the thread
// concerned, behind the look: inlined, or with the sums put back in tensor memory, it cost the launches without such values 1-5 %
// (vgg2d one row per push 9.30 ms without any of it, 9.35 so, 9.41-9.77 the other ways; one push 1.35, 1.35, 1.36-1.37).
template <int AX>
__device__ __noinline__ void own_taps_only(const WinArgs& a, uint32_t sW, int k, int s, int xw, int step)
{
    const __nv_bfloat16* in = (const __nv_bfloat16*)a.in;
    const int p = 16 * k / a.Cout, o = AX == 0 ? step : step * a.P + p;
    const int x = AX == 0 ? xw * a.P + p : 0, ty = o * a.stride - a.base_ty;            // ty: the first tap's input row
    const bool emit = o < a.done_rel, carried = a.carried && ty < 0;
    float* ring = (float*)a.ring;
#pragma unroll 1
    for (int n = 16 * k; n < 16 * k + 16; ++n) {
        const int co = n - p * a.Cout;
        const uint32_t phase = a.swb == 128 ? (uint32_t)(n & 7) : (a.swb == 64 ? (uint32_t)((n >> 1) & 3) : (uint32_t)((n >> 2) & 1));
        float sum = 0.f;
#pragma unroll 1
        for (int ky = 0; ky < a.Kh; ++ky) {
            if ((unsigned)(ty + ky) >= (unsigned)a.n_in) continue;
#pragma unroll 1
            for (int i = 0; i < a.Kw * a.Cin; ++i) {
                const int e = AX == 0 ? (x * a.stride_x - a.pad_x) * a.Cin + i : i;     // value of the stream's row
                if ((unsigned)e >= (unsigned)(a.Win * a.Cin)) continue;
                const long long at = ((long long)(ty + ky) * a.S + s) * a.Win * a.Cin + e;
                if (!IDF_OK_AT(a.status, at, a.in_elems)) continue;
                const uint32_t b = 2u * (uint32_t)(AX == 0 ? 2 * ky * a.run_words + p * a.stride_x * a.Cin + i : (p * a.stride + ky) * a.Cin + i);
                unsigned short w;
                asm volatile("ld.shared.u16 %0, [%1];" : "=h"(w) : "r"(sW + (uint32_t)(n * a.swb) + (((b >> 4) ^ phase) << 4) + (b & 15u)));
                sum = fmaf(__bfloat162float(__ushort_as_bfloat16(w)), __bfloat162float(in[at]), sum);
            }
        }
        const long long ri = ((long long)((a.ring_slot0 + o) % a.ring_rows) * a.S + s) * a.Wout * a.Cout + (long long)x * a.Cout + co;
        if ((carried || !emit) && !IDF_OK_AT(a.status, ri, a.ring_elems)) continue;
        if (carried) sum += ((const float*)a.ring_in)[ri];
        if (!emit) { ring[ri] = sum; continue; }
        if (a.bias) sum += ((const float*)a.bias)[co];
        if (a.relu) sum = a.out_elem == E_BF16 ? (sum < 0.f ? 0.f : sum) : fmaxf(sum, 0.f);      // (as emit16f)
        const long long at = (a.out_row_first + o) * a.out_row_stride + (long long)s * a.out_stream_stride + (long long)x * a.Cout + co;
        if (!IDF_OK_AT(a.status, at, a.out_elems)) continue;
        if (a.out_elem == E_BF16) ((__nv_bfloat16*)a.out)[at] = __float2bfloat16_rn(sum);
        else ((float*)a.out)[at] = sum;
    }
}
__device__ __forceinline__ bool is_nan(uint32_t v) { return __uint_as_float(v) != __uint_as_float(v); }

// AX 0: a window runs along x; 1: along the rows (1D nets).  RWT: words of a run of a 3-row layer, known at compile time
// (the whole window is then fetched one step ahead and leaves in 16-byte stores), or 0.
template <int DT, int AX, int RWT>
__global__ void __launch_bounds__(WIN_THREADS, 1)
conv_win_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ WinArgs a)
{
    constexpr int ES = DT == 1 ? 2 : 1;
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ __align__(8) unsigned long long s_bars[2 * WIN_STAGES + 5];

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t stage_bytes = 128u * (uint32_t)a.swb;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sW = base;                                                       // [N][swb]
    const uint32_t sA = (sW + (uint32_t)a.N * a.swb + 1023u) & ~1023u;
    const uint32_t bar_full = smem_u32(s_bars), bar_empty = bar_full + 8u * WIN_STAGES, bar_w = bar_empty + 8u * WIN_STAGES;
    const uint32_t bar_acc = bar_w + 8u, bar_free = bar_acc + 16u;

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int i = 0; i < WIN_STAGES; ++i) { mbar_init(bar_full + 8u * i, 4); mbar_init(bar_empty + 8u * i, 1); }
        mbar_init(bar_w, 1);
        for (int i = 0; i < 2; ++i) { mbar_init(bar_acc + 8u * i, 1); mbar_init(bar_free + 8u * i, 4 * WIN_EPI_GROUPS); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar_w, (uint32_t)a.N * a.swb);                               // the parameters do not depend on earlier kernels
        tma_load_2d(sW, &tmW, bar_w, 0, 0);
    }
    if (warp == WIN_MMA_WARP) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // window rows nobody writes (beyond the last window, the K tail) must hold finite values: zero, once
    for (uint32_t i = threadIdx.x; i < WIN_STAGES * stage_bytes / 16u; i += WIN_THREADS) st_shared16(sA + 16u * i, 0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;

    if (warp < WIN_MMA_WARP) {
        // ------------------------------ builders -----------------------------------------------
        const int set = warp >> 2, m = (warp & 3) * 32 + lane;
        const uint32_t phase = a.swb == 128 ? (uint32_t)(m & 7) : (a.swb == 64 ? (uint32_t)((m >> 1) & 3) : (uint32_t)((m >> 2) & 1));
        const uint32_t row_at = sA + (uint32_t)m * a.swb;
        const int row_bytes = a.Win * a.Cin * ES;
        const long long row_pitch = (long long)a.S * row_bytes;                     // from one input row to the next
        unsigned int n_events = 0;
        bool ok = true;
        WinWalk w;
        w.start(a);
        // where this thread's window lies in its stream's rows
        bool live = false;
        int b0 = 0, own = 0;
        const unsigned char* in_s = (const unsigned char*)a.in;
        auto geometry = [&]() {
            const int col = w.tile * 128 + m;
            live = col < a.ncol;
            const int s = AX == 0 ? col / a.nxw : col, xw = AX == 0 ? col - s * a.nxw : 0;
            b0 = (xw * a.P * a.stride_x - a.pad_x) * a.Cin * ES;
            own = live && w.part == 0 ? (xw == a.nxw - 1 ? 4 * WIN_MAX_WORDS : a.P * a.Cin * ES) : 0;   // (events: bytes of a run that are this window's to count)
            in_s = (const unsigned char*)a.in + (long long)s * row_bytes;
        };
        int stage = set;                                                            // steps go round the stages (and the two sets)
        uint32_t ph = 1;
        for (int k = 0; k < set && !w.at_end(a); ++k) w.next(a);
        if (!w.at_end(a)) geometry();
        auto wait_empty = [&]() {
            int got = 1;
            if (lane == 0) got = mbar_wait(bar_empty + 8u * stage, ph, abort_flag) ? 1 : 0;
            return __shfl_sync(0xffffffffu, got, 0) != 0;
        };
        auto advance = [&]() {
            stage += WIN_BUILD_SETS;
            if (stage >= WIN_STAGES) { stage -= WIN_STAGES; ph ^= 1u; }
            if (w.i + WIN_BUILD_SETS < w.n) { w.i += WIN_BUILD_SETS; return; }
            for (int k = 0; k < WIN_BUILD_SETS && !w.at_end(a); ++k) w.next(a);
            if (!w.at_end(a)) geometry();
        };
        if constexpr (AX == 0 && RWT > 0) {
            // Per item: which bytes of a run lie in the stream's row, and which of them are this window's to count as events.
            // What decides the time of a builder is its instruction count (one dependent chain per warp), so nothing of this is
            // worked out per step.
            uint32_t raw[3][RWT + 1], sh[3], mask[RWT], own_mask[RWT], packed_events = 0;
            const uintptr_t in_lo = (uintptr_t)a.in & ~(uintptr_t)3, in_hi = ((uintptr_t)a.in + (unsigned long long)a.n_in * row_pitch + 3) & ~(uintptr_t)3;
            auto masks = [&]() {
#pragma unroll
                for (int j = 0; j < RWT; ++j) {
                    mask[j] = byte_mask(-(b0 + 4 * j), b0 + 4 * j + 4 - row_bytes);
                    own_mask[j] = byte_mask(0, 4 * j + 4 - own);
                }
            };
            auto fetch = [&]() {
                const int r0 = w.step() * a.stride - a.base_ty;
                const uintptr_t row = (uintptr_t)in_s + (long long)r0 * row_pitch + b0;
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    const uintptr_t at = row + ky * row_pitch;
                    sh[ky] = 8u * (uint32_t)(at & 3);
                    const uintptr_t p = at & ~(uintptr_t)3;
                    const bool have = live && (unsigned)(r0 + ky) < (unsigned)a.n_in;
                    // (words beside the row are masked; only those beside the whole input must not be touched)
                    if (have && p >= in_lo && p + 4 * (RWT + 1) <= in_hi) {
#pragma unroll
                        for (int j = 0; j <= RWT; ++j) raw[ky][j] = __ldg((const uint32_t*)p + j);
                    } else {
#pragma unroll
                        for (int j = 0; j <= RWT; ++j)
                            raw[ky][j] = (have && p + 4 * j >= in_lo && p + 4 * j + 4 <= in_hi) ? __ldg((const uint32_t*)p + j) : 0u;
                    }
                }
            };
            int item = -1;
            if (!w.at_end(a)) { masks(); item = w.it; fetch(); }
            while (!w.at_end(a) && ok) {
                const uint32_t at = row_at + (uint32_t)stage * stage_bytes, bar = bar_full + 8u * stage;
                if (!wait_empty()) { ok = false; break; }
                // four words of the window at a time
#pragma unroll
                for (int c = 0; c < (3 * RWT + 3) / 4; ++c) {
                    uint32_t v[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        constexpr int RW1 = RWT;                                    // (k / RWT, k % RWT are known at compile time)
                        const int k = 4 * c + u, ky = k / RW1, j = k - ky * RW1;
                        v[u] = 0u;
                        if (k < 3 * RWT) {
                            v[u] = __funnelshift_r(raw[ky][j], raw[ky][j + 1], sh[ky]) & mask[j];
                            // (events; stride 1: every input row is tap row 0 of exactly one visited output row)
                            if (DT == 2 && ky == 0) packed_events += nonzero_bytes(v[u] & own_mask[j]) >> 7;
                        }
                    }
                    if (live) st_shared16(at + (((uint32_t)c ^ phase) << 4), v[0], v[1], v[2], v[3]);
                }
                if (DT == 2) { n_events = __dp4a(packed_events, 0x01010101u, n_events); packed_events = 0; }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the tensor core reads these rows through the async proxy
                __syncwarp();
                if (lane == 0) mbar_arrive(bar);
                advance();
                if (!w.at_end(a)) {
                    if (w.it != item) { masks(); item = w.it; }
                    fetch();                                                        // in flight while the other set's step is built
                }
            }
        } else {
            while (!w.at_end(a) && ok) {
                const uint32_t at = row_at + (uint32_t)stage * stage_bytes;
                const int step = w.step();
                if (AX == 0) {
                    if (!wait_empty()) { ok = false; break; }
                    for (int ky = 0; ky < a.Kh && live; ++ky) {
                        const int ri = step * a.stride + ky - a.base_ty;
                        const bool have = (unsigned)ri < (unsigned)a.n_in && IDF_OK_AT(a.status, ((long long)(ri + 1) * a.S) * a.Win * a.Cin - 1, a.in_elems);
                        const uintptr_t from = (uintptr_t)in_s + (intptr_t)(ri * row_pitch + b0);
                        const int al = (int)(from & 3);
                        const uint32_t* p = (const uint32_t*)(from - al);
                        for (int j0 = 0; j0 < a.run_words; j0 += 8) {
                            uint32_t raw[9];
#pragma unroll
                            for (int j = 0; j <= 8; ++j)       // (a word is touched only if it holds a byte of the row)
                                raw[j] = (have && j0 + j <= a.run_words && (unsigned)(b0 - al + 4 * (j0 + j) + 3) < (unsigned)(row_bytes + 3)) ? __ldg(p + j0 + j) : 0u;
#pragma unroll
                            for (int j = 0; j < 8; ++j) {
                                if (j0 + j >= a.run_words) break;
                                const int q = b0 + 4 * (j0 + j);
                                const uint32_t x = __funnelshift_r(raw[j], raw[j + 1], 8u * (uint32_t)al) & byte_mask(-q, q + 4 - row_bytes);
                                if (DT == 2 && a.events && ky == 0) n_events += __popc(nonzero_bytes(x & byte_mask(0, 4 * (j0 + j) + 4 - own)));
                                const uint32_t k = (uint32_t)(ky * a.run_words + j0 + j);
                                asm volatile("st.shared.b32 [%0], %1;" ::"r"(at + (((k >> 2) ^ phase) << 4) + 4u * (k & 3u)), "r"(x) : "memory");
                            }
                        }
                    }
                } else {
                    // P output rows of one stream: (P - 1)*stride + Kh samples of Cin values, a stream apart in memory each.
                    // The first 16-byte pieces are fetched before the wait for the stage.
                    constexpr int EPC = 16 / ES;                                    // values of a 16-byte piece
                    constexpr int G = ES == 2 ? 3 : 1;                              // pieces in flight
                    const int n_val = ((a.P - 1) * a.stride + a.Kh) * a.Cin;
                    int ri = step * a.P * a.stride - a.base_ty, ci = 0;
                    const unsigned char* p = in_s + (long long)ri * row_pitch;
                    bool waited = false;
                    for (int e0 = 0; e0 < n_val; e0 += G * EPC) {
                        uint32_t x[G * EPC];
#pragma unroll
                        for (int u = 0; u < G * EPC; ++u) {
                            const bool have = live && e0 + u < n_val && (unsigned)ri < (unsigned)a.n_in &&
                                              IDF_OK_AT(a.status, ((long long)ri * a.S * a.Win) * a.Cin + ci, a.in_elems);
                            x[u] = 0u;
                            if (have) x[u] = ES == 2 ? (uint32_t)__ldg((const unsigned short*)p + ci) : (uint32_t)__ldg(p + ci);
                            if (++ci == a.Cin) { ci = 0; ++ri; p += row_pitch; }
                        }
                        if (!waited) { ok = wait_empty(); waited = true; }
                        if (!ok) break;
#pragma unroll
                        for (int g = 0; g < G; ++g) {
                            if (e0 + g * EPC >= n_val || !live) break;
                            const uint32_t* y = x + g * EPC;
                            uint32_t v[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q)
                                v[q] = ES == 2 ? (y[(2 * q) % EPC] | (y[(2 * q + 1) % EPC] << 16))
                                               : (y[(4 * q) % EPC] | (y[(4 * q + 1) % EPC] << 8) | (y[(4 * q + 2) % EPC] << 16) | (y[(4 * q + 3) % EPC] << 24));
                            st_shared16(at + (((uint32_t)(e0 / EPC + g) ^ phase) << 4), v[0], v[1], v[2], v[3]);
                        }
                    }
                    if (!ok) break;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_full + 8u * stage);
                advance();
            }
        }
        if (DT == 2 && AX == 0 && a.events) {
            for (int o = 16; o; o >>= 1) n_events += __shfl_xor_sync(0xffffffffu, n_events, o);
            if (lane == 0 && n_events) atomicAdd(a.events, (unsigned long long)n_events);
        }
    } else if (warp == WIN_MMA_WARP) {
        // ------------------------------ MMA issuer ---------------------------------------------
        const uint64_t desc_hi = make_smem_desc(0, a.swb);
        const uint32_t idesc = (DT == 1 ? ((1u << 4) | (1u << 7) | (1u << 10)) : ((2u << 4) | (1u << 7) | (1u << 10))) |
                               ((128u >> 4) << 24) | ((uint32_t)(a.part_cols >> 3) << 17);
        const uint64_t bdesc0 = desc_hi | (uint64_t)((sW & 0x3FFFFu) >> 4);
        const uint32_t part_units = (uint32_t)a.part_cols * a.swb >> 4;       // (a multiple of eight rows: the swizzle pattern starts over)
        bool ok = mbar_wait(bar_w, 0, abort_flag);
        const bool issuer = elect_one();
        int t = 0, stage = 0;
        uint32_t ph = 0;
        WinWalk w;
        for (w.start(a); !w.at_end(a) && ok; w.next(a), ++t) {
            const int acc = t & 1;
            if (!mbar_wait(bar_free + 8u * acc, (uint32_t)((t >> 1) & 1) ^ 1u, abort_flag)) { ok = false; break; }
            if (!mbar_wait(bar_full + 8u * stage, ph, abort_flag)) { ok = false; break; }
            tc_fence_after();
            if (issuer) {
                const uint64_t adesc = desc_hi | (uint64_t)(((sA + (uint32_t)stage * stage_bytes) & 0x3FFFFu) >> 4);
                const uint32_t d = tmem_base + 256u * acc;
                const uint64_t bdesc = bdesc0 + (uint64_t)((uint32_t)w.part * part_units);
                if (a.ksteps == 1) umma_tile<DT, 1, true>(d, adesc, bdesc, idesc);
                else if (a.ksteps == 2) umma_tile<DT, 2, true>(d, adesc, bdesc, idesc);
                else if (a.ksteps == 3) umma_tile<DT, 3, true>(d, adesc, bdesc, idesc);
                else umma_tile<DT, 4, true>(d, adesc, bdesc, idesc);
                umma_commit(bar_empty + 8u * stage);
                umma_commit(bar_acc + 8u * acc);
            }
            __syncwarp();
            if (++stage == WIN_STAGES) { stage = 0; ph ^= 1u; }
        }
    } else {
        // ------------------------------ epilogue -----------------------------------------------
        const int q = warp & 3, grp = (warp - WIN_MMA_WARP - 1) >> 2;               // TMEM lane quarter; column groups in turn
        const int m = q * 32 + lane;
        const uint32_t tlane = tmem_base + ((uint32_t)(q * 32) << 16);
        const int oes = a.out_elem == E_F32 ? 4 : (a.out_elem == E_BF16 ? 2 : 1);
        const int n_chunk = (a.part_cols + 31) >> 5;
        unsigned char* out = (unsigned char*)a.out;
        uint32_t* ring = (uint32_t*)a.ring;
        const uint32_t* ring_in = (const uint32_t*)a.ring_in;
        const long long ring_row = (long long)a.Wout * a.Cout;
        bool ok = true;
        int t = 0, first = grp;                                                    // this group's first chunk in the step at hand
        int s = 0, xw = 0, n_pos = 0;
        long long o_base = 0;                                                      // window's element offset in an output row
        WinWalk w;
        w.start(a);
        bool fresh = true;
        while (!w.at_end(a) && ok) {
            if (fresh) {
                const int col = w.tile * 128 + m;
                s = AX == 0 ? col / a.nxw : col;
                xw = AX == 0 ? col - s * a.nxw : 0;
                n_pos = col < a.ncol ? (AX == 0 ? min(a.P, a.Wout - xw * a.P) : a.P) : 0;     // outputs of this window that exist
                o_base = (long long)s * a.out_stream_stride + (AX == 0 ? (long long)xw * a.P * a.Cout : 0);
            }
            const int step = w.step();
            const int acc = t & 1;
            const int k_part = w.part * n_chunk;                                     // the item's first piece of 32 columns
            const uint32_t trow = tlane + 256u * acc - 32u * (uint32_t)k_part;
            const long long o_row = o_base + (a.out_row_first + (AX == 0 ? step : step * a.P)) * a.out_row_stride;
            auto wait_acc = [&]() {
                int got = 1;
                if (lane == 0) got = mbar_wait(bar_acc + 8u * acc, (uint32_t)((t >> 1) & 1), abort_flag) ? 1 : 0;
                got = __shfl_sync(0xffffffffu, got, 0);
                tc_fence_after();
                return got != 0;
            };
            if (step >= a.e0_end && step < a.e1_begin) {
                // a step that exchanges nothing with the ring: 32 columns at a time
                if (!wait_acc()) { ok = false; break; }
                const int n_col = n_pos * a.Cout;
                unsigned char* dst = out + o_row * oes;
                int k = k_part + first;
                for (; k < k_part + n_chunk; k += WIN_EPI_GROUPS) {
                    const int c = 32 * k;
                    uint32_t v[32];
                    // where the two halves (16 channels of one output each) go: side by side in a row (2D), or a row each (1D)
                    unsigned char *d0 = dst + c * oes, *d1 = d0 + 16 * oes;
                    const uint32_t *b_lo = nullptr, *b_hi = nullptr;
                    if (AX == 1 || a.bias) {
                        const int p0 = (int)((2u * k * a.inv_c16) >> 16), p1 = (int)(((2u * k + 1u) * a.inv_c16) >> 16);
                        const int co0 = c - p0 * a.Cout, co1 = c + 16 - p1 * a.Cout;
                        if (a.bias) { b_lo = (const uint32_t*)a.bias + co0; b_hi = (const uint32_t*)a.bias + co1; }
                        if (AX == 1) {
                            d0 = dst + (p0 * a.out_row_stride + co0) * oes;
                            d1 = dst + (p1 * a.out_row_stride + co1) * oes;
                        }
                    }
                    const bool lo = c < n_col && IDF_OK_AT(a.status, (d0 - out) / oes, a.out_elems - 15);
                    const bool hi = c + 16 < n_col && IDF_OK_AT(a.status, (d1 - out) / oes, a.out_elems - 15);
                    __syncwarp();
                    if (c + 32 <= a.N) tmem_ld<32>(trow + c, v);
                    else tmem_ld<16>(trow + c, v);
                    if (DT == 2) {
                        uint32_t pk[8];
                        if (!a.bias) {
                            pack_i8<32>(v, nullptr, a.relu, a.shift, pk);
                        } else {
                            pack_i8<16>(v, (const int*)b_lo, a.relu, a.shift, pk);
                            pack_i8<16>(v + 16, (const int*)b_hi, a.relu, a.shift, pk + 4);
                        }
                        if (a.out_wide) {
                            if (lo) st_global_v8(d0, pk);
                        } else {
                            if (lo) st_global_v4(d0, pk);
                            if (hi) st_global_v4(d1, pk + 4);
                        }
                    } else {
                        if (a.out_elem == E_BF16) {
                            if (lo) emit16f<E_BF16>(v, (const float*)b_lo, a.relu, d0, a.out_wide);
                            if (hi) emit16f<E_BF16>(v + 16, (const float*)b_hi, a.relu, d1, a.out_wide);
                        } else {
                            if (lo) emit16f<E_F32>(v, (const float*)b_lo, a.relu, d0, a.out_wide);
                            if (hi) emit16f<E_F32>(v + 16, (const float*)b_hi, a.relu, d1, a.out_wide);
                        }
                        const bool odd_lo = lo && is_nan(v[0]), odd_hi = hi && is_nan(v[16]);
                        if (odd_lo || odd_hi)
#pragma unroll 1
                            for (int h = odd_lo ? 0 : 1; h < (odd_hi ? 2 : 1); ++h) own_taps_only<AX>(a, sW, 2 * k + h, s, xw, step);
                    }
                }
                first = k - k_part - n_chunk;
            } else {
                // A step that exchanges rows with the ring, 16 columns at a time.  The columns' groups are fixed here; in an
                // ordered 1D item the group goes by ring slot (a column run is a row of its own there).
                bool waited = false;
                for (int k = 2 * k_part; k < 2 * (k_part + n_chunk); ++k) {
                    const int c = 16 * k;
                    const int p = (int)(((uint32_t)k * a.inv_c16) >> 16), co = c - p * a.Cout;
                    const int o = AX == 0 ? step : step * a.P + p;                  // visited row (the same in all lanes)
                    const int slot = (a.ring_slot0 + o) % a.ring_rows;
                    if ((AX == 1 && a.ordered ? slot : k) % WIN_EPI_GROUPS != grp || c >= a.N || o >= a.n_rows) continue;
                    const bool emit = o < a.done_rel, carried = a.carried && o * a.stride < a.base_ty;
                    const long long ri = ((long long)slot * a.S + s) * ring_row + (AX == 0 ? (long long)(xw * a.P + p) * a.Cout : 0) + co;
                    const bool have = p < n_pos && IDF_OK_AT(a.status, ri, a.ring_elems - 15);
                    uint32_t r[16], v[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) r[j] = 0u;
                    if (have && carried) {                                         // (in flight while the accumulator is waited for)
                        ld_global_v8(ring_in + ri, *(uint32_t(*)[8])r);
                        ld_global_v8(ring_in + ri + 8, *(uint32_t(*)[8])(r + 8));
                    }
                    if (!waited) { waited = true; ok = wait_acc(); }
                    if (!ok) break;
                    __syncwarp();
                    tmem_ld<16>(trow + c, v);
                    if (!have) continue;
                    if (DT == 1 && is_nan(v[0])) { own_taps_only<AX>(a, sW, k, s, xw, step); continue; }
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        v[j] = DT == 1 ? __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(r[j])) : v[j] + r[j];
                    if (!emit) {
                        st_global_v8(ring + ri, *(uint32_t(*)[8])v);
                        st_global_v8(ring + ri + 8, *(uint32_t(*)[8])(v + 8));
                        continue;
                    }
                    if (carried && a.clear) {                                      // the slot is free again
                        const uint32_t z[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                        st_global_v8(ring + ri, z);
                        st_global_v8(ring + ri + 8, z);
                    }
                    const long long e = AX == 0 ? o_row + c : o_row + (long long)p * a.out_row_stride + co;
                    if (!IDF_OK_AT(a.status, e, a.out_elems - 15)) continue;
                    const uint32_t* b = a.bias ? (const uint32_t*)a.bias + co : nullptr;
                    if (DT == 2) {
                        uint32_t pk[4];
                        pack_i8<16>(v, (const int*)b, a.relu, a.shift, pk);
                        st_global_v4(out + e, pk);
                    } else if (a.out_elem == E_BF16) {
                        emit16f<E_BF16>(v, (const float*)b, a.relu, out + 2 * e, a.out_wide);
                    } else {
                        emit16f<E_F32>(v, (const float*)b, a.relu, out + 4 * e, a.out_wide);
                    }
                }
                if (ok && !waited) ok = wait_acc();
                if (!ok) break;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_free + 8u * acc);                       // one arrival per warp
            ++t;
            fresh = w.next(a);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (s_abort) {
        if (threadIdx.x == 0) {
            for (uint32_t i = 0; i < 4096 && !mbar_try_wait(bar_w, 0); ++i) __nanosleep(64);   // the CTA's own copy must land first
            atomicOr(a.status, 1u);
        }
        __syncthreads();
    }
    if (warp == WIN_MMA_WARP) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

}  // namespace

bool win_make_plan(int dtype, int S, int Wout, int Cin, int Cout, int Kh, int Kw, int stride, int stride_x, int one_d, WinPlan* p)
{
    *p = WinPlan{};
    if (dtype != 1 && dtype != 2) return false;
    if (Cout % 16 != 0 || Cout > 256) return false;
    const int es = dtype == 1 ? 2 : 1;
    // words of a window of P outputs; runs of 3-row layers are padded to the lengths known at compile time
    auto words = [&](int P, int* run) {
        *run = one_d ? (((P - 1) * stride + Kh) * Cin * es + 3) / 4 : (((P - 1) * stride_x + Kw) * Cin * es + 3) / 4;
        if (!one_d && Kh == 3) *run = *run <= 2 ? 2 : (*run <= 5 ? 5 : (*run <= 9 ? 9 : *run));
        return one_d ? *run : Kh * *run;
    };
    // The widest window whose outputs fit one instruction's 256 columns and whose input fits a 128-byte row; narrower where
    // the windows of one output row would otherwise be too few tiles of 128 to keep the SMs busy when rows arrive one at a
    // time (three visited rows each): a narrow window only means fewer zeros in B and more steps.
    int P = 256 / Cout, run = 0;
    while (P >= 1 && words(P, &run) > WIN_MAX_WORDS) --P;
    if (P < 1) return false;
    p->widest = P;
    if (one_d) {
        while (P > 2 && ((long long)S + 127) / 128 * (64 / P) < 64) P = (P + 1) / 2;
    } else {
        if (P > Wout) P = Wout;
        while (P > 1 && (long long)S * ((Wout + P - 1) / P) < 24LL * 128) P = (P + 1) / 2;
        const int n = (Wout + P - 1) / P;                // an even share of the row
        P = (Wout + n - 1) / n;
    }
    p->n_words = words(P, &run);
    p->P = P;
    p->run_words = run;
    p->one_d = one_d;
    p->nxw = one_d ? 1 : (Wout + P - 1) / P;
    p->swb = p->n_words <= 8 ? 32 : (p->n_words <= 16 ? 64 : 128);
    p->ksteps = (p->n_words + 7) / 8;
    p->N = P * Cout;
    p->smem_bytes = 1024 + ((size_t)p->N * p->swb + 1023) / 1024 * 1024 + (size_t)WIN_STAGES * 128 * p->swb;
    p->w_bytes = (size_t)p->N * p->swb;
    p->ok = 1;
    return true;
}

// The banded weight matrix [N][swb bytes] from weights [Cout][Kh][Kw][Cin] in the activation type.
void win_pack_weights(const WinPlan& p, int dtype, const void* w, int Cin, int Cout, int Kh, int Kw, int stride, int stride_x, void* dst)
{
    const size_t es = dtype == 1 ? 2 : 1;
    memset(dst, 0, p.w_bytes);
    for (int q = 0; q < p.P; ++q)
        for (int co = 0; co < Cout; ++co)
            for (int ky = 0; ky < Kh; ++ky)
                for (int kx = 0; kx < Kw; ++kx) {
                    const size_t at = p.one_d ? (size_t)(q * stride + ky) * Cin * es
                                              : (size_t)ky * p.run_words * 4 + (size_t)(q * stride_x + kx) * Cin * es;
                    memcpy((unsigned char*)dst + (size_t)(q * Cout + co) * p.swb + at,
                           (const unsigned char*)w + (((size_t)co * Kh + ky) * Kw + kx) * Cin * es, (size_t)Cin * es);
                }
}

int win_encode_weights(const WinPlan& p, int dtype, const void* d_w, void* map_out)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return -1;
    const int es = dtype == 1 ? 2 : 1;
    cuuint64_t dims[2] = {(cuuint64_t)(p.swb / es), (cuuint64_t)p.N};
    cuuint64_t strides[1] = {(cuuint64_t)p.swb};
    cuuint32_t box[2] = {(cuuint32_t)(p.swb / es), (cuuint32_t)p.N};
    cuuint32_t est[2] = {1, 1};
    CUresult r = enc((CUtensorMap*)map_out, dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 2,
                     const_cast<void*>(d_w), dims, strides, box, est, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(p.swb),
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

// cudaErrorNotSupported: the launch cannot take this path (output buffer not 16-byte aligned).
cudaError_t launch_conv_win(const ConvArgs& a, const WinPlan& p, int dtype, const void* w_map, int count_events, cudaStream_t st)
{
    if (!p.ok || a.pool_fused || a.o_end <= a.o_begin) return cudaErrorNotSupported;
    if (((uintptr_t)a.out & 15) != 0) return cudaErrorNotSupported;
    WinArgs t{};
    t.in = a.in; t.bias = a.bias; t.ring = a.ring; t.ring_in = a.ring; t.out = a.out; t.status = a.status;
    t.events = count_events ? a.event_counter : nullptr;
    t.clear = count_events;
    t.out_row_stride = a.out_row_stride; t.out_stream_stride = a.out_stream_stride;
    t.out_row_first = a.o_begin - a.out_row_base;
    t.n_in = (int)(a.r1 - a.r0); t.n_rows = (int)(a.o_end - a.o_begin); t.done_rel = (int)(a.done_end - a.o_begin);
    t.base_ty = (int)(a.r0 + a.pad - a.o_begin * a.stride); t.carried = a.r0 > 0;
    t.ring_slot0 = (int)(a.o_begin % a.ring_rows); t.ring_rows = a.ring_rows;
    t.S = a.S; t.Win = a.Win; t.Wout = a.Wout; t.Cin = a.Cin; t.Cout = a.Cout; t.Kh = a.Kh; t.Kw = a.Kw; t.stride = a.stride;
    t.stride_x = a.stride_x; t.pad_x = a.pad_x; t.relu = a.relu; t.shift = a.shift; t.out_elem = a.out_elem;
    t.P = p.P; t.nxw = p.nxw; t.run_words = p.run_words; t.swb = p.swb; t.ksteps = p.ksteps; t.N = p.N;
    t.inv_c16 = (65536u + a.Cout / 16 - 1) / (a.Cout / 16);
    t.out_wide = ((uintptr_t)a.out & 31) == 0 && (dtype == 1 || a.Cout % 32 == 0);
    if ((long long)a.S * p.nxw > 0x3fffffffLL) return cudaErrorNotSupported;
    t.ncol = a.S * p.nxw;
    t.n_tiles = (t.ncol + 127) / 128;
    t.in_elems = a.in_elems; t.out_elems = a.out_elems; t.ring_elems = a.ring_elems;
    // rows [c0, c1) exchange nothing with the ring
    int c0 = 0, c1 = t.done_rel;
    if (t.carried) while (c0 < t.n_rows && c0 * t.stride < t.base_ty) ++c0;
    if (c1 < c0) c1 = c0;
    const int rows_per_step = p.one_d ? p.P : 1;
    t.n_steps = (t.n_rows + rows_per_step - 1) / rows_per_step;
    t.e0_end = (c0 + rows_per_step - 1) / rows_per_step;
    t.e1_begin = c1 == t.n_rows && c1 % rows_per_step == 0 ? t.n_steps : c1 / rows_per_step;
    if (t.e1_begin < t.e0_end) t.e0_end = t.e1_begin = t.n_steps;                   // every step exchanges rows with the ring
    t.ordered = t.n_rows > t.ring_rows && (t.e0_end > 0 || t.e1_begin < t.n_steps);
    // An ordered item takes its steps one after the other, 4-5 us each where outputs have many channels.  Where that is what the launch
    // waits for, the carried rows are read from a copy of the ring instead, and every step is an item of its own (the copy is a launch of
    // 2-3 us).  1D steps are runs of P rows that share ring slots all over, two of them pay; 2D steps are rows, three: 450 thin layers, mean
    // time against never copying 0.93 (1D 16 -> 128 k2, 152 streams in fives: 7.4 -> 2.9 ms; 1 -> 96 k3, 231 streams in 17s: 2.2 -> 0.96;
    // audio1d frames 1.302 -> 1.238, 5 vgg2d streams in 29s 0.487 -> 0.476).  Above 2000 steps the copy is the longer part.
    const int n_exchange = t.e0_end + (t.n_steps - t.e1_begin);
    if (t.ordered && !t.clear && a.ring_scratch && n_exchange >= (p.one_d ? 2 : 3) && (long long)t.n_steps * t.n_tiles <= 2000) {
        if (t.carried) {
            cudaError_t ce = launch_ring_copy(a.ring_scratch, a.ring, (long long)a.ring_rows * a.S * a.Wout * a.Cout, st);
            if (ce != cudaSuccess) return ce;
            t.ring_in = a.ring_scratch;
        }
        t.ordered = 0;
    }
    // steps per work item: about four items per CTA, at most 16 (neighbouring rows share their input through the L1)
    const int n_free = t.ordered ? t.e1_begin - t.e0_end : t.n_steps;
    const long long R = (long long)n_free * t.n_tiles / (148 * 4);
    t.R = (int)(R < 1 ? 1 : (R > 16 ? 16 : R));
    long long n_items = (long long)(t.ordered + (n_free + t.R - 1) / t.R) * t.n_tiles;
    // A launch of few items (a row pushed at a time: three visited rows, all of them exchanged with the ring, whose 64-byte pieces are
    // what takes the time) spreads an item's columns over several CTAs, which build the same windows, until every SM has an item
    // (3 -> 64 bf16, 64 streams of 224-wide rows pushed one by one, 84 items: 14.1 us whole, 10.5 in two parts, 11.2 in four).
    t.parts = 1;
    while (!t.ordered && t.R == 1 && p.N % (64 * t.parts) == 0 && n_items * t.parts < 148) t.parts *= 2;
    t.part_cols = p.N / t.parts;
    n_items *= t.parts;
    if (n_items > 0x3fffffffLL) return cudaErrorNotSupported;
    t.n_items = (int)n_items;
    typedef void (*KernelFn)(const CUtensorMap, const WinArgs);
    static const KernelFn kernels[2][5] = {
        {conv_win_kernel<1, 0, 0>, conv_win_kernel<1, 1, 0>, conv_win_kernel<1, 0, 2>, conv_win_kernel<1, 0, 5>, conv_win_kernel<1, 0, 9>},
        {conv_win_kernel<2, 0, 0>, conv_win_kernel<2, 1, 0>, conv_win_kernel<2, 0, 2>, conv_win_kernel<2, 0, 5>, conv_win_kernel<2, 0, 9>}};
    int k = p.one_d ? 1 : 0;
    if (!p.one_d && a.Kh == 3) k = p.run_words == 2 ? 2 : (p.run_words == 5 ? 3 : (p.run_words == 9 ? 4 : 0));
    const KernelFn fn = kernels[dtype - 1][k];
    static bool attr_set[2][5][64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dtype - 1][k][dev]) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 1024 + 256 * 128 + WIN_STAGES * 128 * 128);
        if (e != cudaSuccess) return e;
        attr_set[dtype - 1][k][dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(t.n_items < 148 ? t.n_items : 148)); cfg.blockDim = dim3(WIN_THREADS); cfg.dynamicSmemBytes = p.smem_bytes; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = (debug_flags() & IDF_DEBUG_NO_PDL) ? 0 : 1;
    cudaError_t le = cudaLaunchKernelEx(&cfg, fn, *(const CUtensorMap*)w_map, t);
    if (le != cudaSuccess) return le;
    return cudaGetLastError();
}

}  // namespace idf
