// Tensor-core path of the dense Δ-row update (Eq. 4 for a whole row of events at once) with the
// row finalisation (Eq. 2-3) as its epilogue, for bf16 (fp32 state) and int8 (int32 state) nets.
//
// One CTA owns a tile of 128 (stream, x) positions times Ntile output channels of one conv layer
// and walks the block's input rows in order.  While it does so the layer's ring rows for that tile
// live in tensor memory: every ring row is a TMEM accumulator of Ntile columns, and input row r adds
// its contribution to the accumulator of every output row it reaches, one tcgen05.mma per kernel tap
// (ky, kx) and 32-byte K step:   C_o[m, n] += sum_ci  Δ_r[m shifted by kx, ci] * W[ky][kx][n][ci].
//   - the CTA's weight slice (all taps, Ntile channels) is fetched once by TMA and stays in shared
//     memory (weight-stationary);
//   - Δ-rows stream through a ring of shared-memory stages, one TMA box per (input row, kx, K block);
//     the kx shift and the zero padding in x come from the box's start coordinate (out-of-range
//     coordinates read zeros);
//   - an accumulator starts from what its row has so far: zero, or, for a row begun by an earlier
//     block, the partial sums that block left in the ring in global memory (copied in at the start
//     of the launch);
//   - when an input row was the last one an output row was waiting for, the epilogue warps read that
//     accumulator, add the bias, apply f, round or requantise, and write the row for the next layer;
//     rows still open at the end of the block go back to the ring in global memory.
// Warp roles: warp 0 = TMA producer and row scheduler, warp 1 = TMEM owner and MMA issuer,
// warps 2.. = epilogue groups of four warps (one warp per TMEM lane quarter) that take output rows in turn.
// Every wait is bounded; on expiry the kernel records IDF_ERR_TIMEOUT in the status word and leaves.
#include "../../include/idf.h"
#include "idf_ptx.h"

#include <cstdlib>

namespace idf {

namespace {

// Two builds of the kernel: one CTA per SM with three epilogue groups (four warps each, taking output rows in turn), and a light
// one with two groups, half the shared and tensor memory and at most 102 registers, of which an SM holds two.  tc_make_plan says
// which layers take it and what it measured.
constexpr int FULL_GROUPS = 3, LIGHT_GROUPS = 2;
constexpr int tc_threads(int groups) { return 64 + 128 * groups; }
constexpr int tc_rowq(int groups) { return groups == FULL_GROUPS ? 64 : 32; }      // row-schedule queue: two chunks
constexpr size_t LIGHT_SMEM = 113408;        // dynamic shared memory of a light CTA: half an SM less the static part

// Where an emitted row goes first: a shared-memory tile [tile row][panel of pwb bytes], written in
// the swizzle the output tensor map expects, from which one thread sends it out with a TMA store.
struct StageSink {
    uint32_t row_base;     // shared address of this thread's tile row in panel 0
    uint32_t panel_bytes;  // bytes of one panel (staged rows * pwb)
    uint32_t pwb_log2;     // log2(panel row bytes)
    uint32_t phase;        // swizzle phase of this row (XORed into the 16-byte chunk index)
};
__device__ __forceinline__ uint32_t stage_at(const StageSink& k, uint32_t col_byte)
{
    const uint32_t panel = col_byte >> k.pwb_log2;
    const uint32_t within = col_byte & ((1u << k.pwb_log2) - 1u);
    return k.row_base + panel * k.panel_bytes + ((((within >> 4) ^ k.phase)) << 4) + (within & 15u);
}
// V (2 or 4) words, in one access
template <int V>
__device__ __forceinline__ void stage_store(const StageSink& k, uint32_t col_byte, const uint32_t* v)
{
    const uint32_t addr = stage_at(k, col_byte);
    if (V == 4) asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v[0]), "r"(v[1]), "r"(v[V - 2]), "r"(v[V - 1]) : "memory");
    else asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(v[0]), "r"(v[1]) : "memory");
}
template <int V>
__device__ __forceinline__ void stage_load(const StageSink& k, uint32_t col_byte, uint32_t* v)
{
    const uint32_t addr = stage_at(k, col_byte);
    if (V == 4) asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(addr) : "memory");
    else asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(addr) : "memory");
}
// 2x2 max-pooling folded into the emission of a conv layer's rows.  A thread owns one (stream, x)
// position; its x neighbour is the next lane.  The x-pooled first row of a pair waits in the group's
// staging tile (or, across launches, in the pool layer's state in global memory) until the second
// row arrives; the pooled row then leaves through the TMA store.
struct PoolCtx {
    int on;            // pooling is folded into this launch
    int writer;        // this thread holds half the channels of an in-tile pooled position
    int second;        // the row at hand is the second of its pair
    int from_state;    // ... and the first one was emitted by an earlier launch
    int to_state;      // the row at hand is a first row whose partner comes with a later launch
    int drop;          // a first row at the end of input: never completed, nothing is kept
    StageSink sink;    // pooled tile (half the positions)
    unsigned char* state;   // this thread's pooled position in the pool layer's state, at the CTA's first channel
};
template <int NW, int OP>
__device__ __forceinline__ void deliver(uint32_t (&ow)[NW], const StageSink& sink, uint32_t col_byte, const PoolCtx& pc, bool state_ok)
{
    if (!pc.on) {
#pragma unroll
        for (int j4 = 0; j4 < NW / 4; ++j4)
            stage_store<4>(sink, col_byte + 16u * j4, ow + 4 * j4);
        return;
    }
    // The two lanes of a pair share the channels: each sends half of its words, takes the maximum over the other half and carries those
    // on (int8 64 -> 64 with pool, 2048 streams of 126-wide rows, 64 rows: 0.780 ms with both lanes taking all of them, 0.748 so).
    constexpr int H = NW / 2;
    const bool odd = threadIdx.x & 1;
    uint32_t m[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
        const uint32_t other = __shfl_xor_sync(0xffffffffu, odd ? ow[j] : ow[H + j], 1);
        m[j] = word_max<OP>(odd ? ow[H + j] : ow[j], other);
    }
    if (!pc.writer || pc.drop) return;
    if (odd) col_byte += 4u * H;
    constexpr int V = H < 4 ? H : 4;                       // words at a time
#pragma unroll
    for (int j = 0; j < H; j += V) {
        const uint32_t col = col_byte + 4u * j;
        uint32_t h[4];
        if (pc.second) {
            if (!pc.from_state) {
                stage_load<V>(pc.sink, col, h);
            } else {
#pragma unroll
                for (int u = 0; u < V; ++u) h[u] = 0u;
                if (state_ok) {
                    if (V == 4) { const uint4 g = *(const uint4*)(pc.state + col); h[0] = g.x; h[1] = g.y; h[2] = g.z; h[3] = g.w; }
                    else { const uint2 g = *(const uint2*)(pc.state + col); h[0] = g.x; h[1] = g.y; }
                }
            }
#pragma unroll
            for (int u = 0; u < V; ++u) m[j + u] = word_max<OP>(m[j + u], h[u]);
        }
        if (!pc.to_state) {
            stage_store<V>(pc.sink, col, m + j);
        } else if (state_ok) {
            if (V == 4) *(uint4*)(pc.state + col) = make_uint4(m[j], m[j + 1], m[j + V - 2], m[j + V - 1]);
            else *(uint2*)(pc.state + col) = make_uint2(m[j], m[j + 1]);
        }
    }
}
// Row finalisation of W accumulator columns of one (stream, x) position: add what earlier blocks
// left in the ring, then either park the sum in the ring (row still open) or emit f(c + b) in the
// layer's output type.
template <int DT, int W, typename TS>
__device__ __forceinline__ void finalise_chunk(const uint32_t (&v)[W], bool emit, TS* rp,
                                               const TS* bias_c, const StageSink& sink, uint32_t col_byte, int out_elem,
                                               int relu, int shift, const PoolCtx& pc, bool state_ok)
{
    if (!emit) {
#pragma unroll
        for (int j8 = 0; j8 < W / 8; ++j8) st_global_v8(rp + 8 * j8, *(const uint32_t(*)[8])(v + 8 * j8));
        return;
    }
    if (DT == 1) {
        float f[W];
#pragma unroll
        for (int j = 0; j < W; ++j) f[j] = __uint_as_float(v[j]);
        if (bias_c) {
#pragma unroll
            for (int j4 = 0; j4 < W / 4; ++j4) {
                const float4 b4 = ((const float4*)bias_c)[j4];
                f[4 * j4] += b4.x; f[4 * j4 + 1] += b4.y; f[4 * j4 + 2] += b4.z; f[4 * j4 + 3] += b4.w;
            }
        }
        if (out_elem == E_BF16) {
            // two values per instruction: round to nearest even, with the ReLU folded into the conversion
            uint32_t pk[W / 2];
            if (relu) {
#pragma unroll
                for (int j = 0; j < W / 2; ++j)
                    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(f[2 * j + 1]), "f"(f[2 * j]));
            } else {
#pragma unroll
                for (int j = 0; j < W / 2; ++j)
                    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(f[2 * j + 1]), "f"(f[2 * j]));
            }
            deliver<W / 2, 0>(pk, sink, col_byte, pc, state_ok);
        } else {
            if (relu) {
#pragma unroll
                for (int j = 0; j < W; ++j) f[j] = fmaxf(f[j], 0.f);
            }
            uint32_t fw[W];
#pragma unroll
            for (int j = 0; j < W; ++j) fw[j] = __float_as_uint(f[j]);
            deliver<W, 1>(fw, sink, col_byte, pc, state_ok);
        }
    } else {
        uint32_t pk[W / 4];
        pack_i8<W>(v, (const int*)bias_c, relu, shift, pk);
        deliver<W / 4, 2>(pk, sink, col_byte, pc, state_ok);
    }
}

struct TcArgs {
    const void* bias;
    void* ring;
    const void* ring_in;         // where the rows begun by earlier blocks are read: the ring, or a copy of it made before a
                                 // launch whose row chunks run in CTAs of their own (one parks rows while another still reads)
    void* out;
    unsigned int* status;
    long long out_row_stride, out_stream_stride, out_row_base;
    long long o_begin;           // absolute index of the first visited output row
    int r0_positive;             // input rows arrived before this block (r0 > 0)
    int n_rows;                  // input rows in this block
    int n_orows;                 // visited output rows: o_begin + [0, n_orows)
    int done_rel;                // rows with relative index < done_rel are emitted, the others go back to the ring
    int sched_rel;               // rows below it are completed by an input row of this block; rows in [sched_rel, done_rel)
                                 // wait only for bottom padding and are completed by the block's last row (end of input)
    int base_ty;                 // r0 + pad - o_begin*stride: input row ri reaches relative output row
                                 // (base_ty + ri - ky) / stride through tap ky when that is a whole number >= 0
    int S, Wout, Cout, Kh, Kw, stride, pad_x, relu, shift, ring_rows, out_elem;
    int BX, BXP, BS, n_xt, Ntile, n_nt, KB, n_kb, swb, nslot, nstage, tmem_cols;
    int shift_mode;              // 1: one box per (row, K block) holds the kx halo, taps address it at row offsets
    int pair;                    // 1: A rows are single 16-byte positions, a K step reads two neighbouring ones (see tc_make_plan)
    int sx;                      // x stride of the conv (1, or more when every kx tap has a box of its own: the tensor map then
                                 // walks the input row in steps of sx, so a box still holds BXP consecutive OUTPUT positions)
    int n_chunks, chunk_rows, chunk_shift;   // the block's output rows are cut into n_chunks runs of chunk_rows rows (the first one
                                 // chunk_shift shorter), one CTA each: see the kernel's prologue
    int a_stage_bytes;
    int n_box, a_box_pitch;      // TMA boxes per stage (one per kx tap when the taps cannot share a haloed box) and their distance in bytes
    int out_esize, out_pwb, out_panels, out_stage_bytes;   // emitted rows: staging panels of out_pwb-byte rows
    int out_stage_rows;          // rows of one staging panel: 128, or 64 when only pooled rows are staged
    int out_groups;              // epilogue groups at work, each with its own staging tile(s)
    int out_bufs;                // staging tiles per group (1 or 2, used in turn)
    int out_row_dim;             // position of the row coordinate in the output tensor map (2 or 3)
    int out_row_first;           // tensor-map row index of relative output row 0
    // 2x2 max-pooling folded into the emission (the output tensor map then describes the pooled rows)
    int pool;                    // 1: emit pooled rows
    int pool_keep;               // 1: a trailing first row of a pair waits in pool_state for a later launch; 0: end of input, it is dropped
    void* pool_state;            // [S][Wout/2][Cout] in the output type: x-pooled first row of an open pair
    long long pool_row_base;     // pooled row p goes to tensor-map row p - pool_row_base
    // small pieces of o_begin, so that the row loop needs no 64-bit arithmetic
    int o_begin_par;             // o_begin & 1
    int o_begin_half_mod;        // (o_begin >> 1) mod out_groups
    int ring_slot0;              // o_begin mod ring_rows
    int pool_row_first;          // (o_begin >> 1) - pool_row_base: tensor-map row of the pair that holds o_begin
    long long ring_elems, pool_state_bytes;   // extents of ring (state words) and pool_state (bytes): range-checked build
    unsigned int smem_bytes;     // dynamic shared memory of the launch (range-checked build)
};

// KX3: the common case of 128-byte rows with three kx taps read row-shifted from one haloed box, known at compile time
// (the MMA warp's loop is what the kernel's speed hangs on: every constant it sees helps)
template <int DT, int KSTEPS, int KX3, int GROUPS>
__global__ void __launch_bounds__(tc_threads(GROUPS), GROUPS == FULL_GROUPS ? 1 : 2)
conv_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW,
               const __grid_constant__ CUtensorMap tmO, const TcArgs a)
{
    typedef typename Acc<DT>::S TS;
    constexpr int ROWQ = tc_rowq(GROUPS), CHUNK = ROWQ / 2;
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ int s_issued;
    __shared__ __align__(16) uint32_t s_rowq[ROWQ][16];                // per input row: what the MMA thread must do

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the next kernel may start its own prologue
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int taps = a.Kh * a.Kw;
    const uint32_t w_tile_bytes = (uint32_t)a.Ntile * a.swb;
    const uint32_t a_stage_bytes = (uint32_t)a.a_stage_bytes;
    const uint32_t a_box_bytes = (uint32_t)a.BXP * a.BS * (a.pair ? 16u : (uint32_t)a.swb);
    // (rows of 128 bytes always share one haloed box: for that instantiation the compiler sees the constant)
    const int n_box = KSTEPS == 4 ? 1 : a.n_box;

    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sW = base;
    const uint32_t sA = (sW + (uint32_t)taps * a.n_kb * w_tile_bytes + 1023u) & ~1023u;
    const uint32_t sOut = sA + (uint32_t)a.nstage * a_stage_bytes;               // one staging tile per epilogue group
    const uint32_t bars = sOut + (uint32_t)(a.out_groups * a.out_bufs) * (uint32_t)a.out_stage_bytes;
    const uint32_t bar_full = bars;
    const uint32_t bar_empty = bar_full + 8u * a.nstage;
    const uint32_t bar_w = bar_empty + 8u * a.nstage;
    const uint32_t bar_ready = bar_w + 8u * taps;
    const uint32_t bar_free = bar_ready + 8u * a.nslot;
    const uint32_t bar_start = bar_free + 8u * a.nslot;    // every slot the launch uses holds what its first row starts from

    const int nt = blockIdx.x % a.n_nt;
    const int mt_all = blockIdx.x / a.n_nt;
    const int n_mt_all = a.n_xt * ((a.S + a.BS - 1) / a.BS);
    const int mt = mt_all % n_mt_all;
    // Row chunks.  When a layer has few (position, channel) tiles, the block's output rows are cut into runs and
    // every run gets CTAs of its own: a run needs only the input rows its output rows reach, which it reads again
    // at its edges instead of taking partial sums from its neighbour.  Inside a chunk everything is as in a block
    // that starts at the chunk's first output row: taps into rows of other chunks drop out, only the first chunk
    // takes up the ring, only the last one parks rows in it.
    const int chunk = mt_all / n_mt_all;
    const int c_oa = chunk == 0 ? 0 : chunk * a.chunk_rows - a.chunk_shift;                       // first relative output row
    const int c_ob = chunk == a.n_chunks - 1 ? a.n_orows : (chunk + 1) * a.chunk_rows - a.chunk_shift;
    int c_ra = c_oa * a.stride - a.base_ty;                                                        // first input row that reaches it
    if (c_ra < 0) c_ra = 0;
    int c_rb = (c_ob - 1) * a.stride - a.base_ty + a.Kh;                                           // one past the last
    if (c_rb > a.n_rows || chunk == a.n_chunks - 1) c_rb = a.n_rows;
    const int c_base_ty = a.base_ty + c_ra - c_oa * a.stride;
    const int c_n_orows = c_ob - c_oa;
    const int c_done_rel = min(max(a.done_rel - c_oa, 0), c_n_orows);
    const int c_sched_rel = min(max(a.sched_rel - c_oa, 0), c_n_orows);
    const bool c_r0_positive = a.r0_positive && chunk == 0;
    const int xt = mt % a.n_xt, stile = mt / a.n_xt;
    const int x0 = xt * a.BX, s0 = stile * a.BS, n0 = nt * a.Ntile;

    if (threadIdx.x == 0) {
        s_abort = 0;
        s_issued = 0;
        if (!IDF_OK_AT(a.status, (bar_start - smem_u32(smem_raw)) + 7, a.smem_bytes)) s_abort = 1;
        // The weights come first: they do not depend on earlier kernels of the stream (their fetch overlaps the
        // previous kernel's tail under programmatic dependent launch), and a launch that brings a single row has
        // little else to hide their latency behind.  One copy per K block carries all taps of the CTA's channel
        // slice (the parameters are stored tap by tap in the order the stacked tiles want, see tc_weight_slot).
        mbar_init(bar_w, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(bar_w, (uint32_t)(taps * a.n_kb) * w_tile_bytes);
        for (int kb = 0; kb < a.n_kb; ++kb)
            tma_load_3d(sW + (uint32_t)(kb * taps) * w_tile_bytes, &tmW, bar_w, kb * a.KB, n0, 0);
    }
    // (one barrier to a lane: one thread initialising them all takes longer than everything else up to here)
    if (warp == 2) {
        if (lane < a.nstage) { mbar_init(bar_full + 8u * lane, 1); mbar_init(bar_empty + 8u * lane, 1); }
        if (lane < a.nslot) { mbar_init(bar_ready + 8u * lane, 1); mbar_init(bar_free + 8u * lane, 4); }
        if (lane == 31) mbar_init(bar_start, 4 * GROUPS);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // everything below reads or writes buffers that earlier kernels of the stream produce or consume
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const uint32_t tmem_base = s_tmem_base;
    volatile int* abort_flag = &s_abort;
    const int n_rows = c_rb - c_ra;

    if (warp == 0) {
        // ------------------------------ TMA producer + row scheduler ---------------------------
        // One thread issues every MMA and the tensor pipe runs only a couple of instructions ahead
        // of it, so that thread must do as little else as possible.  This thread, which mostly waits
        // for free stages, therefore also works out for every input row which accumulators it feeds
        // and leaves the answer in a small queue next to the data (published by the stage's barrier).
        // With t0 = base_ty + ri the taps of input row ri are ky = ph, ph+s, ... (ph = t0 mod s), and
        // tap ky = ph + j*s reaches relative output row hi - j (hi = t0 div s).
        // The 32 lanes work out the schedule of 32 rows at a time (one row each, closed form), then
        // lane 0 issues those rows' copies.
        const uint32_t idesc0 = (DT == 1 ? ((1u << 4) | (1u << 7) | (1u << 10)) : ((2u << 4) | (1u << 7) | (1u << 10))) |
                                ((128u >> 4) << 24);
        const int max_rows = 256 / a.Ntile;              // ring rows one instruction can cover (N <= 256)
        const int s = a.stride, nslot = a.nslot;
        int stage = 0, t = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (int r_chunk = 0; r_chunk < n_rows && ok; r_chunk += CHUNK) {
            {
                const int ri = r_chunk + lane;
                if (lane < CHUNK && ri < n_rows) {
                    uint32_t* q = s_rowq[ri & (ROWQ - 1)];
                    const int t0 = c_base_ty + ri;
                    const int hi = t0 / s, ph = t0 - hi * s;
                    const int slot_hi = hi % nslot, u_hi = hi / nslot;
                    // a new output row starts when ph == 0: its slot's previous row must have been read out
                    const bool fresh = (ri > 0 && ph == 0 && hi >= nslot && hi < c_n_orows);
                    q[0] = fresh ? bar_free + 8u * (uint32_t)slot_hi : 0u;
                    q[1] = (uint32_t)((u_hi & 1) ^ 1);              // phase u_hi - 1 of the slot: its row before this one has left
                    // the row completed by input row ri is (t0 - (Kh-1)) / s when that is a whole number >= 0
                    const int tf = t0 - (a.Kh - 1);
                    const int of = tf >= 0 ? tf / s : -1;
                    q[3] = (tf >= 0 && of * s == tf && of < c_sched_rel) ? bar_ready + 8u * (uint32_t)(of % nslot) : 0u;
                    // taps ky = ph, ph+s, ... < Kh; those that would reach rows above the map drop out
                    const int cnt = (a.Kh - ph + s - 1) / s;
                    int n_t = cnt;
                    if (n_t > hi + 1) n_t = hi + 1;
                    int sl = (slot_hi - (n_t - 1)) % nslot;
                    if (sl < 0) sl += nslot;
                    int poff = 0;
                    for (int p = 0; p < ph; ++p) poff += (a.Kh - p + s - 1) / s;
                    uint32_t blk = (uint32_t)(poff + cnt - n_t);
                    // ... and so do those that reach rows beyond this chunk (the highest rows = the first taps)
                    if (hi > c_n_orows - 1) n_t -= hi - (c_n_orows - 1);
                    // segments: runs of rows whose slots are consecutive TMEM column blocks (N <= 256 each)
                    int n_seg = 0;
                    for (int rem = n_t; rem > 0 && n_seg < 4; ++n_seg) {
                        int len = rem;
                        if (len > nslot - sl) len = nslot - sl;
                        if (len > max_rows) len = max_rows;
                        q[4 + 3 * n_seg] = tmem_base + (uint32_t)(sl * a.Ntile);
                        q[5 + 3 * n_seg] = (blk * w_tile_bytes) >> 4;
                        q[6 + 3 * n_seg] = idesc0 | ((uint32_t)((len * a.Ntile) >> 3) << 17);
                        rem -= len; blk += (uint32_t)len; sl += len;
                        if (sl == nslot) sl = 0;
                    }
                    q[2] = (uint32_t)n_seg;
                }
            }
            __syncwarp();
            if (lane == 0) {
                const int r_end = r_chunk + CHUNK < n_rows ? r_chunk + CHUNK : n_rows;
                for (int ri = r_chunk; ri < r_end && ok; ++ri) {
                    // A row that starts a new output row needs that row's slot read out and cleared.  Waiting
                    // here, before the row's first copy, means the MMA thread learns it from the copy's
                    // barrier and has one barrier less to look at.
                    const uint32_t* qr = s_rowq[ri & (ROWQ - 1)];
                    if (qr[0] && !mbar_wait(qr[0], qr[1], abort_flag)) { ok = false; break; }
                    // one stage per (row, K block): the haloed box all kx taps share, or one box per kx tap side by side
                    for (int kb = 0; kb < a.n_kb; ++kb) {
                        if (!mbar_wait(bar_empty + 8u * stage, phase ^ 1u, abort_flag)) { ok = false; break; }
                        if (!IDF_OK_AT(a.status, (sA - smem_u32(smem_raw)) + (uint32_t)stage * a_stage_bytes + (uint32_t)(n_box - 1) * a.a_box_pitch + a_box_bytes - 1,
                                       bars - smem_u32(smem_raw))) { ok = false; break; }
                        mbar_expect_tx(bar_full + 8u * stage, (uint32_t)n_box * a_box_bytes);
                        for (int xl = 0; xl < n_box; ++xl)
                            tma_load_4d(sA + (uint32_t)stage * a_stage_bytes + (uint32_t)xl * a.a_box_pitch, &tmA, bar_full + 8u * stage,
                                        a.pair ? 2 * (x0 - a.pad_x) : kb * a.KB, a.pair ? 0 : x0 * a.sx - a.pad_x + xl, s0, c_ra + ri);
                        ++t;
                        if (++stage == a.nstage) { stage = 0; phase ^= 1u; }
                    }
                }
            }
            ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
        }
        if (lane == 0) s_issued = t;     // copies in flight, for the clean-up after a failed wait
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ---------------------------------------------
        // The whole warp runs this loop in step (every value in it is the same in all lanes) and one
        // elected lane issues the tensor-core instructions.  The tensor pipe runs only a few instructions
        // behind the issuing lane, so every cycle spent here on anything but issuing is a cycle the pipe
        // idles.  Hence: the barrier of the NEXT tile is looked at (non-blocking) before the current
        // tile's MMAs are issued and the answer is read after them, the next row's schedule entry is
        // fetched the same way, and the wait for a free accumulator slot is the producer's (a tile of a
        // row only arrives once its slot is free).
        {
            const uint64_t desc_hi = make_smem_desc(0, a.swb);
            const int n_kx = KX3 ? 3 : (a.shift_mode ? a.Kw : n_box);   // kx taps of a stage: row-shifted reads of one box, or one box each
            const int nslot = a.nslot;
            const uint32_t kx_bytes = a.pair ? 2u : ((KSTEPS == 4 || a.shift_mode) ? (uint32_t)a.swb >> 4 : (uint32_t)a.a_box_pitch >> 4);
            // weight tiles in shared memory: [K block][kx][stacked ky block]
            const uint32_t wtile_kx = ((uint32_t)a.Kh * w_tile_bytes) >> 4;              // descriptor units per kx
            const uint32_t wtile_kb = ((uint32_t)taps * w_tile_bytes) >> 4;
            const uint32_t a_stage_units = a_stage_bytes >> 4;
            const int nstage = a.nstage, n_kb = a.n_kb;
            bool ok = true;
            // Every slot holds what its first row starts from.  This is a barrier of its own, not the slots' first free phase: the
            // producer may be a slot's whole turn ahead, and a parity would not tell it that phase from the one it needs.
            ok = mbar_wait(bar_start, 0, abort_flag);
            ok = ok && mbar_wait(bar_w, 0, abort_flag);          // the CTA's weight slice has landed
            // (paired positions: no swizzle, 8 rows of 16 bytes are 128 bytes, and the second half of a K step is the next position)
            const uint64_t adesc_base = (a.pair ? ((uint64_t)1 << 16) | ((uint64_t)8 << 32) | ((uint64_t)1 << 46) : desc_hi) | (uint64_t)((sA & 0x3FFFFu) >> 4);
            const uint64_t bdesc_base = desc_hi | (uint64_t)((sW & 0x3FFFFu) >> 4);
            const int n_st = n_kb;                               // tiles (stages) per input row
            const bool issuer = elect_one();                     // the lane that issues (the warp stays converged)
            ok = ok && mbar_wait(bar_full, 0, abort_flag);       // first tile of the first row
            tc_fence_after();
            uint4 hdr = make_uint4(0, 0, 0, 0), sa = hdr, sb = hdr, sc = hdr;
            if (ok) {
                const uint4* q = (const uint4*)s_rowq[0];
                hdr = q[0]; sa = q[1]; sb = q[2]; sc = q[3];
            }
            // The loop runs over tiles (input row, kx box, K block), software-pipelined by hand: everything the NEXT
            // tile needs (stage, barrier, descriptors, and on a row's last tile the next row's schedule entry) is worked
            // out between the first and the last MMA group of the CURRENT tile, while the pipe is busy, so that between
            // the last MMA of one tile and the first MMA of the next there is only the commit and a handful of moves.
            // tap kx reads the same tile kxi rows further down: the swizzle is a function of the absolute
            // shared-memory address, so a start address moved by whole rows still meets the pattern the TMA
            // wrote (base-offset field stays 0).
            int ri = 0, st = 0, kb = 0, stage = 0;
            uint32_t phase = 0;
            uint64_t adesc_cur = adesc_base, bdesc_cur = bdesc_base;       // the tile at hand
            const long long n_tiles = (long long)n_rows * n_st;
            for (long long tile = 0; tile < n_tiles && ok; ++tile) {
                const bool row_end = st == n_st - 1;
                const bool last_row = ri == n_rows - 1;
                // ---- first MMA group of the tile
                if (issuer && hdr.z > 0) {
                    umma_tile<DT, KSTEPS>(sa.x, adesc_cur, bdesc_cur + (uint64_t)sa.y, sa.z);
                    if (hdr.z > 1) {
                        umma_tile<DT, KSTEPS>(sa.w, adesc_cur, bdesc_cur + (uint64_t)sb.x, sb.y);
                        if (hdr.z > 2) umma_tile<DT, KSTEPS>(sb.z, adesc_cur, bdesc_cur + (uint64_t)sb.w, sc.x);
                        if (hdr.z > 3) umma_tile<DT, KSTEPS>(sc.y, adesc_cur, bdesc_cur + (uint64_t)sc.z, sc.w);
                    }
                }
                // ---- the next tile, worked out while those run
                int n_stage = stage + 1;
                uint32_t n_phase = phase;
                uint64_t adesc_nx = adesc_cur + a_stage_units;
                if (n_stage == nstage) { n_stage = 0; n_phase ^= 1u; adesc_nx = adesc_base; }
                uint64_t bdesc_nx = bdesc_cur + wtile_kb;
                int n_kbi = kb + 1;
                if (n_kbi == n_kb) { n_kbi = 0; bdesc_nx = bdesc_base; }
                uint32_t next_ok = 1u;
                if (!(last_row && row_end)) next_ok = mbar_test(bar_full + 8u * n_stage, n_phase);
                uint4 nh = hdr, na = sa, nb = sb, nc = sc;
                // schedule entries are published a chunk of rows at a time, ahead of the first copy of those rows
                const bool early_info = row_end && !last_row && ((ri + 1) & (CHUNK - 1)) != 0;
                const uint4* qn = (const uint4*)s_rowq[(ri + 1) & (ROWQ - 1)];
                if (early_info) { nh = qn[0]; na = qn[1]; nb = qn[2]; nc = qn[3]; }
                // ---- the other kx taps of the tile (row-shifted reads of the same box)
                {
                    uint64_t adesc = adesc_cur + kx_bytes, bdesc = bdesc_cur + wtile_kx;
                    for (int kxi = 1; kxi < n_kx; ++kxi, adesc += kx_bytes, bdesc += wtile_kx) {
                        if (issuer && hdr.z > 0) {
                            umma_tile<DT, KSTEPS>(sa.x, adesc, bdesc + (uint64_t)sa.y, sa.z);
                            if (hdr.z > 1) {
                                umma_tile<DT, KSTEPS>(sa.w, adesc, bdesc + (uint64_t)sb.x, sb.y);
                                if (hdr.z > 2) umma_tile<DT, KSTEPS>(sb.z, adesc, bdesc + (uint64_t)sb.w, sc.x);
                                if (hdr.z > 3) umma_tile<DT, KSTEPS>(sc.y, adesc, bdesc + (uint64_t)sc.z, sc.w);
                            }
                        }
                    }
                }
                if (issuer) {
                    umma_commit(bar_empty + 8u * stage);
                    if (row_end) {
                        // the accumulator this input row completed; on the block's last row also everything still open
                        // (to be parked in the ring, or emitted if only bottom padding was missing)
                        if (hdr.w) umma_commit(hdr.w);
                        if (last_row)
                            for (int orel = c_sched_rel; orel < c_n_orows; ++orel) umma_commit(bar_ready + 8u * (uint32_t)(orel % nslot));
                    }
                }
                if (!next_ok && !mbar_wait(bar_full + 8u * n_stage, n_phase, abort_flag)) { ok = false; break; }
                stage = n_stage; phase = n_phase; adesc_cur = adesc_nx; bdesc_cur = bdesc_nx; kb = n_kbi;
                if (row_end) {
                    if (last_row) break;
                    if (!early_info) { nh = qn[0]; na = qn[1]; nb = qn[2]; nc = qn[3]; }   // (published with the tile just waited for)
                    hdr = nh; sa = na; sb = nb; sc = nc;
                    st = 0; ++ri;
                    tc_fence_after();                            // the next row may start on a slot the epilogue has just cleared
                } else {
                    ++st;
                }
            }
        }
        __syncwarp();
    } else {
        // ------------------------------ epilogue: row finalisation -----------------------------
        // Groups of four warps (one warp per TMEM lane quarter) take the output rows in turn.
        // An emitted row is first laid out in the group's shared-memory tile (each thread writes its
        // own tile row, swizzled), then one thread hands the tile to a TMA store, which writes whole
        // lines and clips whatever lies outside the map.
        const int q = warp & 3;                          // TMEM lane quarter this warp may read
        const int grp = (warp - 2) >> 2;
        const bool leader = (warp - 2) == grp * 4 && lane == 0;
        const int m = q * 32 + lane;                     // row of the tile = TMEM lane
        const int bs = m / a.BXP, bx = m - bs * a.BXP;
        const int s = s0 + bs, x = x0 + bx;
        const bool in_tile = (bs < a.BS) && (bx < a.BX);
        const bool valid = in_tile && (s < a.S) && (x < a.Wout);
        const bool wide = GROUPS == FULL_GROUPS && (a.Ntile & 31) == 0;     // (32 columns at a time take more registers than the light build has)
        const TS* bias = a.bias ? (const TS*)a.bias + n0 : nullptr;
        const long long row_elems = (long long)a.Wout * a.Cout;
        TS* ring_pos = (TS*)a.ring + (long long)s * row_elems + (long long)x * a.Cout + n0;   // + ring slot * S * row_elems
        const long long ring_slot_stride = (long long)a.S * row_elems;
        const uint32_t tlane = tmem_base + ((uint32_t)(q * 32) << 16);
        const int md = bs * a.BX + bx;                   // row of the dense output tile
        StageSink sink;
        sink.pwb_log2 = 31u - (uint32_t)__clz(a.out_pwb);
        sink.panel_bytes = (uint32_t)a.out_stage_rows * (uint32_t)a.out_pwb;
        sink.row_base = sOut + (uint32_t)(grp * a.out_bufs) * a.out_stage_bytes + (uint32_t)md * a.out_pwb;
        sink.phase = a.out_pwb == 128 ? (uint32_t)(md & 7) : (a.out_pwb == 64 ? (uint32_t)((md >> 1) & 3)
                   : (a.out_pwb == 32 ? (uint32_t)((md >> 2) & 1) : 0u));
        uint32_t stg = sOut + (uint32_t)(grp * a.out_bufs) * a.out_stage_bytes;     // the staging tile in use
        uint32_t buf_step = a.out_bufs > 1 ? (uint32_t)a.out_stage_bytes : 0u;      // to the group's other tile (sign flips per store)
        const int panel_cols = a.out_pwb / a.out_esize;
        PoolCtx pc;
        pc.on = a.pool; pc.second = 0; pc.from_state = 0; pc.to_state = 0; pc.drop = 0;
        pc.writer = in_tile;
        const int mdp = bs * (a.BX >> 1) + (bx >> 1);   // row of the pooled tile
        pc.sink = sink;
        pc.sink.row_base = stg + (uint32_t)mdp * a.out_pwb;
        pc.sink.phase = a.out_pwb == 128 ? (uint32_t)(mdp & 7) : (a.out_pwb == 64 ? (uint32_t)((mdp >> 1) & 3)
                      : (a.out_pwb == 32 ? (uint32_t)((mdp >> 2) & 1) : 0u));
        const int wp = a.Wout >> 1;
        const bool state_ok = valid && (x >> 1) < wp;
        pc.state = (unsigned char*)a.pool_state + (((long long)s * wp + (x >> 1)) * a.Cout + n0) * a.out_esize;
        bool ok = true;
        // Every ring slot in tensor memory starts from what its row has so far (all MMAs accumulate): zero, or, for a
        // row begun by an earlier block, the partial sums that block left in the ring in global memory.  Taking those
        // up here, while weights and the first rows are still on their way, keeps the ring's read latency out of the
        // path between the last MMA and the emission.  A launch that brings one row waits for little else, so the groups share
        // the carried rows by columns and a thread's loads go out together, not one piece of 16 columns after the other.
        {
            constexpr int PIECES = GROUPS == FULL_GROUPS ? 3 : 2;
            const long long carry_off0 = (const TS*)a.ring_in - (const TS*)a.ring;
            const int n_init = c_n_orows < a.nslot ? c_n_orows : a.nslot;
            const int per_slot = 31 - __clz(a.Ntile >> 4);                              // log2 of the pieces of a slot (Ntile is a power of two)
            for (int i0 = grp * PIECES; i0 < n_init << per_slot; i0 += GROUPS * PIECES) {
                uint32_t v[PIECES][16];
#pragma unroll
                for (int u = 0; u < PIECES; ++u) {
                    const int slot = (i0 + u) >> per_slot, c = ((i0 + u) - (slot << per_slot)) * 16;
                    // (slot and carried_row are the same in all threads: the tensor-memory stores below are warp-wide instructions and
                    // every branch around them must be uniform; what differs per thread is only whether it has values to load)
                    const bool carried_row = slot < n_init && c_r0_positive && slot * a.stride - c_base_ty < 0;
                    bool carried = carried_row && valid;
                    const TS* rp = ring_pos + carry_off0 + c;
                    if (carried_row) rp += (long long)((a.ring_slot0 + c_oa + slot) % a.ring_rows) * ring_slot_stride;
#ifdef IDF_BOUNDS
                    if (carried && !IDF_OK_AT(a.status, (rp - carry_off0 - (const TS*)a.ring) + 15, a.ring_elems)) carried = false;
#endif
                    if (carried) {
                        ld_global_v8(rp, *(uint32_t(*)[8])v[u]);
                        ld_global_v8(rp + 8, *(uint32_t(*)[8])(v[u] + 8));
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[u][j] = 0u;
                    }
                }
                __syncwarp();
#pragma unroll
                for (int u = 0; u < PIECES; ++u)
                    if (i0 + u < n_init << per_slot) tmem_st16(tlane + (uint32_t)((i0 + u) << 4), v[u]);
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_start);   // one arrival per warp
        }
        // Rows left open by this block go back to the ring in global memory; those that meet in one ring slot stay in
        // one group, in order.  (Rows begun by an earlier block were read above, before the first MMA, so nothing
        // reads a ring slot any more once rows are written.)  The other rows go round the groups.
        const int n_cin = c_r0_positive ? (c_base_ty + a.stride - 1) / a.stride : 0;
        // Per-row bookkeeping is kept with small counters that step from row to row (a division or a 64-bit
        // operation per row and thread costs more than the row's arithmetic): TMEM slot and barrier parity of the row,
        // its ring slot in global memory, the parity of its absolute index, the group whose turn it is.
        const int G = a.out_groups;
        int slot_c = 0;                                       // orel mod nslot
        uint32_t par_c = 0;                                   // (orel div nslot) & 1
        int turn = 0;                                         // orel mod G
        int absp = (a.o_begin_par + c_oa) & 1;                // parity of the row's absolute index
        int pair_turn = (a.o_begin_half_mod + ((a.o_begin_par + c_oa) >> 1)) % G;   // (absolute index div 2) mod G
        int rslot_c = (a.ring_slot0 + c_oa) % a.ring_rows;    // absolute index mod ring_rows
        int rslot_g = rslot_c % G;                            // ... mod G: the group that owns the ring slot
        for (int orel = 0; orel < c_n_orows && ok && grp < G; ++orel) {
            int owner;
            if (!a.pool) {
                // (rows that meet in one ring slot stay in one group, which takes them in order)
                owner = (orel < n_cin || orel >= c_done_rel) ? rslot_g : turn;
            } else {
                // both rows of a pooling pair go to one group; pairs touching the global ring or the pool layer's state
                // (first < 0: the pair's first row came with an earlier launch) go to group 0
                const int first = orel - absp;
                owner = (first < 0 || first < n_cin || first + 1 >= c_done_rel) ? 0 : pair_turn;
                // a launch that emits at most one row has no pair to keep together and one row at most that touches the
                // pool layer's state: its rows spread over the groups by ring slot as above
                if (c_done_rel <= 1) owner = rslot_g;
            }
            const int slot = slot_c, rslot = rslot_c, row_odd = absp;
            const uint32_t par = par_c;
            // the counters move on to the next row
            if (++slot_c == a.nslot) { slot_c = 0; par_c ^= 1u; }
            if (++turn == G) turn = 0;
            if (++rslot_c == a.ring_rows) rslot_c = 0;
            if (++rslot_g == G) rslot_g = 0;
            if (rslot_c == 0) rslot_g = 0;
            if (absp && ++pair_turn == G) pair_turn = 0;
            absp ^= 1;
            if (owner != grp) continue;
            const bool emit = orel < c_done_rel;
            // one thread of the group polls the barrier; the named barrier below releases the other warps.
            // The tile must have been drained by the group's previous store before anyone writes it again: that
            // wait comes first, it overlaps the wait for the row.
            int got = 1;
            if (leader) {
                // (with two tiles the latest store may still be draining: it reads the other one)
                if (emit) {
                    if (a.out_bufs > 1) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                }
                got = mbar_wait_relaxed(bar_ready + 8u * slot, par, abort_flag) ? 1 : 0;
            }
            // (the barrier also makes the whole group leave together if any of its waits ran out)
            if (!named_bar_and(1 + grp, 128, got != 0)) { ok = false; break; }
            tc_fence_after();
            const bool pool_emit = a.pool && emit;
            if (pool_emit) {
                pc.second = row_odd;
                pc.from_state = pc.second && orel == 0;
                const bool trailing = !pc.second && orel == c_done_rel - 1 && c_oa + c_done_rel == a.done_rel;   // the block's last emitted row
                pc.to_state = trailing && a.pool_keep;
                pc.drop = trailing && !a.pool_keep;
            }
            TS* rp = ring_pos + (long long)rslot * ring_slot_stride;
            const uint32_t trow = tlane + (uint32_t)(slot * a.Ntile);
            bool fine = true;           // range-checked build: false skips this row's accesses (the barriers still run)
#ifdef IDF_BOUNDS
            {
                fine = IDF_OK_AT(a.status, slot * a.Ntile + a.Ntile - 1, a.tmem_cols);
                if (valid && !emit) fine = fine && IDF_OK_AT(a.status, (rp - (TS*)a.ring) + a.Ntile - 1, a.ring_elems);
                if (pool_emit && state_ok && (pc.from_state || pc.to_state))
                    fine = fine && IDF_OK_AT(a.status, (pc.state - (unsigned char*)a.pool_state) + (long long)a.Ntile * a.out_esize - 1, a.pool_state_bytes);
                // (a launch that emits pooled rows stages them in the half-size tile; the full-size addresses are not used then)
                const uint32_t stage_row = a.pool ? pc.sink.row_base : sink.row_base;
                if (emit && (a.pool ? pc.writer != 0 : in_tile))
                    fine = fine && IDF_OK_AT(a.status, (stage_row - smem_u32(smem_raw)) + (uint32_t)(a.out_panels - 1) * sink.panel_bytes + a.out_pwb - 1,
                                             bars - smem_u32(smem_raw));
                fine = __all_sync(0xffffffffu, fine) != 0;     // (the tensor-memory loads below are warp-wide instructions)
            }
#endif
            {
                if (GROUPS == FULL_GROUPS && wide) {
                    for (int c = 0; c < a.Ntile; c += 32) {
                        uint32_t v[32];
                        if (!fine) continue;
                        __syncwarp();                         // (the finalisation of the previous chunk is per thread)
                        tmem_ld<32>(trow + c, v);
                        tmem_st_zero<32>(trow + c);           // the slot's next row starts from zero
                        if (pool_emit || (emit ? in_tile : valid))
                            finalise_chunk<DT, 32, TS>(v, emit, rp + c, bias ? bias + c : nullptr, sink,
                                                       (uint32_t)(c * a.out_esize), a.out_elem, a.relu, a.shift, pc, state_ok);
                    }
                } else {
                    for (int c = 0; c < a.Ntile; c += 16) {
                        uint32_t v[16];
                        if (!fine) continue;
                        __syncwarp();
                        tmem_ld<16>(trow + c, v);
                        tmem_st_zero<16>(trow + c);
                        if (pool_emit || (emit ? in_tile : valid))
                            finalise_chunk<DT, 16, TS>(v, emit, rp + c, bias ? bias + c : nullptr, sink,
                                                       (uint32_t)(c * a.out_esize), a.out_elem, a.relu, a.shift, pc, state_ok);
                    }
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_free + 8u * slot);   // one arrival per warp
            }
            if (emit && (!a.pool || pc.second)) {      // with pooling only the second row of a pair sends a (pooled) row out
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                named_bar_sync(1 + grp, 128);
                if (leader) {
                    const int orow = a.pool ? a.pool_row_first + ((a.o_begin_par + c_oa + orel) >> 1) : a.out_row_first + c_oa + orel;
                    const int xc = a.pool ? (x0 >> 1) : x0;
                    for (int pnl = 0; pnl < a.out_panels; ++pnl) {
                        if (a.out_row_dim == 3)
                            tma_store_4d(&tmO, stg + (uint32_t)pnl * sink.panel_bytes, n0 + pnl * panel_cols, xc, s0, orow);
                        else
                            tma_store_4d(&tmO, stg + (uint32_t)pnl * sink.panel_bytes, n0 + pnl * panel_cols, xc, orow, s0);
                    }
                    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                }
                // the group's next row is laid out in its other tile
                stg += buf_step; sink.row_base += buf_step; pc.sink.row_base += buf_step;
                buf_step = 0u - buf_step;
            }
        }
        if (leader) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    tc_fence_before();
    __syncthreads();
    if (s_abort) {
        if (threadIdx.x == 0) {
            // let this CTA's own copies land before its shared memory is given back (bounded)
            for (uint32_t i = 0; i < 4096 && !mbar_try_wait(bar_w, 0); ++i) __nanosleep(64);
            const int issued = s_issued;
            for (int st = 0; st < a.nstage; ++st) {
                int last = -1;
                for (int t = st; t < issued; t += a.nstage) last = t;
                if (last < 0) continue;
                const uint32_t par = (uint32_t)((last / a.nstage) & 1);
                for (uint32_t i = 0; i < 4096 && !mbar_try_wait(bar_full + 8u * st, par); ++i) __nanosleep(64);
            }
            atomicExch(a.status, 1u);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)a.tmem_cols) : "memory");
    }
}

// The plan for one of the two builds.
bool make_plan(int dtype, int S, int Win, int Wout, int Cin, int Cout, int Kh, int Kw, int stride_x, int ring_rows,
               int out_esize, int pooled, int pair, int light, TcPlan* p)
{
    *p = TcPlan{};
    if (dtype != 1 && dtype != 2) return false;
    const int esize = dtype == 1 ? 2 : 1;
    const int row_bytes = Cin * esize;
    if (stride_x < 1 || stride_x > 8) return false;     // (a tensor map's traversal stride is at most 8)
    if (!(row_bytes == 32 || row_bytes == 64 || (row_bytes >= 128 && row_bytes % 128 == 0))) return false;
    if (Kh * Kw > 32 || Cout % 16 != 0) return false;
    p->swb = row_bytes >= 128 ? 128 : row_bytes;
    p->KB = p->swb / esize;
    p->n_kb = Cin / p->KB;
    // One box per (input row, K block) carries the Kw-1 halo positions of every stream in the tile and the kx taps read it at
    // row offsets (the swizzle is a function of the absolute shared-memory address, whatever its span).  A box per kx tap, as
    // x-strided layers whose positions cannot be taken in groups need, moves Kw times the rows through the copy engine
    // (32 -> 64 channels int8, stride 2, 2048 streams of 254-wide rows: 2.15 ms with three strided boxes, 1.93 ms as groups of
    // two positions).
    // `pair`: a position is 16 bytes, half a K step.  The input row then lies in shared memory as it is (no swizzle, rows of 16
    // bytes) and a K step is two neighbouring positions: the leading-dimension offset of the A descriptor is one row.  Cin and Kw
    // are those of the pairs: 32 bytes, half the taps (rounded up; the odd one has zero weights).  No x-unfold pass is needed
    // (16 -> 32 channels int8, 4096 streams of 26-wide rows with pool: 0.183 -> 0.149 ms).
    p->light = light;
    const size_t limit = light ? LIGHT_SMEM : SMEM_LIMIT, slack = light ? 1536 : 10240;
    const int tmem_max = light ? 256 : 512;
    p->pair = pair;
    if (pair && (row_bytes != 32 || stride_x != 1)) return false;
    p->shift_mode = Kw > 1 && stride_x == 1;
    const int halo = pair ? 2 * Kw : (p->shift_mode ? Kw - 1 : 0);      // (paired: one position more than the taps read, an even number)
    const int max_bx = pair ? 128 - halo : 128;          // (a paired box is counted in half positions, at most 256)
    if (Wout >= max_bx) {
        p->n_xt = (Wout + max_bx - 1) / max_bx;
        p->BX = (Wout + p->n_xt - 1) / p->n_xt;
        // (pooled pairs lie in one tile: an odd share is made even, positions past the row are clipped.  vgg2d, 5 streams of 157-wide
        // rows in groups of 29: 0.557 ms with the first pooling launches apart, 0.54 with them folded)
        if (pooled) p->BX += p->BX & 1;
        p->BS = 1;
    } else {
        p->n_xt = 1;
        p->BX = Wout + (pooled && Wout + halo > 64 ? Wout & 1 : 0);     // (one stream to a tile)
        p->BS = 1 + (128 - p->BX) / (p->BX + halo);   // (BS-1)*(BX+halo) + BX <= 128 output lanes
        if (p->BS > S) p->BS = S;
    }
    p->BXP = p->BX + halo;
    // An x-strided layer needs one box per kx tap (the tap's positions x' * stride + kx - pad are then one strided
    // walk of the input row, which the tensor map does); the haloed tile of the row-shift mode has no such form.
    if (stride_x != 1 && (p->swb == 128 || Kw == 1)) return false;
    p->sx = stride_x;
    if (p->BXP * stride_x > 256) return false;          // the box is given in input positions
    // A stage holds exactly the TMA box (BS streams x BXP positions).  The MMAs read 128 rows from row kx on,
    // so for the last positions they run past the box into whatever follows in shared memory: those are
    // lanes outside the tile, whose accumulators nobody reads.
    // (the boxes of an x-strided layer lie side by side in the stage, under one barrier)
    const int n_box = stride_x != 1 ? Kw : 1;
    const size_t pos_bytes = pair ? 16 : p->swb;
    const size_t box_pitch = ((size_t)p->BS * p->BXP * pos_bytes + 1023) / 1024 * 1024;
    const size_t a_stage = (size_t)n_box * box_pitch;
    p->a_stage_bytes = (int)a_stage;
    p->n_box = n_box;
    p->a_box_pitch = (int)box_pitch;
    p->n_mt = p->n_xt * ((S + p->BS - 1) / p->BS);
    const int taps = Kh * Kw;
    // a launch that emits pooled rows stages half a tile of positions
    const int stage_rows = pooled ? 64 : 128;
    int best = 0, best_units = -1;
    for (int nt = 256; nt >= 16; nt >>= 1) {
        if (Cout % nt) continue;
        // TMEM slots.  An epilogue group tells the uses of a slot apart by the parity of its barrier, so it must have seen the row that
        // used the slot before a row of its own: no group may skip as many rows as there are slots.  Its first row comes after at
        // most the rows begun by an earlier block (Kh - 1 at stride 1, at most ring_rows) and a turn of all groups, by rows or by pairs.
        const int n_cin = ring_rows == Kh ? Kh - 1 : ring_rows, groups = light ? LIGHT_GROUPS : FULL_GROUPS;
        const int slots = tmem_max / nt > 16 ? 16 : tmem_max / nt;
        if (slots < ring_rows + 1 || slots < n_cin + (pooled ? 2 : 1) * groups) continue;
        if ((ring_rows + 256 / nt - 1) / (256 / nt) + 1 > 4) continue;   // at most 4 MMA segments per input row
        const size_t wb = (size_t)taps * p->n_kb * nt * p->swb;
        if (wb + (light ? 2 : 3) * a_stage + (size_t)stage_rows * nt * out_esize + slack > limit) continue;   // one staging tile at least
        const int units = p->n_mt * (Cout / nt);
        if (units >= (light ? 1 : 120)) { best = nt; break; }          // enough CTAs for the 148 SMs: take the widest such tile
        // 1D nets come in long blocks of rows, which row chunks spread over the SMs: there the widest tile that fits
        // wins, because every channel slice fetches the Δ-rows again (audio1d's 128-channel layers with 16-channel
        // tiles moved 4.2 GB per layer through the L2)
        if (Win == 1) { best = nt; break; }
        if (units > best_units) { best_units = units; best = nt; }
    }
    if (!best) return false;
    p->Ntile = best;
    p->n_nt = Cout / best;
    p->nslot = tmem_max / best;
    if (p->nslot > 16) p->nslot = 16;
    // as many resident rows as tensor memory holds: the fewer input rows whose window of ring rows
    // wraps around the slot array, the fewer split MMAs
    int cols = 32;
    while (cols < p->nslot * best) cols <<= 1;
    p->tmem_cols = cols;
    const size_t wb = ((size_t)taps * p->n_kb * best * p->swb + 1023) / 1024 * 1024;
    p->out_esize = out_esize;
    p->out_pwb = best * out_esize >= 128 ? 128 : best * out_esize;
    p->out_panels = best * out_esize / p->out_pwb;
    p->out_stage_rows = stage_rows;
    p->out_stage_bytes = p->out_panels * stage_rows * p->out_pwb;
    // as many epilogue groups (one staging tile each) as still leave three Δ-row stages
    p->out_groups = 1;
    p->out_bufs = 1;
    // layers with many short K blocks per row (little MMA work per tile) need a deeper pipeline to cover the
    // copy latency more than they need a second epilogue group
    const size_t want_stages = light ? 2 : (p->n_kb >= 4 ? 4 : 3);
    for (int g = light ? LIGHT_GROUPS : FULL_GROUPS; g > 1; --g)
        if (wb + want_stages * a_stage + (size_t)g * p->out_stage_bytes + slack <= limit) { p->out_groups = g; break; }
    // a second staging tile per group where it still leaves one more Δ-row stage than wanted
    if (!light && wb + (want_stages + 1) * a_stage + 2 * (size_t)p->out_groups * p->out_stage_bytes + slack <= limit) p->out_bufs = 2;
    // the MMAs' run past a small box (see a_stage) must end inside this CTA's shared memory: what follows the
    // last stage (the staging tiles) covers it, or padding is added behind them
    const size_t overrun = (size_t)(128 + halo) * pos_bytes > box_pitch ? (size_t)(128 + halo) * pos_bytes - box_pitch : 0;
    const size_t tail_have = (size_t)p->out_groups * p->out_bufs * p->out_stage_bytes;
    const size_t tail_pad = overrun > tail_have ? (overrun - tail_have + 1023) / 1024 * 1024 : 0;
    const size_t reserve = light ? 1536 : 8192 + 1024;
    if (limit < reserve + wb + tail_have + tail_pad + 2 * a_stage) return false;
    const size_t room = limit - reserve - wb - tail_have - tail_pad;   // static shared memory and alignment slack stay free
    int nstage = (int)(room / a_stage);
    if (nstage > 8) nstage = 8;
    if (nstage < 2) return false;
    p->nstage = nstage;
    p->smem_bytes = 1024 + wb + (size_t)nstage * a_stage + tail_have + tail_pad + 8 * (2 * nstage + taps + 2 * p->nslot + 1) + 64;
    p->w_bytes = (size_t)taps * Cout * Cin * esize;
    p->ok = 1;
    return true;
}

}  // namespace

// Which build.  A layer of few input channels has little tensor-core work per row and is bound by its epilogue and by the waits
// between the roles of one CTA; a second CTA on the SM adds a fourth group and fills those waits.  Its price is half the room:
// where that costs a narrower channel tile the input is read again for each, and the full build is the better one
// (int8 64 -> 64 with pool, 2048 streams of 126-wide rows: 0.80 ms full, 0.89 light with half the tile; bf16 128 -> 128, 64 x 112: 0.201
// and 0.228; bf16 256 -> 256, 64 x 56: 0.256 and 0.346).  With the same tile the light build wins as soon as there are more CTAs
// than SMs (int8 32 -> 64 stride 2, 254-wide rows: 128 streams 44 us full, 47 light; 192: 82 and 53; 2048: 531 and 339;
// int8 16 -> 32 with pool, 26-wide rows: 512 streams 28 and 30, 768: 47 and 37, 4096: 152 and 111; bf16 16 -> 32, 128-wide rows: 128
// streams 50 and 49, 256: 92 and 57, 1024: 313 and 200; one-row pushes of int8 64 -> 32, 128-wide rows: 128 streams 12 and 13, 1024: 47 and 29).
bool tc_make_plan(int dtype, int S, int Win, int Wout, int Cin, int Cout, int Kh, int Kw, int stride_x, int ring_rows,
                  int out_esize, int pooled, int pair, TcPlan* p)
{
    if (!make_plan(dtype, S, Win, Wout, Cin, Cout, Kh, Kw, stride_x, ring_rows, out_esize, pooled, pair, 0, p)) return false;
    TcPlan light;
    if (make_plan(dtype, S, Win, Wout, Cin, Cout, Kh, Kw, stride_x, ring_rows, out_esize, pooled, pair, 1, &light) &&
        light.Ntile == p->Ntile && light.n_mt * light.n_nt > 148)
        *p = light;
    return true;
}

// Where tap (ky, kx) of a layer goes in the tensor-core copy of its parameters, [tap'][Cout][Cin]: kx by kx, and
// inside a kx the Kh tap rows in the order of the stacked weight tiles (weight_block), so that one copy delivers
// a channel slice with all its taps in the shared-memory order the MMA schedule addresses.
int tc_weight_slot(int ky, int kx, int Kh, int stride) { return kx * Kh + weight_block(ky, Kh, stride); }

int tc_encode_weights(const TcPlan& p, int dtype, const void* d_w, int taps, int Cin, int Cout, void* map_out)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return -1;
    const int esize = dtype == 1 ? 2 : 1;
    if (taps > 256) return -1;
    cuuint64_t dims[3] = {(cuuint64_t)Cin, (cuuint64_t)Cout, (cuuint64_t)taps};
    cuuint64_t strides[2] = {(cuuint64_t)Cin * esize, (cuuint64_t)Cout * Cin * esize};
    cuuint32_t box[3] = {(cuuint32_t)p.KB, (cuuint32_t)p.Ntile, (cuuint32_t)taps};   // all taps of a channel slice and K block
    cuuint32_t es[3] = {1, 1, 1};
    CUresult r = enc((CUtensorMap*)map_out, dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 3,
                     const_cast<void*>(d_w), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(p.swb),
                     CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? 0 : -1;
}

// Returns cudaErrorNotSupported when the launch cannot take this path (the caller then uses the
// CUDA-core kernel): unaligned input pointer or a tensor map the driver rejects.
cudaError_t launch_conv_tc(const ConvArgs& a, const TcPlan& p, int dtype, const void* w_map, int n_in_rows,
                           unsigned int* status, cudaStream_t st)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc || !p.ok) return cudaErrorNotSupported;
    if (((uintptr_t)a.in & 15) != 0 || n_in_rows < 1) return cudaErrorNotSupported;
    const int esize = dtype == 1 ? 2 : 1;
    CUtensorMap tmA;
    const long long stream_elems = a.in_stream_elems ? a.in_stream_elems : (long long)a.Win * a.Cin;
    cuuint64_t dims[4] = {(cuuint64_t)a.Cin, (cuuint64_t)a.Win, (cuuint64_t)a.S, (cuuint64_t)n_in_rows};
    cuuint64_t strides[3] = {(cuuint64_t)a.Cin * esize, (cuuint64_t)stream_elems * esize, (cuuint64_t)a.S * stream_elems * esize};
    // (with a traversal stride the box is counted in input positions and delivers every sx-th of them)
    cuuint32_t box[4] = {(cuuint32_t)p.KB, (cuuint32_t)(p.BXP * p.sx), (cuuint32_t)p.BS, 1};
    cuuint32_t es[4] = {1, 1, 1, 1}, es_in[4] = {1, (cuuint32_t)p.sx, 1, 1};
    if (a.stride_x != p.sx) return cudaErrorNotSupported;
    if (p.pair) {
        // (a stream's row in 8-byte units, two to a position; a.Win counts positions)
        dims[0] = (cuuint64_t)a.Win * 2; dims[1] = 1;
        strides[0] = (cuuint64_t)a.Win * 16;
        box[0] = (cuuint32_t)p.BXP * 2; box[1] = 1;
    }
    CUresult r = enc(&tmA, p.pair ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8, 4,
                     const_cast<void*>(a.in), dims, strides, box, es_in, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     p.pair ? CU_TENSOR_MAP_SWIZZLE_NONE : swizzle_of(p.swb), CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorNotSupported;

    // emitted rows leave through a TMA store: [channel][x][stream][row] or [channel][x][row][stream]
    CUtensorMap tmO;
    const int row_dim = a.out_row_stride > a.out_stream_stride ? 3 : 2;
    {
        const int oes = p.out_esize;
        const int ow = a.pool_fused ? a.Wout / 2 : a.Wout;            // width of the rows that leave the kernel
        const int obx = a.pool_fused ? p.BX / 2 : p.BX;
        if (a.pool_fused && ((p.BX & 1) || ow < 1 || !a.pool_state)) return cudaErrorNotSupported;
        if ((a.pool_fused != 0) != (p.out_stage_rows == 64)) return cudaErrorNotSupported;   // the plan's staging tile must fit the rows that leave
        cuuint64_t od[4] = {(cuuint64_t)a.Cout, (cuuint64_t)ow, 0, 0};
        cuuint64_t os[3] = {(cuuint64_t)a.Cout * oes, 0, 0};
        cuuint32_t ob[4] = {(cuuint32_t)(p.out_pwb / oes), (cuuint32_t)obx, 1, 1};
        od[row_dim] = (cuuint64_t)a.out_rows_extent; od[5 - row_dim] = (cuuint64_t)a.S;
        os[row_dim - 1] = (cuuint64_t)a.out_row_stride * oes; os[4 - row_dim] = (cuuint64_t)a.out_stream_stride * oes;
        ob[5 - row_dim] = (cuuint32_t)p.BS;
        if (((uintptr_t)a.out & 15) != 0 || a.out_rows_extent < 1) return cudaErrorNotSupported;
        const CUtensorMapDataType odt = a.out_elem == E_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                      : (a.out_elem == E_F32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_UINT8);
        const CUtensorMapSwizzle osw = p.out_pwb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B
                                     : (p.out_pwb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                     : (p.out_pwb == 32 ? CU_TENSOR_MAP_SWIZZLE_32B : CU_TENSOR_MAP_SWIZZLE_NONE));
        CUresult ro = enc(&tmO, odt, 4, a.out, od, os, ob, es, CU_TENSOR_MAP_INTERLEAVE_NONE, osw,
                          CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (ro != CUDA_SUCCESS) return cudaErrorNotSupported;
    }

    TcArgs t{};
    t.bias = a.bias; t.ring = a.ring; t.out = a.out; t.status = status;
    t.out_row_stride = a.out_row_stride; t.out_stream_stride = a.out_stream_stride; t.out_row_base = a.out_row_base;
    t.o_begin = a.o_begin; t.r0_positive = a.r0 > 0; t.n_rows = (int)(a.r1 - a.r0); t.n_orows = (int)(a.o_end - a.o_begin);
    t.done_rel = (int)(a.done_end - a.o_begin);
    {
        // rows whose last tap is a real input row of this block (the others below done_end end on bottom padding)
        const long long q = a.r1 + a.pad - a.Kh;
        long long sched = q < 0 ? 0 : q / a.stride + 1;
        if (sched < a.o_begin) sched = a.o_begin;
        if (sched > a.done_end) sched = a.done_end;
        t.sched_rel = (int)(sched - a.o_begin);
    }
    t.base_ty = (int)(a.r0 + a.pad - a.o_begin * a.stride);
    t.S = a.S; t.Wout = a.Wout; t.Cout = a.Cout; t.Kh = a.Kh; t.Kw = a.Kw; t.stride = a.stride;
    t.pad_x = a.pad_x; t.relu = a.relu; t.shift = a.shift; t.ring_rows = a.ring_rows; t.out_elem = a.out_elem;
    t.BX = p.BX; t.BS = p.BS; t.n_xt = p.n_xt; t.Ntile = p.Ntile; t.n_nt = p.n_nt; t.KB = p.KB; t.n_kb = p.n_kb;
    t.swb = p.swb; t.nslot = p.nslot; t.nstage = p.nstage; t.tmem_cols = p.tmem_cols;
    t.BXP = p.BXP; t.shift_mode = p.shift_mode; t.pair = p.pair; t.sx = p.sx; t.a_stage_bytes = p.a_stage_bytes; t.n_box = p.n_box; t.a_box_pitch = p.a_box_pitch;
    t.out_esize = p.out_esize; t.out_pwb = p.out_pwb; t.out_panels = p.out_panels; t.out_stage_bytes = p.out_stage_bytes; t.out_stage_rows = p.out_stage_rows; t.out_groups = p.out_groups; t.out_bufs = p.out_bufs;
    t.out_row_dim = row_dim; t.out_row_first = (int)(a.o_begin - a.out_row_base);
    t.pool = a.pool_fused; t.pool_keep = a.pool_keep; t.pool_state = a.pool_state; t.pool_row_base = a.out_row_base;
    t.o_begin_par = (int)(a.o_begin & 1);
    t.o_begin_half_mod = (int)((a.o_begin >> 1) % p.out_groups);
    t.ring_slot0 = (int)(a.o_begin % a.ring_rows);
    t.pool_row_first = (int)((a.o_begin >> 1) - a.out_row_base);
    t.ring_elems = a.ring_elems; t.pool_state_bytes = a.pool_state_elems * p.out_esize; t.smem_bytes = (unsigned int)p.smem_bytes;
    // row chunks: a layer with few tiles (few streams, narrow rows) spreads the block's rows over more CTAs
    t.n_chunks = 1; t.chunk_rows = t.n_orows; t.chunk_shift = 0;
    {
        const int units = p.n_mt * p.n_nt;
        // (a run reads Kh - 1 rows of its neighbour's: 3x3 layers in runs of 8 rows still gain, 5 vgg2d streams of 131 157-wide rows in one
        // push 213 us with runs of 16 and more, 175 with 8, 199 with 4)
        int min_rows = 2 * a.ring_rows + 2;
        if (min_rows < 8) min_rows = 8;
        const bool no_chunks = (debug_flags() & IDF_DEBUG_NO_ROW_CHUNKS) != 0;
        // (a block that continues rows of an earlier one needs room for the copy of the ring, see ring_in)
        // a launch that takes a first row out of the pool layer's state (its first row is the second of a pair) and
        // also parks one there (its last emitted row is the first of a pair) keeps both in one CTA: read before write
        const bool pool_state_rw = a.pool_fused && a.pool_keep && (a.o_begin & 1) && (a.done_end & 1);
        if (!no_chunks && !pool_state_rw && units < 120 && t.n_orows >= 2 * min_rows && (a.r0 == 0 || a.ring_scratch)) {
            int want = 296 / units;                                 // at most two full waves of CTAs on the 148 SMs
            if (want > t.n_orows / min_rows) want = t.n_orows / min_rows;
            if (want > 1) {
                int rows = (t.n_orows + want - 1) / want;
                rows += rows & 1;                                   // even: a pooling pair stays in one chunk
                t.chunk_shift = a.pool_fused ? (int)(a.o_begin & 1) : 0;
                t.chunk_rows = rows;
                t.n_chunks = (t.n_orows + t.chunk_shift + rows - 1) / rows;
            }
        }
    }
    t.ring_in = a.ring;
    if (t.n_chunks > 1 && a.r0 > 0) {
        cudaError_t ce = launch_ring_copy(a.ring_scratch, a.ring, (long long)a.ring_rows * a.S * a.Wout * a.Cout, st);
        if (ce != cudaSuccess) return ce;
        t.ring_in = a.ring_scratch;
    }
    const unsigned grid = (unsigned)(p.n_mt * p.n_nt * t.n_chunks);
    typedef void (*KernelFn)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const TcArgs);
    static const KernelFn kernels[4][4] = {
        {conv_tc_kernel<1, 1, 0, 3>, conv_tc_kernel<1, 2, 0, 3>, conv_tc_kernel<1, 4, 0, 3>, conv_tc_kernel<1, 4, 1, 3>},
        {conv_tc_kernel<2, 1, 0, 3>, conv_tc_kernel<2, 2, 0, 3>, conv_tc_kernel<2, 4, 0, 3>, conv_tc_kernel<2, 4, 1, 3>},
        {conv_tc_kernel<1, 1, 0, 2>, conv_tc_kernel<1, 2, 0, 2>, conv_tc_kernel<1, 4, 0, 2>, conv_tc_kernel<1, 4, 1, 2>},
        {conv_tc_kernel<2, 1, 0, 2>, conv_tc_kernel<2, 2, 0, 2>, conv_tc_kernel<2, 4, 0, 2>, conv_tc_kernel<2, 4, 1, 2>}};
    const int kidx = p.swb == 32 ? 0 : (p.swb == 64 ? 1 : ((p.shift_mode && a.Kw == 3) ? 3 : 2));
    const int kind = dtype - 1 + (p.light ? 2 : 0);
    const KernelFn fn = kernels[kind][kidx];
    static bool attr_set[4][4][64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[kind][kidx][dev]) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(p.light ? LIGHT_SMEM : SMEM_LIMIT - 6144));
        if (e != cudaSuccess) return e;
        attr_set[kind][kidx][dev] = true;
    }
    // programmatic dependent launch: the kernel may be scheduled while its predecessor drains; it
    // touches nothing but its weights until griddepcontrol.wait
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(tc_threads(p.light ? LIGHT_GROUPS : FULL_GROUPS)); cfg.dynamicSmemBytes = p.smem_bytes; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    // (without the attribute the griddepcontrol instructions in the kernels are no-ops)
    const bool use_pdl = (debug_flags() & IDF_DEBUG_NO_PDL) == 0;
    cfg.attrs = attr; cfg.numAttrs = use_pdl ? 1 : 0;
    cudaError_t le = cudaLaunchKernelEx(&cfg, fn, tmA, *(const CUtensorMap*)w_map, tmO, t);
    if (le != cudaSuccess) return le;
    return cudaGetLastError();
}

}  // namespace idf
