// Wide layers on CTA pairs: tiles of whole output rows, the weights streamed.
//
// The row-ring kernel keeps a channel slice of the weights in shared memory and hands every input row from role to role.  For
// layers of many channels that costs twice: the slice is narrow (64 -> 32 columns a tap at 256 channels), so an MMA of N = 96
// waits for its operands, and every slice fetches the input again.  Here two CTAs of a cluster (one tensor-core instruction over
// both, M = 256) share the weight tiles, half of each in either CTA's shared memory, and a work item is R consecutive output rows of 2 x 128
// (stream, x) positions x N channels with all its R accumulators in tensor memory:
//   - the input rows the item reaches are walked once per K block; row i adds tap ky = i - j to the accumulator of row j, so a
//     Delta-row is in shared memory only while it is the row at hand and serves every accumulator it reaches;
//   - a weight tile (ky, kx, K block) is first needed by the item's first row and last by its last one, R - 1 input rows later: the ring of
//     weight stages is that window and what is on its way;
//   - accumulators finish one input row apart, and the next item begins with the one that finished first: emission overlaps the MMAs
//     with a single set of accumulators;
//   - rows begun by an earlier block get what the ring holds added at the end, rows left open are parked there; input rows that this
//     block does not hold are skipped for all accumulators alike (they belong to one i).
// Operand traffic per 64 cycles of MMA at N = 128: 6 KB of shared memory reads (8 KB may be had), against 12 KB for two M = 128 instructions.
// Bound by the tensor pipe (of which the lanes between two streams' positions take an eighth at 56 or 112 positions) and, at an item's
// ends, by rows with one accumulator to serve.  Two warps issue: with one, every row's hand-over left the pipe idle (256 -> 256 channels 182
// us, 169 with two).  An accumulator is given back by a relaxed arrival: a releasing one waited for the emission's own stores, 1000 to 2000
// cycles (179 -> 170 us).  What a row wants done is worked out by the producer warp, not by the issuing ones.
// Measured on B200 against the row-ring kernel, us: bf16 3x3, 64 streams: 256 -> 256 channels, 56 x 56 257 -> 169 (1400 TFLOP/s), with pool
// 259 -> 174; 128 -> 256 105 -> 96; 128 -> 128, 112 x 112, with pool 194 -> 175; 64 -> 128 110 -> 101; int8 128 -> 128, 256 x 56 x 56 115 -> 95.
// Roles, per CTA: warp 0 input rows (TMA), warps 1-2 MMA (first CTA of the pair), warp 3 weight tiles (TMA), warps 4-19 emission.
#include "../../include/idf.h"
#include "idf_ptx.h"

namespace idf {

int tc_weight_slot(int ky, int kx, int Kh, int stride);

namespace {

constexpr int PAIR_GROUPS = 4;                             // emission groups of four warps, each with a share of an accumulator's columns
constexpr int PAIR_W_WARP = 1 + PAIR_MMA_WARPS, PAIR_EPI_WARP = PAIR_W_WARP + 1;
constexpr int PAIR_THREADS = 32 * (PAIR_EPI_WARP + 4 * PAIR_GROUPS);

struct PairArgs {
    const void* bias;
    void* ring;
    const void* ring_in;         // where the rows begun by earlier blocks are read: the ring, or a copy of it
    void* out;
    void* pool_state;            // [S][Wout/2][Cout] in the output type: x-pooled first row of an open pair
    const void* pool_in;         // where the one that an earlier launch left is read: the same, or a copy of it
    unsigned int* status;
    long long out_row_stride, out_stream_stride, out_row_first;    // elements; output row of row 0 (pooled: of the pair that row 0 begins)
    long long out_elems, ring_elems, pool_elems;
    // rows are counted from the first visited one (pooled: from the even row at or below it)
    int n_in, row_lo, row_hi, done, base_ty, carried;      // visited [row_lo, row_hi), emitted below done; tap ky of row o reads input row o + ky - base_ty
    int ring_slot0, ring_rows;
    int S, Wout, Cout, Kh, Kw, pad_x, relu, shift, out_elem, out_wide, pool_keep;
    int BX, BXP, BS, n_xt, n_mt;
    int N, n_nt, R, KB, n_kb, swb, n_a, n_b, a_bytes, b_bytes, b_tile, a_box_bytes;      // a stage of weights: the Kw tiles of one tap row
    int row_step;                // rows of a unit of work: 1, or the two of a pooled pair
    int n_u, units;              // units of a column of work (position pair x channel slice), in all
    unsigned int smem_bytes;
};

__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.relaxed.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        if (mbar_try_wait_cluster(bar, parity)) return true;
        if ((i & 31u) == 31u) {
            if (*abort_flag) return false;
            __nanosleep(32);
        }
    }
    *abort_flag = 1;
    return false;
}
// loads into this CTA's shared memory that complete on a barrier of the pair's first CTA
__device__ __forceinline__ void tma_pair_4d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_pair_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
// arrives on the barrier at this offset in both CTAs once all MMAs issued so far are done
__device__ __forceinline__ void pair_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
// One 32-byte K step over both CTAs.  Descriptors differ in their low words only; fresh: the accumulator is overwritten.
template <int DT>
__device__ __forceinline__ void pair_mma(uint32_t tmem_d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi, uint32_t idesc, uint32_t fresh)
{
    if (DT == 1)
        asm volatile("{\n\t.reg .pred q;\n\t.reg .b64 a1, b1;\n\tmov.b64 a1, {%1, %2};\n\tmov.b64 b1, {%3, %4};\n\tsetp.eq.b32 q, %6, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %5, q;\n\t}"
                     ::"r"(tmem_d), "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(fresh) : "memory");
    else
        asm volatile("{\n\t.reg .pred q;\n\t.reg .b64 a1, b1;\n\tmov.b64 a1, {%1, %2};\n\tmov.b64 b1, {%3, %4};\n\tsetp.eq.b32 q, %6, 0;\n\t"
                     "tcgen05.mma.cta_group::2.kind::i8 [%0], a1, b1, %5, q;\n\t}"
                     ::"r"(tmem_d), "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(fresh) : "memory");
}

// W sums of one position -> the words of W emitted values
template <int DT, int W>
__device__ __forceinline__ void pack_out(const uint32_t* v, const uint32_t* bias, int bf16, int relu, int shift, uint32_t* pk)
{
    if (DT == 2) pack_i8<W>(v, (const int*)bias, relu, shift, pk);
    else pack_f<W>(v, (const float*)bias, bf16, relu, pk);
}

template <int W>
__device__ __forceinline__ void ring_load(const uint32_t* p, uint32_t* v)
{
#pragma unroll
    for (int j = 0; j < W; j += 8) ld_global_v8(p + j, *(uint32_t(*)[8])(v + j));
}
template <int DT, int W>
__device__ __forceinline__ void ring_add(uint32_t* v, const uint32_t* r)
{
#pragma unroll
    for (int j = 0; j < W; ++j) v[j] = DT == 1 ? __float_as_uint(__uint_as_float(v[j]) + __uint_as_float(r[j])) : v[j] + r[j];
}
// NW words: 4 to an address of 16-byte alignment, 8, 16 or 32 to one of 32 bytes (wide) or 16, 32 bytes at a time
template <int NW>
__device__ __forceinline__ void store_words(unsigned char* p, const uint32_t* v, int wide)
{
    if (NW == 4) { st_global_v4(p, v); return; }
#pragma unroll
    for (int j = 0; j + 8 <= NW; j += 8) st_global_32(p + 4 * j, v + j, wide);
}
// A thread's position in the work item at hand (emission).
struct PairSpot {
    int s, x, n0;                // stream, position, first channel of the slice
    bool valid;                  // a position of the map
    long long ring, out;         // element offsets at channel n0: in a ring row, and in the output (row 0; pooled: pair 0, this thread's share of the channels)
};
__device__ __forceinline__ const uint32_t* bias_at(const PairArgs& a, int co) { return a.bias ? (const uint32_t*)a.bias + co : nullptr; }
__device__ __forceinline__ long long ring_row(const PairArgs& a, int row)
{
    return (long long)((a.ring_slot0 + row) % a.ring_rows) * a.S * a.Wout * a.Cout;
}
// 16 columns from column c on of what an earlier block left of a row; false: nothing
__device__ __forceinline__ bool ring_fetch(const PairArgs& a, const PairSpot& p, int row, int c, uint32_t* r)
{
    const long long at = ring_row(a, row) + p.ring + c;
    const bool have = a.carried && row < a.base_ty && p.valid && IDF_OK_AT(a.status, at, a.ring_elems - 15);
    if (have) ring_load<16>((const uint32_t*)a.ring_in + at, r);
    return have;
}
// ... is added; true: the row is complete and its sums are to be emitted, else they are parked
template <int DT>
__device__ __forceinline__ bool ring_exchange(const PairArgs& a, const PairSpot& p, int row, int c, uint32_t* v, bool have, const uint32_t* r)
{
    if (have) ring_add<DT, 16>(v, r);
    if (row < a.done) return true;
    const long long at = ring_row(a, row) + p.ring + c;
    if (p.valid && IDF_OK_AT(a.status, at, a.ring_elems - 15)) {
        st_global_v8((uint32_t*)a.ring + at, *(uint32_t(*)[8])v);
        st_global_v8((uint32_t*)a.ring + at + 8, *(uint32_t(*)[8])(v + 8));
    }
    return false;
}
template <int DT, int W>
__device__ __forceinline__ bool exchange_words(const PairArgs& a, const PairSpot& p, int row, int c, uint32_t* v)
{
    bool emit = true;
#pragma unroll
    for (int h = 0; h < W; h += 16) {
        uint32_t r[16];
        const bool have = ring_fetch(a, p, row, c + h, r);
        emit = ring_exchange<DT>(a, p, row, c + h, v + h, have, r);
    }
    return emit;
}
template <int DT, int W>
__device__ __forceinline__ void emit_words(const PairArgs& a, const PairSpot& p, int row, int c, const uint32_t* v)
{
    const long long at = p.out + (a.out_row_first + row) * a.out_row_stride + c;
    if (!p.valid || !IDF_OK_AT(a.status, at, a.out_elems - W + 1)) return;
    unsigned char* out = (unsigned char*)a.out;
    const uint32_t* bias = bias_at(a, p.n0 + c);
    uint32_t pk[W];
    if (DT == 2) {
        pack_out<2, W>(v, bias, 0, a.relu, a.shift, pk);
        store_words<W / 4>(out + at, pk, a.out_wide);
    } else if (a.out_elem == E_BF16) {
        pack_out<1, W>(v, bias, 1, a.relu, 0, pk);
        store_words<W / 2>(out + 2 * at, pk, a.out_wide);
    } else {
        pack_out<1, W>(v, bias, 0, a.relu, 0, pk);
        store_words<W>(out + 4 * at, pk, a.out_wide);
    }
}

// One accumulator: this thread's columns c0, c0 + step, .. in pieces of W.  It is given back as soon as its last piece is in registers.
template <int DT, int W, typename Release>
__device__ __forceinline__ void emit_plain(const PairArgs& a, const PairSpot& p, int row, bool has, uint32_t tcol, int c0, Release release)
{
    constexpr int STEP = W * PAIR_GROUPS;
    const bool plain = row < a.done && !(a.carried && row < a.base_ty);
    if (c0 >= a.N && has) release();
    for (int c = c0; c < a.N; c += STEP) {
        uint32_t v[W];
        if (has) {
            __syncwarp();
            tmem_ld<W>(tcol + c, v);
            if (c + STEP >= a.N) release();
        } else {
#pragma unroll
            for (int j = 0; j < W; ++j) v[j] = 0u;
        }
        if (plain || exchange_words<DT, W>(a, p, row, c, v)) emit_words<DT, W>(a, p, row, c, v);
    }
}

// A pair of rows, row (even) and row + 1 as far as they are in use (use0, use1), with the 2x2 max-pool behind the layer folded in.
// OP 0: two bf16, 1: one fp32, 2: four int8 to a word.  The two lanes of a pooled position share its channels.
template <int DT, int OP, int W, typename Wait, typename Release>
__device__ __forceinline__ bool emit_pooled(const PairArgs& a, const PairSpot& p, int row, bool use0, bool use1, bool has0, bool has1,
                                            uint32_t tcol, int c0, Wait wait, Release release)
{
    constexpr int NW = OP == 0 ? W / 2 : (OP == 1 ? W : W / 4), H = NW / 2, ES = OP == 0 ? 2 : (OP == 1 ? 4 : 1), STEP = W * PAIR_GROUPS;
    const bool emit0 = use0 && row < a.done, emit1 = use1 && row + 1 < a.done;
    const bool odd = threadIdx.x & 1;
    const int wp = a.Wout >> 1, xp = p.x >> 1;
    const bool here = p.valid && xp < wp;
    if (c0 >= a.N) {
        if (has0) { if (!wait(0)) return false; release(0); }
        if (has1) { if (!wait(1)) return false; release(1); }
        return true;
    }
    for (int c = c0; c < a.N; c += STEP) {
        uint32_t best[NW];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (!(k ? use1 : use0)) continue;
            uint32_t v[W];
            if (k ? has1 : has0) {
                if (c == c0 && !wait(k)) return false;
                __syncwarp();
                tmem_ld<W>(tcol + (uint32_t)(k * a.N + c), v);
                if (c + STEP >= a.N) release(k);
            } else {
#pragma unroll
                for (int j = 0; j < W; ++j) v[j] = 0u;
            }
            const bool plain = row + k < a.done && !(a.carried && row + k < a.base_ty);
            if (!plain && !exchange_words<DT, W>(a, p, row + k, c, v)) continue;
            uint32_t pk[NW];
            pack_out<DT, W>(v, bias_at(a, p.n0 + c), OP == 0, a.relu, a.shift, pk);
            if (k && emit0) {
#pragma unroll
                for (int j = 0; j < NW; ++j) best[j] = word_max<OP>(best[j], pk[j]);
            } else {
#pragma unroll
                for (int j = 0; j < NW; ++j) best[j] = pk[j];
            }
        }
        if (!emit0 && !emit1) continue;
        __syncwarp();
        uint32_t m[H];
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const uint32_t other = __shfl_xor_sync(0xffffffffu, odd ? best[j] : best[H + j], 1);
            m[j] = word_max<OP>(odd ? best[H + j] : best[j], other);
        }
        const int share = odd ? 4 * H / ES : 0;
        if (!emit0 || !emit1) {
            // the pair's other row came with an earlier launch, or comes with a later one
            const long long at = ((long long)p.s * wp + xp) * a.Cout + p.n0 + c + share;
            if (!here || !IDF_OK_AT(a.status, at, a.pool_elems - 4 * H / ES + 1)) continue;
            if (!emit1) {
                unsigned char* st = (unsigned char*)a.pool_state + at * ES;
                if (a.pool_keep) {
#pragma unroll
                    for (int j = 0; j < H; j += 4) st_global_v4(st + 4 * j, m + j);
                }
                continue;
            }
#pragma unroll
            for (int j = 0; j < H; j += 4) {
                const uint4 g = *(const uint4*)((const unsigned char*)a.pool_in + at * ES + 4 * j);
                m[j] = word_max<OP>(m[j], g.x); m[j + 1] = word_max<OP>(m[j + 1], g.y);
                m[j + 2] = word_max<OP>(m[j + 2], g.z); m[j + 3] = word_max<OP>(m[j + 3], g.w);
            }
        }
        const long long at = p.out + (a.out_row_first + (row >> 1)) * a.out_row_stride + c + share;
        if (here && IDF_OK_AT(a.status, at, a.out_elems - 4 * H / ES + 1)) store_words<H>((unsigned char*)a.out + at * ES, m, a.out_wide);
    }
    return true;
}

// KW: kx taps known at compile time (the MMA warp's loop is then straight code), or 0
template <int DT, int KSTEPS, int KW, int POOL>
__global__ void __launch_bounds__(PAIR_THREADS, 1)
conv_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ PairArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ uint4 s_sched[PAIR_MAX_A];                              // per input row at hand: what the MMA warp has to do with it
    __shared__ __align__(8) unsigned long long s_bars[2 * PAIR_MAX_A + 2 * PAIR_MAX_B + 2 * PAIR_MAX_R + PAIR_MMA_WARPS];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const uint32_t sA = (smem_u32(smem_raw) + 1023u) & ~1023u, sB = sA + (uint32_t)(a.n_a * a.a_bytes);
    const uint32_t a_full = smem_u32(s_bars), a_empty = a_full + 8u * PAIR_MAX_A;
    const uint32_t b_full = a_empty + 8u * PAIR_MAX_A, b_empty = b_full + 8u * PAIR_MAX_B;
    const uint32_t acc_full = b_empty + 8u * PAIR_MAX_B, acc_free = acc_full + 8u * PAIR_MAX_R, bar_done = acc_free + 8u * PAIR_MAX_R;

    if (threadIdx.x == 0) {
        s_abort = 0;
        if (!IDF_OK_AT(a.status, sB + (uint32_t)(a.n_b * a.b_bytes) - smem_u32(smem_raw) - 1u, a.smem_bytes) || !IDF_OK_AT(a.status, a.n_a - 1, PAIR_MAX_A) ||
            !IDF_OK_AT(a.status, a.n_b - 1, PAIR_MAX_B) || !IDF_OK_AT(a.status, a.R - 1, PAIR_MAX_R)) s_abort = 1;
    }
    if (warp == 2) {
        // ("full" barriers are those of the pair's first CTA: its producer's arrival and the bytes of both; "empty" ones are each CTA's own)
        if (lane < a.n_a) { mbar_init(a_full + 8u * lane, 1); mbar_init(a_empty + 8u * lane, PAIR_MMA_WARPS); }
        if (lane < a.n_b) { mbar_init(b_full + 8u * lane, 1); mbar_init(b_empty + 8u * lane, PAIR_MMA_WARPS); }
        if (lane < PAIR_MAX_R) { mbar_init(acc_full + 8u * lane, 1); mbar_init(acc_free + 8u * lane, 2 * 4 * PAIR_GROUPS); }
        if (lane < PAIR_MMA_WARPS) mbar_init(bar_done + 8u * lane, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"((uint32_t)PAIR_TMEM) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    tc_fence_after();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    volatile int* abort_flag = &s_abort;
    const uint32_t tmem_base = s_tmem_base;
    if (warp != PAIR_W_WARP) asm volatile("griddepcontrol.wait;" ::: "memory");                       // (the parameters do not depend on earlier kernels)
    PairWalk w;

    if (warp == 0) {
        // ------------------------------ input rows ---------------------------------------------
        if (lane == 0) {
            const uint32_t full0 = map_to_rank(a_full, 0);
            int stage = 0;
            uint32_t ph = 1;
            bool ok = true;
            // (no item without input rows: the schedule goes by rows)
            auto skip = [&](bool m) { while (m && w.i_lo > w.i_hi) m = w.next(a); return m; };
            bool more = w.start(a, blockIdx.x >> 1, gridDim.x >> 1);
            for (more = skip(more); more && ok;) {
                const int mt = 2 * (w.col / a.n_nt) + (int)rank, xt = mt % a.n_xt, x0 = xt * a.BX - a.pad_x, s0 = (mt / a.n_xt) * a.BS;
                PairWalk v = w;                                      // the item at hand
                more = w.next(a);
                more = skip(more);
                for (int kb = 0; kb < a.n_kb && ok; ++kb)
                    for (int i = v.i_lo; i <= v.i_hi; ++i) {
                        // What the MMA warp has to do with this row, section by section (accumulators j_hi, j_hi - 1, ..): one bit each.
                        const int j_hi = min(v.nr - 1, i), j_end = max(v.j_lo, i - a.Kh + 1), n = j_hi - j_end + 1;
                        const uint32_t all = (1u << n) - 1u, oldest = 1u << (n - 1);
                        const uint32_t first = i == v.i_lo ? all : (j_end == v.j_lo ? oldest : 0u);                 // its tap row is wanted for the first time
                        const uint32_t release = i == v.i_hi ? all : (j_hi == v.nr - 1 ? 1u : 0u);                  // ... for the last time
                        const uint32_t fresh = kb != 0 ? 0u : (i == v.i_lo ? all : (i < v.nr ? 1u : 0u));           // the accumulator's first row
                        const uint32_t done = kb != a.n_kb - 1 ? 0u : (i == v.i_hi ? all : (i - a.Kh + 1 >= v.j_lo ? oldest : 0u));    // ... its last one
                        const bool end = !more && kb == a.n_kb - 1 && i == v.i_hi;
                        if (!IDF_OK_AT(a.status, n - 1, PAIR_MAX_R) || !IDF_OK_AT(a.status, (j_hi - n + 1) * a.N, PAIR_TMEM) || !IDF_OK_AT(a.status, (j_hi + 1) * a.N - 1, PAIR_TMEM) ||
                            !IDF_OK_AT(a.status, v.row0 + i - a.base_ty, a.n_in) || !IDF_OK_AT(a.status, stage, a.n_a)) { *abort_flag = 1; ok = false; break; }
                        if (!mbar_wait(a_empty + 8u * stage, ph, abort_flag)) { ok = false; break; }
                        if (rank == 0) {
                            s_sched[stage] = make_uint4((uint32_t)n | (uint32_t)j_hi << 8 | (end ? 1u << 16 : 0u), first | release << 16, fresh | done << 16,
                                                        tmem_base + (uint32_t)(j_hi * a.N));
                            mbar_expect_tx(a_full + 8u * stage, 2u * (uint32_t)a.a_box_bytes);
                        }
                        tma_pair_4d(sA + (uint32_t)(stage * a.a_bytes), &tmA, full0 + 8u * stage, kb * a.KB, x0, s0, v.row0 + i - a.base_ty);
                        if (++stage == a.n_a) { stage = 0; ph ^= 1u; }
                    }
            }
            // the first CTA's last commits must have arrived here before this CTA may leave
            if (ok) pair_drain(stage, ph, a.n_a, [&](int s, uint32_t parity) { return mbar_wait(a_empty + 8u * s, parity, abort_flag); });
        }
        __syncwarp();
    } else if (warp == PAIR_W_WARP) {
        // ------------------------------ weight tiles -------------------------------------------
        if (lane == 0) {
            const uint32_t full0 = map_to_rank(b_full, 0);
            const uint32_t half = (uint32_t)(a.N / 2) * a.swb;
            // A stage that is not free at once is waited for behind the dependency wait: the wait is bounded, and before that it would last as
            // long as the kernel in front of this one does.
            int stage = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (bool more = w.start(a, blockIdx.x >> 1, gridDim.x >> 1); more && ok; more = w.next(a)) {
                const int n0 = (w.col % a.n_nt) * a.N + (int)rank * (a.N / 2);
                for (int kb = 0; kb < a.n_kb && ok; ++kb)
                    for (int i = w.i_lo; i <= w.i_hi && ok; ++i)
                        // the tap rows that input row i is the first to use, in the order the MMAs want them
                        for (int j = min(w.nr - 1, i); j >= max(w.j_lo, i - a.Kh + 1); --j) {
                            if (i != w.i_lo && j != w.j_lo) continue;
                            if (!IDF_OK_AT(a.status, i - j, a.Kh) || !IDF_OK_AT(a.status, n0 + a.N / 2 - 1, a.Cout) || !IDF_OK_AT(a.status, stage, a.n_b)) { *abort_flag = 1; ok = false; break; }
                            if (!mbar_test(b_empty + 8u * stage, ph)) {
                                asm volatile("griddepcontrol.wait;" ::: "memory");
                                if (!mbar_wait(b_empty + 8u * stage, ph, abort_flag)) { ok = false; break; }
                            }
                            if (rank == 0) mbar_expect_tx(b_full + 8u * stage, 2u * (uint32_t)a.Kw * half);
                            // (slot of a tap in the parameters: see tc_weight_slot, stride 1)
                            for (int kx = 0; kx < a.Kw; ++kx)
                                tma_pair_3d(sB + (uint32_t)(stage * a.b_bytes + kx * a.b_tile), &tmW, full0 + 8u * stage, kb * a.KB, n0, kx * a.Kh + a.Kh - 1 - (i - j));
                            if (++stage == a.n_b) { stage = 0; ph ^= 1u; }
                        }
            }
            asm volatile("griddepcontrol.wait;" ::: "memory");
            if (ok) pair_drain(stage, ph, a.n_b, [&](int s, uint32_t parity) { return mbar_wait(b_empty + 8u * s, parity, abort_flag); });
        }
        __syncwarp();
    } else if (warp < PAIR_W_WARP) {
        // ------------------------------ MMA issuers --------------------------------------------
        // Two warps: the tensor pipe holds only a few instructions, and what a warp has to do between two rows would leave it idle.  An
        // accumulator belongs to one of them (every other one), which issues all that is added to it, in order.
        if (rank == 0) {
            const uint32_t mine = (uint32_t)warp & 1u;                      // j & 1 of this warp's accumulators
            const uint64_t desc = make_smem_desc(0, a.swb);
            const uint32_t d_hi = (uint32_t)(desc >> 32), d_lo = (uint32_t)desc;
            const uint32_t idesc = (DT == 1 ? ((1u << 4) | (1u << 7) | (1u << 10)) : ((2u << 4) | (1u << 7) | (1u << 10))) |
                                   ((256u >> 4) << 24) | ((uint32_t)(a.N >> 3) << 17);
            constexpr uint32_t POS = 2 * KSTEPS;                            // one position of the input row, in descriptor units
            const uint32_t a_base = d_lo | ((sA & 0x3FFFFu) >> 4), b_base = d_lo | ((sB & 0x3FFFFu) >> 4);
            const uint32_t a_units = (uint32_t)a.a_bytes >> 4, b_units = (uint32_t)a.b_bytes >> 4, b_tile = (uint32_t)a.b_tile >> 4;
            const uint32_t b_span = (uint32_t)a.n_b * b_units, b_end = b_base + b_span;
            const bool issuer = elect_one();
            const int Kw = KW ? KW : a.Kw, n_a = a.n_a, n_b = a.n_b;
            const uint32_t N = (uint32_t)a.N, sched = smem_u32(s_sched);
            // stages: input row at hand; oldest tap row still wanted; next one to be waited for
            int sa = 0, tail = 0, head = 0;
            uint32_t pa = 0, ph_head = 0, free_ph = 0xffffffffu;
            bool more = w.start(a, blockIdx.x >> 1, gridDim.x >> 1), ok = true;
            while (more && w.i_lo > w.i_hi) more = w.next(a);
            // The tensor pipe runs only some instructions behind this warp, which therefore works nothing out: what a row wants done comes with
            // the row (the producer's schedule), and what the next row needs is looked at (barriers without blocking, its schedule entry
            // if it has landed) before the MMAs of the row at hand are issued.
            uint32_t what = 0, uses = 0, acts = 0, d = 0, b_ok = 0;
            auto entry = [&](int stage) {
                asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(what), "=r"(uses), "=r"(acts), "=r"(d) : "r"(sched + 16u * (uint32_t)stage) : "memory");
            };
            if (more) {
                ok = mbar_wait(a_full, 0, abort_flag);
                entry(0);
            }
            while (more && ok) {
                const uint32_t alo = a_base + (uint32_t)sa * a_units, a_bar = a_empty + 8u * sa, j_hi = (what >> 8) & 0xffu;
                if (++sa == n_a) { sa = 0; pa ^= 1u; }
                const uint32_t a_ok = mbar_test(a_full + 8u * sa, pa);
                // accumulators that begin with this row must have been read out, tap rows it is the first to use must have landed
                if (acts & 0xffffu) {
                    for (uint32_t left = acts & 0xffffu, j = j_hi; left && ok; left >>= 1, --j)
                        if ((left & 1u) && (j & 1u) == mine) {
                            ok = mbar_wait_cluster(acc_free + 8u * j, (free_ph >> j) & 1u, abort_flag);
                            free_ph ^= 1u << j;
                        }
                    tc_fence_after();
                }
                for (uint32_t left = uses & 0xffffu; left && ok; left &= left - 1u) {
                    if (!b_ok) ok = mbar_wait(b_full + 8u * head, ph_head, abort_flag);
                    b_ok = 0;
                    if (++head == n_b) { head = 0; ph_head ^= 1u; }
                }
                if (!ok) break;
                b_ok = mbar_test(b_full + 8u * head, ph_head);
                const uint32_t k0 = (j_hi ^ mine) & 1u;                        // first section of this warp
                uint32_t n = what & 0xffu, act = acts >> k0, dd = d - k0 * N, blo = b_base + (uint32_t)tail * b_units + k0 * b_units;
                const uint32_t done_bits = acts >> 16;
                const bool end = (what & 0x10000u) != 0;
                if (blo >= b_end) blo -= b_span;
                uint32_t release = uses >> 16;
                if (a_ok && !end) entry(sa);
                for (uint32_t k = k0; k < n; k += 2u, act >>= 2, dd -= 2u * N) {
                    if (issuer) {
#pragma unroll
                        for (int kx = 0; kx < Kw; ++kx)
#pragma unroll
                            for (int ks = 0; ks < KSTEPS; ++ks)
                                pair_mma<DT>(dd, alo + (uint32_t)kx * POS + 2u * ks, d_hi, blo + (uint32_t)kx * b_tile + 2u * ks, d_hi, idesc,
                                             kx == 0 && ks == 0 ? act & 1u : 0u);
                    }
                    blo += 2u * b_units;
                    if (blo >= b_end) blo -= b_span;
                }
                // (tap rows are given back in the order in which they came, the oldest first)
                for (; release; release &= release - 1u) {
                    if (issuer) pair_commit(b_empty + 8u * tail);
                    if (++tail == n_b) tail = 0;
                }
                if (issuer) {
                    pair_commit(a_bar);
                    for (uint32_t left = done_bits >> k0, bar = acc_full + 8u * (j_hi - k0); left; left >>= 2, bar -= 16u)
                        if (left & 1u) pair_commit(bar);
                }
                __syncwarp();
                if (end) break;
                if (!a_ok) {
                    ok = mbar_wait(a_full + 8u * sa, pa, abort_flag);
                    entry(sa);
                }
            }
            // (what has been issued finishes before either CTA gives its memory back)
            if (!ok)
                pair_give_up(warp - 1, [&](int k) { if (issuer) pair_commit(bar_done + 8u * k); },
                             [&](int k) {
                                 if (mbar_try_wait(bar_done + 8u * k, 0)) return true;
                                 __nanosleep(64);
                                 return false;
                             });
        }
        __syncwarp();
    } else {
        // ------------------------------ emission -----------------------------------------------
        const int q = warp & 3, grp = (warp - PAIR_EPI_WARP) >> 2;                                       // TMEM lane quarter, share of the columns
        const int m = q * 32 + lane, bs = m / a.BXP, bx = m - bs * a.BXP;
        const uint32_t free0 = map_to_rank(acc_free, 0);
        PairSpot p;
        const uint32_t tlane = tmem_base + ((uint32_t)(q * 32) << 16);
        bool ok = true;
        uint32_t ph = 0;
        auto wait_acc = [&](int j) {
            int got = 1;
            if (lane == 0) got = mbar_wait(acc_full + 8u * j, (ph >> j) & 1u, abort_flag) ? 1 : 0;
            ph ^= 1u << j;
            got = __shfl_sync(0xffffffffu, got, 0);
            tc_fence_after();
            return got != 0;
        };
        auto release_acc = [&](int j) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(free0 + 8u * j);
        };
        const bool wide = a.N >= 32 * PAIR_GROUPS;
        for (bool more = w.start(a, blockIdx.x >> 1, gridDim.x >> 1); more && ok; more = w.next(a)) {
            const int mt = 2 * (w.col / a.n_nt) + (int)rank, xt = mt % a.n_xt;
            p.n0 = (w.col % a.n_nt) * a.N;
            p.s = (mt / a.n_xt) * a.BS + bs;
            p.x = xt * a.BX + bx;
            p.valid = bs < a.BS && bx < a.BX && p.s < a.S && p.x < a.Wout;
            p.ring = ((long long)p.s * a.Wout + p.x) * a.Cout + p.n0;
            p.out = (long long)p.s * a.out_stream_stride + (long long)(POOL ? p.x >> 1 : p.x) * a.Cout + p.n0;
            if (!IDF_OK_AT(a.status, w.nr * a.N - 1, PAIR_TMEM) || !IDF_OK_AT(a.status, w.nr - 1, a.R)) { *abort_flag = 1; break; }
            if (!POOL) {
                for (int j = w.j_lo; j < w.nr; ++j) {
                    const bool has = w.has_taps(a, j);
                    const uint32_t tcol = tlane + (uint32_t)(j * a.N);
                    if (has && !wait_acc(j)) { ok = false; break; }
                    auto release = [&]() { release_acc(j); };
                    if (wide) emit_plain<DT, 32>(a, p, w.row0 + j, has, tcol, 32 * grp, release);
                    else emit_plain<DT, 16>(a, p, w.row0 + j, has, tcol, 16 * grp, release);
                }
            } else {
                for (int j = 0; j < w.nr && ok; j += 2) {
                    const bool use0 = j >= w.j_lo, use1 = j + 1 < w.nr;
                    const bool has0 = use0 && w.has_taps(a, j), has1 = use1 && w.has_taps(a, j + 1);
                    const uint32_t tcol = tlane + (uint32_t)(j * a.N);
                    auto wait = [&](int k) { return wait_acc(j + k); };
                    auto release = [&](int k) { release_acc(j + k); };
                    if (DT == 1 && a.out_elem == E_F32)
                        ok = emit_pooled<1, 1, 16>(a, p, w.row0 + j, use0, use1, has0, has1, tcol, 16 * grp, wait, release);
                    else
                        ok = emit_pooled<DT, DT == 1 ? 0 : 2, DT == 1 ? 16 : 32>(a, p, w.row0 + j, use0, use1, has0, has1, tcol, (DT == 1 ? 16 : 32) * grp, wait, release);
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (s_abort) {
        if (threadIdx.x == 0) {
            // this CTA's own copies must land before its shared memory is given back.  They complete on the first CTA's barriers, which the
            // second one cannot look at: a bounded pause, long against any copy, does for both.
            for (uint32_t i = 0; i < 64; ++i) __nanosleep(4096);
            atomicOr(a.status, 1u);
        }
        __syncthreads();
    }
    // neither CTA leaves while the other's instructions read its memory or signal its barriers
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)PAIR_TMEM) : "memory");
    }
}

}  // namespace

bool pair_make_plan(int dtype, int Win, int Cin, int Cout, int Kh, int Kw, int stride, PairPlan* p)
{
    *p = PairPlan{};
    if (dtype != 1 && dtype != 2) return false;
    const int es = dtype == 1 ? 2 : 1, row = Cin * es;
    if (Win == 1 || stride != 1 || Kh * Kw == 1 || Kh * Kw > 256) return false;
    // (fewer than 64 channels to a slice: only where the launches are forced here, which the library's rule never does)
    if (!(row == 64 || (row >= 128 && row % 128 == 0)) || Cout % 32 != 0) return false;
    p->swb = row >= 128 ? 128 : row;
    p->KB = p->swb / es;
    p->n_kb = Cin / p->KB;
    p->ok = 1;
    return true;
}

// cudaErrorNotSupported: the launch cannot take this path (alignment, no tile that fits, a tensor map the driver rejects).
cudaError_t launch_conv_pair(const ConvArgs& a, PairPlan& p, int dtype, const void* d_w, cudaStream_t st)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc || !p.ok || a.o_end <= a.o_begin || a.r1 <= a.r0 || a.stride != 1 || a.stride_x != 1) return cudaErrorNotSupported;
    if (((uintptr_t)a.in & 15) != 0 || ((uintptr_t)a.out & 15) != 0) return cudaErrorNotSupported;
    const int es = dtype == 1 ? 2 : 1, pooled = a.pool_fused, odd0 = pooled ? (int)(a.o_begin & 1) : 0;
    const long long o0 = a.o_begin - odd0;
    if (a.o_end - o0 > 0x3fffffffLL) return cudaErrorNotSupported;
    PairArgs t{};
    t.row_lo = odd0; t.row_hi = (int)(a.o_end - o0); t.done = (int)(a.done_end - o0);
    PairPlan::Seen& seen = p.seen[t.row_hi & 3];
    if (seen.rows != t.row_hi || seen.pooled != pooled) {
        seen.rows = t.row_hi; seen.pooled = pooled;
        seen.tiles = pair_tiles(a.S, a.Wout, a.Cout, a.Kh, a.Kw, p.swb, p.n_kb, t.row_hi, pooled);
    }
    const PairTiles g = seen.tiles;
    if (!g.ok) return cudaErrorNotSupported;
    t.bias = a.bias; t.ring = a.ring; t.ring_in = a.ring; t.out = a.out; t.pool_state = a.pool_state; t.status = a.status;
    t.out_row_stride = a.out_row_stride; t.out_stream_stride = a.out_stream_stride;
    t.out_row_first = pooled ? (o0 >> 1) - a.out_row_base : o0 - a.out_row_base;
    t.out_elems = a.out_elems; t.ring_elems = a.ring_elems; t.pool_elems = a.pool_state_elems;
    t.n_in = (int)(a.r1 - a.r0); t.base_ty = (int)(a.r0 + a.pad - o0); t.carried = a.r0 > 0;
    t.ring_slot0 = (int)(o0 % a.ring_rows); t.ring_rows = a.ring_rows;
    t.S = a.S; t.Wout = a.Wout; t.Cout = a.Cout; t.Kh = a.Kh; t.Kw = a.Kw; t.pad_x = a.pad_x; t.relu = a.relu; t.shift = a.shift;
    t.out_elem = a.out_elem; t.out_wide = ((uintptr_t)a.out & 31) == 0; t.pool_keep = a.pool_keep;
    t.BX = g.BX; t.BXP = g.BXP; t.BS = g.BS; t.n_xt = g.n_xt; t.n_mt = g.n_mt;
    t.N = g.N; t.n_nt = a.Cout / g.N; t.R = g.R; t.KB = p.KB; t.n_kb = p.n_kb; t.swb = p.swb; t.n_a = g.n_a; t.n_b = g.n_b;
    t.a_bytes = (int)g.a_bytes; t.b_bytes = (int)(g.b_tile * a.Kw); t.b_tile = (int)g.b_tile; t.a_box_bytes = (int)g.a_box;
    t.row_step = g.row_step; t.n_u = g.n_u; t.units = (int)g.units;
    t.pool_in = a.pool_state;
    // a row begun by an earlier block and one left open by this one may share a ring slot and lie in different CTAs; so may the pooled rows
    // that the block takes and parks (both copies are one launch)
    const bool copy_ring = t.carried && a.o_end - a.o_begin > a.ring_rows, copy_pool = pooled && pair_pool_state_both(a.o_begin, a.done_end, a.pool_keep);
    if (copy_ring || copy_pool) {
        if (!a.ring_scratch || (copy_pool && !a.pool_scratch)) return cudaErrorNotSupported;
        cudaError_t ce = launch_state_copy(a.ring_scratch, a.ring, copy_ring ? (long long)a.ring_rows * a.S * a.Wout * a.Cout : 0,
                                           a.pool_scratch, a.pool_state, copy_pool ? a.pool_state_elems * elem_size(a.out_elem) / 4 : 0, st);
        if (ce != cudaSuccess) return ce;
        if (copy_ring) t.ring_in = a.ring_scratch;
        if (copy_pool) t.pool_in = a.pool_scratch;
    }
    CUtensorMap tmA, tmW;
    {
        const CUtensorMapDataType dt = dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8;
        const long long stream_elems = a.in_stream_elems ? a.in_stream_elems : (long long)a.Win * a.Cin;
        cuuint64_t dims[4] = {(cuuint64_t)a.Cin, (cuuint64_t)a.Win, (cuuint64_t)a.S, (cuuint64_t)(a.r1 - a.r0)};
        cuuint64_t strides[3] = {(cuuint64_t)a.Cin * es, (cuuint64_t)stream_elems * es, (cuuint64_t)a.S * stream_elems * es};
        cuuint32_t box[4] = {(cuuint32_t)p.KB, (cuuint32_t)g.BXP, (cuuint32_t)g.BS, 1}, one[4] = {1, 1, 1, 1};
        if (enc(&tmA, dt, 4, const_cast<void*>(a.in), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(p.swb),
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return cudaErrorNotSupported;
        cuuint64_t wd[3] = {(cuuint64_t)a.Cin, (cuuint64_t)a.Cout, (cuuint64_t)(a.Kh * a.Kw)};
        cuuint64_t wst[2] = {(cuuint64_t)a.Cin * es, (cuuint64_t)a.Cout * a.Cin * es};
        cuuint32_t wbox[3] = {(cuuint32_t)p.KB, (cuuint32_t)(g.N / 2), 1};
        if (enc(&tmW, dt, 3, const_cast<void*>(d_w), wd, wst, wbox, one, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(p.swb),
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return cudaErrorNotSupported;
    }
    const size_t smem = 1024 + (size_t)g.n_a * g.a_bytes + (size_t)g.n_b * t.b_bytes;
    t.smem_bytes = (unsigned int)smem;
    typedef void (*KernelFn)(const CUtensorMap, const CUtensorMap, const PairArgs);
#define IDF_PAIR_SET(DT, KS) {{conv_pair_kernel<DT, KS, 0, 0>, conv_pair_kernel<DT, KS, 0, 1>}, {conv_pair_kernel<DT, KS, 3, 0>, conv_pair_kernel<DT, KS, 3, 1>}}
    static const KernelFn kernels[2][2][2][2] = {{IDF_PAIR_SET(1, 2), IDF_PAIR_SET(1, 4)}, {IDF_PAIR_SET(2, 2), IDF_PAIR_SET(2, 4)}};
#undef IDF_PAIR_SET
    const int ks = p.swb == 128, kw = a.Kw == 3, pl = pooled ? 1 : 0;
    const KernelFn fn = kernels[dtype - 1][ks][kw][pl];
    static bool attr_set[2][2][2][2][64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dtype - 1][ks][kw][pl][dev]) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PAIR_SMEM);
        if (e != cudaSuccess) return e;
        attr_set[dtype - 1][ks][kw][pl][dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * g.clusters)); cfg.blockDim = dim3(PAIR_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = (debug_flags() & IDF_DEBUG_NO_PDL) ? 1 : 2;
    cudaError_t le = cudaLaunchKernelEx(&cfg, fn, tmA, tmW, t);
    if (le != cudaSuccess) return le;
    return cudaGetLastError();
}

}  // namespace idf
