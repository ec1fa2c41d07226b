// 1D nets on the tensor cores: time rows x streams as the M dimension.
//
// A 1D layer has one position per stream and row.  The row-ring kernel takes 128 streams at one time step as its M tile and adds
// tap by tap into the rows of a ring in tensor memory, row after row: few streams leave its tile empty, every row pays the
// hand-over between its roles, and the rows of a push are one serial chain.  Here an M tile is 16 consecutive output rows of 8
// streams, and a tap is a shifted view of the input rows in shared memory:
//   - the input rows a work item reaches (up to four M tiles: 64 output rows, (64 - 1)*stride + Kh input rows, of 8 streams) come
//     by one TMA box per K block; a time row of 8 streams is exactly one swizzle atom, so tap ky of output row t is the atom
//     t*stride + ky: the A descriptor starts ky atoms further on and its 8-row groups are `stride` atoms apart.  No im2col, no
//     strided copies; rows before the block or behind its end are zeros (out-of-range fill);
//   - the weight tile of one (K block, tap) serves all M tiles of the item; it stays in shared memory where all fit, else the
//     tiles stream through a ring (16 KB per 1024 cycles of MMA at 128 outputs and four M tiles);
//   - an accumulator is complete after all taps, so nothing but the rows at the edges of a block touches the ring: rows begun by
//     an earlier block start from what it left there (copied into tensor memory before the first MMA), rows left open are
//     parked.  A launch of one item per stream group reads before it writes inside the CTA; a longer one reads from a copy.
// Roles: warp 0 input rows (TMA), warp 1 MMA, warps 2-17 four epilogue groups (one per M tile, or several to a tile's columns),
// warp 18 weight tiles (TMA).  Bound by operand fetch from shared memory: 128 positions x 128 outputs
// read 128 bytes a cycle at the pipe's full rate, all the shared memory has.
// Measured on B200, 48 streams, 160 samples per push, six layers 1->32->64->64->128->128->128 k9 bf16: 142 -> 52 us per push; one
// 128->128 layer, 1024 streams, 1977 rows: 533 us (row-ring kernel 507).  Emission through staged TMA stores instead of 32 bytes per
// thread: 521 us there, but 61 us per push on the small launches.
#include "../../include/idf.h"
#include "idf_ptx.h"
#include "idf_time_tiles.h"

namespace idf {

int tc_weight_slot(int ky, int kx, int Kh, int stride);

namespace {

constexpr int TIME_GROUPS = 4;
constexpr int TIME_THREADS = 32 * (2 + 4 * TIME_GROUPS + 1);
constexpr int TIME_W_WARP = 2 + 4 * TIME_GROUPS;

struct TimeArgs {
    const void* bias;
    void* ring;
    const void* ring_in;         // where the rows begun by earlier blocks are read: the ring, or a copy of it
    void* out;
    unsigned int* status;
    long long out_row_stride, out_stream_stride, out_row_first;    // elements; row index of visited row 0
    long long out_elems, ring_elems;
    int S, Cout, Kh, stride, relu, shift, out_elem, out_wide;
    int n_rows, done_rel, base_ty, carried;       // visited rows, emitted ones; tap ky of row o reads input row o*stride + ky - base_ty
    int ring_slot0, ring_rows;
    int KB, n_kb, swb, N, n_nt, MT, n_sets, n_w, resident, window;   // window: input rows of an item
    int a_bytes, w_bytes;        // of one K block of a window, of one weight tile (both multiples of 1024 in shared memory)
    int n_g, n_items;            // stream groups; items per channel slice (time tiles x groups)
    int cparts;                  // epilogue groups per M tile
    unsigned int smem_bytes;
};

template <int DT, int KSTEPS>
__global__ void __launch_bounds__(TIME_THREADS, 1)
conv_time_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const __grid_constant__ TimeArgs a)
{
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort, s_issued_a, s_issued_w;
    __shared__ __align__(8) unsigned long long s_bars[4 + 2 * TIME_MAX_W + 3 * 8];

    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t sA = base, sW = sA + 2u * (uint32_t)a.a_bytes;
    const uint32_t bar_a = smem_u32(s_bars), bar_ae = bar_a + 16u;                          // window slots: full, empty
    const uint32_t bar_w = bar_ae + 16u, bar_we = bar_w + 8u * TIME_MAX_W;                  // weight tiles: full, empty
    const uint32_t bar_acc = bar_we + 8u * TIME_MAX_W, bar_free = bar_acc + 64u, bar_init = bar_free + 64u;   // accumulators [set][tile]
    const int nt = blockIdx.x % a.n_nt, first = blockIdx.x / a.n_nt, step = gridDim.x / a.n_nt;
    const int n0 = nt * a.N, n_tiles = a.Kh * a.n_kb;

    if (threadIdx.x == 0) {
        s_abort = 0; s_issued_a = 0; s_issued_w = 0;
        if (!IDF_OK_AT(a.status, sW + (uint32_t)a.n_w * a.w_bytes - smem_u32(smem_raw) - 1u, a.smem_bytes)) s_abort = 1;
        for (int i = 0; i < 2; ++i) { mbar_init(bar_a + 8u * i, 1); mbar_init(bar_ae + 8u * i, 1); }
        for (int i = 0; i < a.n_w; ++i) { mbar_init(bar_w + 8u * i, 1); mbar_init(bar_we + 8u * i, 1); }
        for (int i = 0; i < 8; ++i) { mbar_init(bar_acc + 8u * i, 1); mbar_init(bar_free + 8u * i, 4 * a.cparts); mbar_init(bar_init + 8u * i, 4 * a.cparts); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    volatile int* abort_flag = &s_abort;
    const uint32_t tmem_base = s_tmem_base;
    if (warp != TIME_W_WARP) asm volatile("griddepcontrol.wait;" ::: "memory");             // (the parameters do not depend on earlier kernels)

    if (warp == 0) {
        // ------------------------------ input rows ---------------------------------------------
        if (lane == 0) {
            int t = 0;
            bool ok = true;
            for (int it = first; it < a.n_items && ok; it += step) {
                const int tt = it / a.n_g, g = it - tt * a.n_g;
                for (int kb = 0; kb < a.n_kb; ++kb, ++t) {
                    const uint32_t slot = t & 1;
                    if (!mbar_wait(bar_ae + 8u * slot, (uint32_t)((t >> 1) & 1) ^ 1u, abort_flag)) { ok = false; break; }
                    mbar_expect_tx(bar_a + 8u * slot, (uint32_t)a.window * TIME_SB * a.swb);
                    tma_load_3d(sA + slot * a.a_bytes, &tmA, bar_a + 8u * slot, kb * a.KB, g * TIME_SB, tt * a.MT * TIME_TM * a.stride - a.base_ty);
                }
            }
            s_issued_a = t;
        }
        __syncwarp();
    } else if (warp == TIME_W_WARP) {
        // ------------------------------ weight tiles -------------------------------------------
        if (lane == 0) {
            int t = 0, stage = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (int it = first; it < a.n_items && ok; it += step) {
                for (int kb = 0; kb < a.n_kb && ok; ++kb)
                    for (int ky = 0; ky < a.Kh; ++ky, ++t) {
                        // (ahead of the dependency wait only stages that nobody has used are filled: the wait for a used one is bounded, and it
                        // would last as long as the kernel in front of this one does)
                        if (t == a.n_w) asm volatile("griddepcontrol.wait;" ::: "memory");
                        if (!mbar_wait(bar_we + 8u * stage, ph, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(bar_w + 8u * stage, (uint32_t)a.N * a.swb);
                        // (slot of tap ky in the parameters: see tc_weight_slot)
                        tma_load_3d(sW + (uint32_t)stage * a.w_bytes, &tmW, bar_w + 8u * stage, kb * a.KB, n0, weight_block(ky, a.Kh, a.stride));
                        if (++stage == a.n_w) { stage = 0; ph ^= 1u; }
                    }
                if (a.resident) break;                                                       // loaded once
            }
            s_issued_w = t;
            asm volatile("griddepcontrol.wait;" ::: "memory");
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------ MMA issuer ---------------------------------------------
        const uint64_t desc_hi = make_smem_desc(0, a.swb);
        // 8-row groups of A are `stride` time rows apart
        const uint64_t adesc_hi = (desc_hi & ~((uint64_t)0x3fff << 32)) | ((uint64_t)((8u * a.swb * a.stride) >> 4) << 32);
        const uint32_t idesc = (DT == 1 ? ((1u << 4) | (1u << 7) | (1u << 10)) : ((2u << 4) | (1u << 7) | (1u << 10))) |
                               ((128u >> 4) << 24) | ((uint32_t)(a.N >> 3) << 17);
        const uint32_t atom = (8u * a.swb) >> 4;                                             // one time row, in descriptor units
        const uint32_t tile_units = atom * TIME_TM * a.stride;                               // from one M tile to the next
        const bool issuer = elect_one();
        const int MT = a.MT, N = a.N;
        bool ok = true;
        int ta = 0, ws = 0, use = 0;
        uint32_t wph = 0, init_ph = 0;
        for (int it = first; it < a.n_items && ok; it += step, ++use) {
            const int tt = it / a.n_g;
            const bool carried = a.carried && tt * MT * TIME_TM * a.stride < a.base_ty;
            const int set = a.n_sets == 2 ? use & 1 : 0;
            const uint32_t free_ph = (uint32_t)((a.n_sets == 2 ? use >> 1 : use) & 1) ^ 1u;
            for (int m = 0; m < MT && ok; ++m) {
                ok = mbar_wait(bar_free + 8u * (set * 4 + m), free_ph, abort_flag);
                if (ok && carried) ok = mbar_wait(bar_init + 8u * (set * 4 + m), (init_ph >> set) & 1u, abort_flag);
            }
            if (carried) init_ph ^= 1u << set;
            if (!ok) break;
            bool fresh = !carried;
            for (int kb = 0; kb < a.n_kb && ok; ++kb, ++ta) {
                const uint32_t slot = ta & 1;
                if (!mbar_wait(bar_a + 8u * slot, (uint32_t)((ta >> 1) & 1), abort_flag)) { ok = false; break; }
                uint64_t adesc = adesc_hi | (uint64_t)(((sA + slot * a.a_bytes) & 0x3FFFFu) >> 4);
                for (int ky = 0; ky < a.Kh; ++ky, adesc += atom) {
                    if (!mbar_wait(bar_w + 8u * ws, wph, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    const uint64_t bdesc = desc_hi | (uint64_t)(((sW + (uint32_t)ws * a.w_bytes) & 0x3FFFFu) >> 4);
                    if (issuer) {
                        uint64_t ad = adesc;
                        uint32_t d = tmem_base + (uint32_t)(set * MT * N);
                        if (fresh) for (int m = 0; m < MT; ++m, ad += tile_units, d += N) umma_tile<DT, KSTEPS, true>(d, ad, bdesc, idesc);
                        else for (int m = 0; m < MT; ++m, ad += tile_units, d += N) umma_tile<DT, KSTEPS, false>(d, ad, bdesc, idesc);
                        if (!a.resident) umma_commit(bar_we + 8u * ws);
                        if (ky == a.Kh - 1) umma_commit(bar_ae + 8u * slot);
                    }
                    __syncwarp();
                    fresh = false;
                    if (++ws == a.n_w) { ws = 0; if (!a.resident) wph ^= 1u; }
                }
            }
            if (issuer && ok)
                for (int m = 0; m < MT; ++m) umma_commit(bar_acc + 8u * (set * 4 + m));
            __syncwarp();
        }
    } else {
        // ------------------------------ epilogue -----------------------------------------------
        const int q = warp & 3, grp = (warp - 2) >> 2;
        const int m = grp / a.cparts, part = grp - m * a.cparts;                             // M tile and share of its columns
        const int row = q * 32 + lane, t = row >> 3, s8 = row & 7;                           // TMEM lane = (time row, stream)
        const int nc = a.N / a.cparts, c_lo = part * nc, c_hi = c_lo + nc;
        const int oes = a.out_elem == E_F32 ? 4 : (a.out_elem == E_BF16 ? 2 : 1);
        const uint32_t tlane = tmem_base + ((uint32_t)(q * 32) << 16);
        unsigned char* out = (unsigned char*)a.out;
        uint32_t* ring = (uint32_t*)a.ring;
        const uint32_t* ring_in = (const uint32_t*)a.ring_in;
        bool ok = true;
        int use = 0;
        if (m < a.MT)
            for (int it = first; it < a.n_items && ok; it += step, ++use) {
                const int tt = it / a.n_g, g = it - tt * a.n_g;
                const int set = a.n_sets == 2 ? use & 1 : 0;
                const uint32_t ph = (uint32_t)((a.n_sets == 2 ? use >> 1 : use) & 1);
                const uint32_t bar = 8u * (set * 4 + m);
                const uint32_t tcol = tlane + (uint32_t)((set * a.MT + m) * a.N);
                const int o = (tt * a.MT + m) * TIME_TM + t, s = g * TIME_SB + s8;
                const bool valid = o < a.n_rows && s < a.S, emit = o < a.done_rel;
                const long long ring_at = ((long long)((a.ring_slot0 + o) % a.ring_rows) * a.S + s) * a.Cout + n0;
                if (a.carried && tt * a.MT * TIME_TM * a.stride < a.base_ty) {
                    // the item holds rows begun by an earlier block: accumulators start from the ring (zero for the other rows)
                    const bool have = valid && o * a.stride < a.base_ty && IDF_OK_AT(a.status, ring_at + c_hi - 1, a.ring_elems);
                    for (int c = c_lo; c < c_hi; c += 16) {
                        uint32_t v[16];
#pragma unroll
                        for (int j = 0; j < 16; ++j) v[j] = 0u;
                        if (have) {
                            ld_global_v8(ring_in + ring_at + c, *(uint32_t(*)[8])v);
                            ld_global_v8(ring_in + ring_at + c + 8, *(uint32_t(*)[8])(v + 8));
                        }
                        __syncwarp();
                        tmem_st16(tcol + c, v);
                    }
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar_init + bar);
                }
                int got = 1;
                if (lane == 0) got = mbar_wait(bar_acc + bar, ph, abort_flag) ? 1 : 0;
                if (!__shfl_sync(0xffffffffu, got, 0)) { ok = false; break; }
                tc_fence_after();
                const long long out_at = (a.out_row_first + o) * a.out_row_stride + (long long)s * a.out_stream_stride + n0;
                const bool fine = valid && (emit ? IDF_OK_AT(a.status, out_at, a.out_elems - c_hi + 1) : IDF_OK_AT(a.status, ring_at, a.ring_elems - c_hi + 1));
                for (int c = c_lo; c < c_hi; c += 32) {
                    uint32_t v[32];
                    const bool two = c + 16 < c_hi;
                    __syncwarp();
                    if (two) tmem_ld<32>(tcol + c, v);
                    else tmem_ld<16>(tcol + c, v);
                    if (!fine) continue;
                    if (!emit) {
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (j < 2 || two) st_global_v8(ring + ring_at + c + 8 * j, *(uint32_t(*)[8])(v + 8 * j));
                        continue;
                    }
                    unsigned char* d = out + (out_at + c) * oes;
                    const uint32_t* b = a.bias ? (const uint32_t*)a.bias + n0 + c : nullptr;
                    if (DT == 2) {
                        uint32_t pk[8];
                        pack_i8<16>(v, (const int*)b, a.relu, a.shift, pk);
                        if (two) pack_i8<16>(v + 16, b ? (const int*)b + 16 : nullptr, a.relu, a.shift, pk + 4);
                        if (two && a.out_wide) st_global_v8(d, *(uint32_t(*)[8])pk);
                        else { st_global_v4(d, pk); if (two) st_global_v4(d + 16, pk + 4); }
                    } else if (a.out_elem == E_BF16) {
                        emit16f<E_BF16>(v, (const float*)b, a.relu, d, a.out_wide);
                        if (two) emit16f<E_BF16>(v + 16, b ? (const float*)b + 16 : nullptr, a.relu, d + 32, a.out_wide);
                    } else {
                        emit16f<E_F32>(v, (const float*)b, a.relu, d, a.out_wide);
                        if (two) emit16f<E_F32>(v + 16, b ? (const float*)b + 16 : nullptr, a.relu, d + 64, a.out_wide);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_free + bar);
            }
    }

    tc_fence_before();
    __syncthreads();
    if (s_abort) {
        if (threadIdx.x == 0) {
            // this CTA's own copies must land before its shared memory is given back (bounded)
            for (int k = 0; k < 2 && k < s_issued_a; ++k) {
                const int t = s_issued_a - 1 - k;
                for (uint32_t i = 0; i < 4096 && !mbar_try_wait(bar_a + 8u * (t & 1), (uint32_t)((t >> 1) & 1)); ++i) __nanosleep(64);
            }
            for (int k = 0; k < a.n_w && k < s_issued_w; ++k) {
                const int t = s_issued_w - 1 - k;
                for (uint32_t i = 0; i < 4096 && !mbar_try_wait(bar_w + 8u * (t % a.n_w), (uint32_t)((t / a.n_w) & 1)); ++i) __nanosleep(64);
            }
            atomicOr(a.status, 1u);
        }
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

}  // namespace

bool time_make_plan(int dtype, int Cin, int Cout, int Kh, int stride, TimePlan* p)
{
    *p = TimePlan{};
    if (dtype != 1 && dtype != 2) return false;
    const int es = dtype == 1 ? 2 : 1, row = Cin * es;
    if (!(row == 32 || row == 64 || (row >= 128 && row % 128 == 0))) return false;
    if (Cout % 16 != 0 || Kh > 64 || stride > 16) return false;
    p->swb = row >= 128 ? 128 : row;
    p->KB = p->swb / es;
    p->n_kb = Cin / p->KB;
    // the smallest item (one M tile, 16 outputs) must fit
    const size_t a1 = ((size_t)((TIME_TM - 1) * stride + Kh) * TIME_SB * p->swb + 1023) / 1024 * 1024;
    if ((TIME_TM - 1) * stride + Kh > 256 || 1024 + 2 * a1 + 3 * (size_t)128 * p->swb > TIME_SMEM) return false;
    p->ok = 1;
    return true;
}

// cudaErrorNotSupported: the launch cannot take this path (alignment, a tensor map the driver rejects).
cudaError_t launch_conv_time(const ConvArgs& a, const TimePlan& p, int dtype, const void* d_w, cudaStream_t st)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc || !p.ok || a.pool_fused || a.o_end <= a.o_begin || a.r1 <= a.r0) return cudaErrorNotSupported;
    if (((uintptr_t)a.in & 15) != 0 || ((uintptr_t)a.out & 15) != 0) return cudaErrorNotSupported;
    const int es = dtype == 1 ? 2 : 1;
    TimeArgs t{};
    t.bias = a.bias; t.ring = a.ring; t.ring_in = a.ring; t.out = a.out; t.status = a.status;
    t.out_row_stride = a.out_row_stride; t.out_stream_stride = a.out_stream_stride; t.out_row_first = a.o_begin - a.out_row_base;
    t.out_elems = a.out_elems; t.ring_elems = a.ring_elems;
    t.S = a.S; t.Cout = a.Cout; t.Kh = a.Kh; t.stride = a.stride; t.relu = a.relu; t.shift = a.shift; t.out_elem = a.out_elem;
    t.n_rows = (int)(a.o_end - a.o_begin); t.done_rel = (int)(a.done_end - a.o_begin);
    t.base_ty = (int)(a.r0 + a.pad - a.o_begin * a.stride); t.carried = a.r0 > 0;
    t.ring_slot0 = (int)(a.o_begin % a.ring_rows); t.ring_rows = a.ring_rows;
    t.KB = p.KB; t.n_kb = p.n_kb; t.swb = p.swb;
    t.n_g = (a.S + TIME_SB - 1) / TIME_SB;
    const TimeTiles tiles = time_tiles(dtype, a.S, t.n_rows, a.Cout, a.Kh, a.stride, p.swb, p.n_kb);
    const int N = tiles.N, MT = tiles.MT;
    t.N = N; t.n_nt = a.Cout / N; t.MT = MT; t.window = tiles.window; t.resident = tiles.resident; t.n_w = tiles.n_w;
    t.a_bytes = (int)tiles.a_bytes; t.w_bytes = (int)tiles.w_bytes;
    t.n_sets = 2 * MT * N <= 512 ? 2 : 1;
    t.cparts = tiles.cparts;
    t.out_wide = ((uintptr_t)a.out & 31) == 0 && tiles.wide;
    const int n_tt = (t.n_rows + MT * TIME_TM - 1) / (MT * TIME_TM);
    if ((long long)n_tt * t.n_g > 0x3fffffffLL) return cudaErrorNotSupported;
    t.n_items = n_tt * t.n_g;
    if (n_tt > 1 && t.carried) {
        // rows begun by an earlier block and rows left open by this one may share a ring slot and lie in different CTAs
        if (!a.ring_scratch) return cudaErrorNotSupported;
        cudaError_t ce = launch_ring_copy(a.ring_scratch, a.ring, (long long)a.ring_rows * a.S * a.Cout, st);
        if (ce != cudaSuccess) return ce;
        t.ring_in = a.ring_scratch;
    }
    CUtensorMap tmA, tmW;
    {
        const CUtensorMapDataType dt = dtype == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_UINT8;
        cuuint64_t dims[3] = {(cuuint64_t)a.Cin, (cuuint64_t)a.S, (cuuint64_t)(a.r1 - a.r0)};
        cuuint64_t strides[2] = {(cuuint64_t)a.Cin * es, (cuuint64_t)a.S * a.Cin * es};
        cuuint32_t box[3] = {(cuuint32_t)p.KB, (cuuint32_t)TIME_SB, (cuuint32_t)t.window}, one[3] = {1, 1, 1};
        if (enc(&tmA, dt, 3, const_cast<void*>(a.in), dims, strides, box, one, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(p.swb),
                CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return cudaErrorNotSupported;
        cuuint64_t wd[3] = {(cuuint64_t)a.Cin, (cuuint64_t)a.Cout, (cuuint64_t)a.Kh};
        cuuint64_t wst[2] = {(cuuint64_t)a.Cin * es, (cuuint64_t)a.Cout * a.Cin * es};
        cuuint32_t wbox[3] = {(cuuint32_t)p.KB, (cuuint32_t)N, 1};
        if (enc(&tmW, dt, 3, const_cast<void*>(d_w), wd, wst, wbox, one, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(p.swb),
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) return cudaErrorNotSupported;
    }
    const size_t smem = 1024 + 2 * (size_t)t.a_bytes + (size_t)t.n_w * t.w_bytes;
    t.smem_bytes = (unsigned int)smem;
    int per_nt = 148 / t.n_nt;
    if (per_nt < 1) per_nt = 1;
    if (per_nt > t.n_items) per_nt = t.n_items;
    const int ks = p.swb == 32 ? 0 : (p.swb == 64 ? 1 : 2);
    typedef void (*KernelFn)(const CUtensorMap, const CUtensorMap, const TimeArgs);
    static const KernelFn kernels[2][3] = {{conv_time_kernel<1, 1>, conv_time_kernel<1, 2>, conv_time_kernel<1, 4>},
                                           {conv_time_kernel<2, 1>, conv_time_kernel<2, 2>, conv_time_kernel<2, 4>}};
    const KernelFn fn = kernels[dtype - 1][ks];
    static bool attr_set[2][3][64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dtype - 1][ks][dev]) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TIME_SMEM);
        if (e != cudaSuccess) return e;
        attr_set[dtype - 1][ks][dev] = true;
    }
    return launch_pdl(fn, (unsigned)(per_nt * t.n_nt), TIME_THREADS, smem, st, tmA, tmW, t);
}

}  // namespace idf
