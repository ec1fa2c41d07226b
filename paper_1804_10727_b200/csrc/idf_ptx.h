// Device helpers shared by the tensor-core kernels: mbarriers with bounded waits, TMA copies, tcgen05 instructions,
// shared-memory descriptors, tensor-memory loads and stores.
#pragma once
#include "idf_internal.h"

#include <cuda.h>
#include <mutex>

namespace idf {

namespace {

constexpr uint32_t WAIT_LIMIT = 1u << 22;
constexpr size_t SMEM_LIMIT = 232448;        // 227 KB per CTA

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Non-blocking look at a barrier phase (the result may be consumed much later: the round trip to the
// barrier then overlaps whatever is issued in between).
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// Bounded wait: false if the limit ran out or another role has given up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 31u) == 31u) {
            if (*abort_flag) return false;
            __nanosleep(32);
        }
    }
    *abort_flag = 1;
    return false;
}
// The same for roles that are not on the critical path (producer waiting for a free stage, epilogue
// waiting for a finished row): sleep between polls, so the polling warp leaves the issue slots of its
// scheduler to the MMA-issuing warp that shares it.
__device__ __forceinline__ bool mbar_wait_relaxed(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    for (uint32_t i = 0; i < WAIT_LIMIT; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        __nanosleep(200);
        if ((i & 15u) == 15u && *abort_flag) return false;
    }
    *abort_flag = 1;
    return false;
}

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2, int c3)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
        ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}

// true in exactly one lane of a converged warp
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
    return pred != 0;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// All K steps of one shared-memory tile pair in one go: the descriptors move 32 bytes (2 units of 16 B) per step inside the
// swizzled row.  FRESH: the first step overwrites the accumulator, else every step adds to it.
#define IDF_MMA_STEP(kind, i, p) "add.s64 a1, %1, " #i ";\n\tadd.s64 b1, %2, " #i ";\n\t" \
                                 "tcgen05.mma.cta_group::1.kind::" kind " [%0], a1, b1, %3, " p ";\n\t"
#define IDF_MMA_KIND(kind)  \
    if (KSTEPS == 1)  \
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 a1, b1;\n\tsetp.eq.b32 p, 0, 0;\n\tsetp.eq.b32 q, %4, 0;\n\t"  \
                     IDF_MMA_STEP(kind, 0, "q") "}"  \
                     ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(FRESH ? 1 : 0) : "memory");  \
    else if (KSTEPS == 2)  \
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 a1, b1;\n\tsetp.eq.b32 p, 0, 0;\n\tsetp.eq.b32 q, %4, 0;\n\t"  \
                     IDF_MMA_STEP(kind, 0, "q") IDF_MMA_STEP(kind, 2, "p") "}"  \
                     ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(FRESH ? 1 : 0) : "memory");  \
    else if (KSTEPS == 3)  \
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 a1, b1;\n\tsetp.eq.b32 p, 0, 0;\n\tsetp.eq.b32 q, %4, 0;\n\t"  \
                     IDF_MMA_STEP(kind, 0, "q") IDF_MMA_STEP(kind, 2, "p") IDF_MMA_STEP(kind, 4, "p") "}"  \
                     ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(FRESH ? 1 : 0) : "memory");  \
    else  \
        asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 a1, b1;\n\tsetp.eq.b32 p, 0, 0;\n\tsetp.eq.b32 q, %4, 0;\n\t"  \
                     IDF_MMA_STEP(kind, 0, "q") IDF_MMA_STEP(kind, 2, "p") IDF_MMA_STEP(kind, 4, "p") IDF_MMA_STEP(kind, 6, "p") "}"  \
                     ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "n"(FRESH ? 1 : 0) : "memory");
template <int DT, int KSTEPS, bool FRESH = false>
__device__ __forceinline__ void umma_tile(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc)
{
    if (DT == 1) { IDF_MMA_KIND("f16") } else { IDF_MMA_KIND("i8") }
}
#undef IDF_MMA_KIND
#undef IDF_MMA_STEP
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Position of tap row ky inside a stacked weight tile.  The Kh blocks of Ntile rows are ordered so
// that the taps one input row uses (ky = ph, ph+stride, ...) sit next to each other with ky
// descending: their output rows ascend, and so do the ring slots (TMEM columns) they accumulate
// into, which lets one MMA of N = (taps)*Ntile serve several ring rows at once.
__host__ __device__ __forceinline__ int weight_block(int ky, int Kh, int stride)
{
    const int ph = ky % stride;
    int off = 0;
    for (int p = 0; p < ph; ++p) off += (Kh - p + stride - 1) / stride;
    const int cnt = (Kh - ph + stride - 1) / stride;
    return off + cnt - 1 - ky / stride;
}

// shared-memory matrix descriptor, K-major operand in the canonical swizzled layout:
// rows of `swb` bytes, 8-row groups `8*swb` bytes apart
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t swb)
{
    const uint64_t layout = swb == 128 ? 2 : (swb == 64 ? 4 : 6);
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)1 << 16;                           // leading-dimension offset: unused for swizzled K-major
    d |= (uint64_t)((8u * swb) >> 4) << 32;           // stride-dimension offset between 8-row groups
    d |= (uint64_t)1 << 46;                           // descriptor version of this architecture
    d |= layout << 61;
    return d;
}


// TMEM loads of W consecutive accumulator columns of this thread's lane.  The load fills its registers asynchronously until
// the wait; both are one statement, so that the compiler can place nothing (a move, a spill) between them.
template <int W>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* v)
{
    if (W == 16) {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
            "tcgen05.wait::ld.sync.aligned;"
            : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7]),
              "=&r"(v[8]), "=&r"(v[9]), "=&r"(v[10]), "=&r"(v[11]), "=&r"(v[12]), "=&r"(v[13]), "=&r"(v[14]),
              "=&r"(v[15])
            : "r"(taddr) : "memory");
    } else {
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
            "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
            "tcgen05.wait::ld.sync.aligned;"
            : "=&r"(v[0]), "=&r"(v[1]), "=&r"(v[2]), "=&r"(v[3]), "=&r"(v[4]), "=&r"(v[5]), "=&r"(v[6]), "=&r"(v[7]),
              "=&r"(v[8]), "=&r"(v[9]), "=&r"(v[10]), "=&r"(v[11]), "=&r"(v[12]), "=&r"(v[13]), "=&r"(v[14]),
              "=&r"(v[15]), "=&r"(v[16 % W]), "=&r"(v[17 % W]), "=&r"(v[18 % W]), "=&r"(v[19 % W]), "=&r"(v[20 % W]),
              "=&r"(v[21 % W]), "=&r"(v[22 % W]), "=&r"(v[23 % W]), "=&r"(v[24 % W]), "=&r"(v[25 % W]),
              "=&r"(v[26 % W]), "=&r"(v[27 % W]), "=&r"(v[28 % W]), "=&r"(v[29 % W]), "=&r"(v[30 % W]),
              "=&r"(v[31 % W])
            : "r"(taddr) : "memory");
    }
}
template <int W>
__device__ __forceinline__ void tmem_st_zero(uint32_t taddr)
{
    const uint32_t z = 0;
    if (W == 16)
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};"
            ::"r"(taddr), "r"(z) : "memory");
    else
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, "
            "%1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1, %1};"
            ::"r"(taddr), "r"(z) : "memory");
}


// 16 words of this thread's lane into 16 consecutive columns
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap* tm, uint32_t src, int c0, int c1, int c2, int c3)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(tm), "r"(src), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void named_bar_sync(int id, int count)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
// barrier among `count` threads that also tells everyone whether all of them passed `pred`
__device__ __forceinline__ bool named_bar_and(int id, int count, bool pred)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %3, 0;\n\t"
        "bar.red.and.pred q, %1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"(id), "r"(count), "r"((uint32_t)pred) : "memory");
    return r != 0;
}

// Ring rows in global memory are read and written 32 bytes per thread and instruction: a thread's run of channels
// is its own, so narrower accesses would touch every 32-byte sector of the run twice.
__device__ __forceinline__ void ld_global_v8(const void* p, uint32_t (&v)[8])
{
    asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "l"(p));
}
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t (&v)[8])
{
    asm volatile("st.global.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};"
                 :: "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "l"(p) : "memory");
}

// W int32 sums -> W / 4 words of four int8: shift with rounding, ReLU and clamp.  The layers that end here are bound by this
// arithmetic, so it is kept to (two for the shift and) one instruction per value: the saturating pack of two values clamps to
// [-128, 127], and ReLU is the sign bytes (one byte permute) masked out of four values at once.  (A byte-wise minimum on top of an
// unsigned pack costs three times as much: it has no instruction of its own.)
template <int W, bool SHIFT, bool BIAS>
__device__ __forceinline__ void pack_i8_as(const uint32_t* v, const int* bias_c, int relu, int rnd, int shift, uint32_t* pk)
{
#pragma unroll
    for (int j = 0; j < W / 4; ++j) {
        int t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) t[u] = (int)v[4 * j + u];
        if (BIAS) {
            const int4 b4 = ((const int4*)bias_c)[j];
            t[0] += b4.x; t[1] += b4.y; t[2] += b4.z; t[3] += b4.w;
        }
        if (SHIFT) {
#pragma unroll
            for (int u = 0; u < 4; ++u) t[u] = (t[u] + rnd) >> shift;
        }
        uint32_t hi2;
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(hi2) : "r"(t[3]), "r"(t[2]));
        asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(pk[j]) : "r"(t[1]), "r"(t[0]), "r"(hi2));
    }
    if (relu) {
#pragma unroll
        for (int j = 0; j < W / 4; ++j) {
            uint32_t neg;
            asm("prmt.b32 %0, %1, 0, 0xBA98;" : "=r"(neg) : "r"(pk[j]));         // 0xff where a byte is negative
            pk[j] &= ~neg;
        }
    } else {
#pragma unroll
        for (int j = 0; j < W / 4; ++j) pk[j] = __vmaxs4(pk[j], 0x81818181u);    // symmetric: not below -127
    }
}
template <int W>
__device__ __forceinline__ void pack_i8(const uint32_t* v, const int* bias_c, int relu, int shift, uint32_t* pk)
{
    const int rnd = shift > 0 ? 1 << (shift - 1) : 0;
    if (bias_c) pack_i8_as<W, true, true>(v, bias_c, relu, rnd, shift, pk);
    else if (shift > 0) pack_i8_as<W, true, false>(v, bias_c, relu, rnd, shift, pk);
    else pack_i8_as<W, false, false>(v, bias_c, relu, rnd, shift, pk);
}

__device__ __forceinline__ void st_global_v4(void* p, const uint32_t* v)
{
    asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void st_global_32(void* p, const uint32_t* v, int wide)
{
    if (wide) st_global_v8(p, *(const uint32_t(*)[8])v);
    else { st_global_v4(p, v); st_global_v4((unsigned char*)p + 16, v + 4); }
}

// f(c + b) of W fp32 sums: W / 2 words of bf16 pairs, or W of fp32
template <int W>
__device__ __forceinline__ void pack_f(const uint32_t* v, const float* bias_c, int bf16, int relu, uint32_t* pk)
{
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
    if (bf16) {
        if (relu) {
#pragma unroll
            for (int j = 0; j < W / 2; ++j) asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(f[2 * j + 1]), "f"(f[2 * j]));
        } else {
#pragma unroll
            for (int j = 0; j < W / 2; ++j) asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(pk[j]) : "f"(f[2 * j + 1]), "f"(f[2 * j]));
        }
    } else {
#pragma unroll
        for (int j = 0; j < W; ++j) pk[j] = __float_as_uint(relu ? fmaxf(f[j], 0.f) : f[j]);
    }
}
// ... of 16, straight to global memory (wide: dst is 32-byte aligned)
template <int OUT>
__device__ __forceinline__ void emit16f(const uint32_t* v, const float* bias_c, int relu, unsigned char* dst, int wide)
{
    uint32_t pk[16];
    pack_f<16>(v, bias_c, OUT == E_BF16, relu, pk);
    st_global_32(dst, pk, wide);
    if (OUT != E_BF16) st_global_32(dst + 32, pk + 8, wide);
}
// element-wise maximum of two 32-bit words holding OP = 0: two bf16, 1: one fp32, 2: four int8
template <int OP>
__device__ __forceinline__ uint32_t word_max(uint32_t x, uint32_t y)
{
    if (OP == 0) { uint32_t r; asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(y)); return r; }
    if (OP == 1) return __float_as_uint(fmaxf(__uint_as_float(x), __uint_as_float(y)));
    // two bytes at a time: of a 16-bit maximum the upper byte is right whatever the lower bytes are
    uint32_t h, l, r;
    asm("max.s16x2 %0, %1, %2;" : "=r"(h) : "r"(x), "r"(y));
    asm("max.s16x2 %0, %1, %2;" : "=r"(l) : "r"(x << 8), "r"(y << 8));
    asm("prmt.b32 %0, %1, %2, 0x3715;" : "=r"(r) : "r"(h), "r"(l));
    return r;
}
template <int DT> struct Acc;
template <> struct Acc<1> { typedef float S; };
template <> struct Acc<2> { typedef int S; };

// ---- host side: tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qr) == cudaSuccess &&
            qr == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    });
    return fn;
}

CUtensorMapSwizzle swizzle_of(int swb)
{
    return swb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (swb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}

}  // namespace

}  // namespace idf
