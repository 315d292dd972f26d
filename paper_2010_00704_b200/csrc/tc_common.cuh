// Device helpers shared by the tcgen05 engines: mbarrier waits with a bound and back-off,
// tcgen05 instruction wrappers (MMA from shared / tensor memory, commit, ld, st, fences),
// cp.async staging, shared-memory descriptors and the expansions of sign bits to 4-bit codes.
#pragma once
#include "bcnn_common.cuh"
#include <cuda_fp16.h>

namespace bcnn {
namespace tc {

constexpr int BM = 128;                   // rows of an output tile = tensor-memory lanes
constexpr int ROWB = 128;                 // bytes of one expanded row per stage (= 256 elements of K)
constexpr uint32_t WAIT_LIMIT = 1u << 17; // polls before a wait gives up
// upper bound (ns) for which one try_wait may suspend the thread
constexpr uint32_t SUSPEND_HINT_NS = 20000;
constexpr uint32_t SLEEP_NS = 100;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
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
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(SUSPEND_HINT_NS) : "memory");
    return ok != 0;
}
// Bounded wait with back-off.  A polling warp competes with the MMA-issuing warp for issue
// slots, so after a first failed poll the waiter sleeps between polls.  The polling loop is kept
// out of line: the common case is one successful try_wait.
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err, int code,
                                                   uint32_t limit = WAIT_LIMIT)
{
    for (uint32_t it = 0; it < limit; ++it) {
        __nanosleep(SLEEP_NS);
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 255u && *abort_flag) return false;
    }
    *abort_flag = 1;
    if (err) atomicCAS(err, 0, code);
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err, int code,
                                          uint32_t limit = WAIT_LIMIT)
{
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, err, code, limit);
}
// Whole-warp wait: one try_wait per lane and a vote in the common case.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err, int code,
                                               uint32_t limit = WAIT_LIMIT)
{
    bool ok = mbar_try_wait(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    if (!ok) ok = mbar_wait_slow(bar, parity, abort_flag, err, code, limit);
    return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ void mbar_arrive_pred(uint32_t bar, uint32_t pred)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
        "@q mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
        ::"r"(bar), "r"(pred) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool elect_one()
{
    uint32_t pred = 0;
    asm volatile("{\n\t.reg .b32 rx;\n\t.reg .pred px;\n\telect.sync rx|px, 0xffffffff;\n\tselp.u32 %0, 1, 0, px;\n\t}" : "=r"(pred));
    return pred != 0;
}
// 4-bit operands (kind::mxf4: e2m1 x e2m1 with block scales, fp32 accumulators): 64 elements of K per instruction at twice
// the byte kinds' rate - 8.80 POP/s against 4.57 of kind::i8 with A in tensor memory, N = 64 .. 256 (8.54 at N = 32).
// Sums of products +-2 are integers far below 2^24: exact (checked against popcounts up to K = 2^20, all-ones included).
// Every block scale is 1.0 (e8m0 127): the SF_COLS columns at `sf` hold that byte in all 128 lanes, so that every scale
// address an instruction of any width forms there reads 1.0.
constexpr uint32_t SF_COLS = 8;
constexpr uint32_t SF_ONES = 0x7F7F7F7Fu;
__device__ __forceinline__ void tc_mma_f4_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi,
                                             uint32_t idesc, uint32_t sf, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], db, %4, [%5], [%5], p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(sf), "r"(accumulate)
        : "memory");
}
// e2m1 A and B (K-major), e8m0 scales, M = 128, N = n, K = 64.
__device__ __forceinline__ constexpr uint32_t make_idesc_f4(int n)
{
    return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((uint32_t)(BM >> 7) << 27);
}
// 32 columns of this warp's 32 lanes <- 32 registers; returns once the store has completed.
__device__ __forceinline__ void tc_st32(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n\t"
        "tcgen05.wait::st.sync.aligned;"
        ::"r"(taddr),
          "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
// Same without the completion wait, for several stores followed by one tc_wait_st().
__device__ __forceinline__ void tc_st32_nowait(uint32_t taddr, const uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
        "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr),
          "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]),
          "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]),
          "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}
// 16 columns of this warp's 32 lanes <- 16 registers.
__device__ __forceinline__ void tc_st16_nowait(uint32_t taddr, const uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
        ::"r"(taddr),
          "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
          "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
        : "memory");
}
// 8 columns of this warp's 32 lanes <- 8 registers.
__device__ __forceinline__ void tc_st8_nowait(uint32_t taddr, const uint32_t (&v)[8])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ void tc_st4_nowait(uint32_t taddr, const uint32_t (&v)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};"
                 ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
}
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// 32 accumulator columns of this warp's 32 rows.  The load and its completion wait are one asm
// statement so that no use of the destination registers can be scheduled between them.
__device__ __forceinline__ void tc_ld32(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}

// Without the wait, for several loads followed by one tc_wait_ld() (and pin_regs on each destination, tc_slot.cuh).
__device__ __forceinline__ void tc_ld32_nowait(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}

// K-major tile, 128-byte rows, 128-byte swizzle, 8-row groups 1024 bytes apart, descriptor version 1.
__device__ __forceinline__ uint64_t make_desc(uint32_t saddr)
{
    const uint32_t lo = ((saddr & 0x3FFFFu) >> 4) | (1u << 16);
    const uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
    return (static_cast<uint64_t>(hi) << 32) | lo;
}
__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---- 4-bit operands.  Nibble i of word j of an expanded 32-bit group carries bit 4i + j.  Activations are unsigned
// ({0, 2^j / 2}: e2m1 codes 1, 2, 4 are 0.5, 1, 2; bit 3 goes to code 4 as well), weights signed (+-4, +-2, +-1, +-1), so
// that every product with a set activation bit is +-2 and with S = sum over set activation bits of the weight signs
//   accumulator = 2 S,   sum a*g = accumulator + K - 2 popc(G):
// one constant per output channel.  Five logic operations per
// activation word.
__device__ __forceinline__ void expand_a4(uint32_t w, uint32_t *v)
{
    v[0] = w & 0x11111111u;
    v[1] = w & 0x22222222u;
    v[2] = w & 0x44444444u;
    v[3] = (w >> 1) & 0x44444444u;
}
// e2m1 sign bit = the weight bit's complement: (w at bit 3) ^ (magnitude code | 8)
__device__ __forceinline__ uint4 expand_w4(uint32_t w)
{
    return make_uint4(((w << 3) & 0x88888888u) ^ 0xEEEEEEEEu, ((w << 2) & 0x88888888u) ^ 0xCCCCCCCCu,
                      ((w << 1) & 0x88888888u) ^ 0xAAAAAAAAu, (w & 0x88888888u) ^ 0xAAAAAAAAu);
}
// fp32 sums of integers below 2^22 as integers: with INT_BIAS = 1.5 * 2^23 added, the value sits in the low mantissa bits
// (an addition each in fp32 and integer, against a conversion at a quarter of the rate).
constexpr float INT_BIAS = 12582912.0f;
__device__ __forceinline__ int int_of_biased(uint32_t bits) { return (int)(bits - 0x4B400000u); }
__device__ __forceinline__ uint32_t fadd_bits(uint32_t a, uint32_t b)
{
    return __float_as_uint(__fadd_rn(__uint_as_float(a), __uint_as_float(b)));
}
// Output word of 32 accumulator columns: bit = (v + c >= 0) for exact integers v and c, with 2 c + 1 of column i at
// table + 4 i.  2 (v + c) + 1 is an odd integer, so saturated to [0, 1] it is the bit; two chains of 16 Horner steps collect
// the bits as fp32 integers below 2^16.  All of it runs on the fp32 pipe at full rate - an addition and a shift per column
// would take two slots of the logic pipe, which the activations' expansion needs.
__device__ __forceinline__ uint32_t threshold_word(const uint32_t (&v)[32], uint32_t table)
{
    float lo = 0.0f, hi = 0.0f;
#pragma unroll
    for (int i4 = 3; i4 >= 0; --i4) {
        const uint4 a = ld_shared_v4(table + 16u * i4), b = ld_shared_v4(table + 64u + 16u * i4);
        const uint32_t ca[4] = {a.x, a.y, a.z, a.w}, cb[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            lo = fmaf(lo, 2.0f, __saturatef(fmaf(__uint_as_float(v[4 * i4 + i]), 2.0f, __uint_as_float(ca[i]))));
            hi = fmaf(hi, 2.0f, __saturatef(fmaf(__uint_as_float(v[16 + 4 * i4 + i]), 2.0f, __uint_as_float(cb[i]))));
        }
    }
    // integers below 2^16 in the low mantissa bits of 2^23 + x
    return __byte_perm(__float_as_uint(lo + 8388608.0f), __float_as_uint(hi + 8388608.0f), 0x5410);
}
// Two words of 64 consecutive columns at once: four chains instead of two, the next eight columns' constants on their way.
__device__ __forceinline__ void threshold_words(const uint32_t (&v)[2][32], uint32_t table, uint32_t &w0, uint32_t &w1)
{
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    uint4 c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = ld_shared_v4(table + 64u * q + 48u);
#pragma unroll
    for (int i4 = 3; i4 >= 0; --i4) {
        uint32_t cc[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            cc[q][0] = c[q].x; cc[q][1] = c[q].y; cc[q][2] = c[q].z; cc[q][3] = c[q].w;
            if (i4) c[q] = ld_shared_v4(table + 64u * q + 16u * (i4 - 1));
        }
#pragma unroll
        for (int i = 3; i >= 0; --i) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                acc[q] = fmaf(acc[q], 2.0f, __saturatef(fmaf(__uint_as_float(v[q >> 1][16 * (q & 1) + 4 * i4 + i]), 2.0f, __uint_as_float(cc[q][i]))));
        }
    }
    w0 = __byte_perm(__float_as_uint(acc[0] + 8388608.0f), __float_as_uint(acc[1] + 8388608.0f), 0x5410);
    w1 = __byte_perm(__float_as_uint(acc[2] + 8388608.0f), __float_as_uint(acc[3] + 8388608.0f), 0x5410);
}
// ... and 32 exact integers v + c, with c + INT_BIAS of column i at table + 4 i.
__device__ __forceinline__ void biased_ints(const uint32_t (&v)[32], uint32_t table, int (&o)[32])
{
#pragma unroll
    for (int i4 = 0; i4 < 8; ++i4) {
        const uint4 c = ld_shared_v4(table + 16u * i4);
        o[4 * i4] = int_of_biased(fadd_bits(v[4 * i4], c.x));
        o[4 * i4 + 1] = int_of_biased(fadd_bits(v[4 * i4 + 1], c.y));
        o[4 * i4 + 2] = int_of_biased(fadd_bits(v[4 * i4 + 2], c.z));
        o[4 * i4 + 3] = int_of_biased(fadd_bits(v[4 * i4 + 3], c.w));
    }
}
// What an epilogue's column table holds for the constant c (MODE 0: int32, 1: packed, 2: module).
template <int MODE> __device__ __forceinline__ uint32_t table_entry(int c)
{
    return __float_as_uint(MODE == 0 ? (float)c + INT_BIAS : (MODE == 1 ? (float)(2 * c + 1) : (float)c));
}

// K word e (0..7) of a 256-bit stage of a weight row: 16 bytes of a 128-byte-swizzled row; zeros where not live
__device__ __forceinline__ void expand_store_w4(uint32_t w, bool live, uint32_t row_addr, int xr, int e)
{
    const uint4 o = live ? expand_w4(w) : make_uint4(0u, 0u, 0u, 0u);
    st_shared_v4(row_addr + (uint32_t)((e ^ xr) << 4), o.x, o.y, o.z, o.w);
}
// unit scales into this warp's 32 lanes (the four warps of a group cover all lanes); returns once they are written
__device__ __forceinline__ void write_unit_scales(uint32_t taddr)
{
    const uint32_t c8[8] = {SF_ONES, SF_ONES, SF_ONES, SF_ONES, SF_ONES, SF_ONES, SF_ONES, SF_ONES};
    tc_st8_nowait(taddr, c8);
    tc_wait_st();
}

// ---- implicit-im2col gather -----------------------------------------------------------------------
// K is cut into units of GW words that never straddle a tap: GW = 4 (one 16-byte copy) when a pixel
// is a multiple of four words, 2 when it is even, else 1.  The unit table holds, per unit, the word
// offset from the row's top-left input pixel and its tap; a row carries the word offset of its top-left input pixel and the mask of its taps that
// fall inside the image, so one unit costs a mask test, an add and a copy with zero fill.
__host__ __device__ __forceinline__ int gather_width(int cw) { return (cw & 3) == 0 ? 4 : ((cw & 1) == 0 ? 2 : 1); }

template <int V> struct IntC { static constexpr int value = V; };

// Advance of a CTA from one of its row tiles to the next: a constant number of rows, split once into
// whole images, output rows and output columns, so that a row's coordinates follow by carries.
struct TileStep {
    uint32_t rows;
    int db, doh, dow;
    uint32_t pat;            // bit r*kw for every kernel row r
    bool pointwise;          // 1x1, stride 1, no padding: row m reads input pixel m, no coordinates needed
};
__host__ __device__ __forceinline__ TileStep make_tile_step(const ConvProblem &p, uint32_t rows)
{
    TileStep s;
    const uint32_t ohw = (uint32_t)(p.OH * p.OW);
    s.rows = rows;
    s.db = (int)(rows / ohw);
    const uint32_t rem = rows - (uint32_t)s.db * ohw;
    s.doh = (int)(rem / (uint32_t)p.OW);
    s.dow = (int)(rem - (uint32_t)s.doh * (uint32_t)p.OW);
    s.pat = 0;
    for (int r = 0; r < p.kh; ++r) s.pat |= 1u << (r * p.kw);
    s.pointwise = p.kh == 1 && p.kw == 1 && p.stride == 1 && p.pad == 0;
    return s;
}
// A persistent CTA's way through the tiles (n, m), m fastest: from tile blockIdx.x in steps of gridDim.x.  Or ACROSS the columns:
// blocks beside one another take the tile columns of the same rows, a CTA keeps its column (the grid is a multiple of their
// number).  All divisions are the host's: an integer division is some twenty instructions, and in code that runs once an instruction
// costs some ten cycles.
struct TilePos {
    int n, m;
};
struct TileWalk {
    int m_tiles, tiles, extra;       // row tiles; every CTA's tiles, and the number of CTAs that have one more
    int dn, dm;                      // gridDim.x = dn * m_tiles + dm (across: 0, the columns' share of gridDim.x)
    int d;                           // m_tiles (across: the number of columns)
    uint32_t mul, shift;             // exact_div by d
    bool across;
    TileStep step;                   // of the rows of two consecutive tiles, as long as n does not change
    __device__ __forceinline__ int tiles_of(int cta) const { return tiles + (cta < extra ? 1 : 0); }
    __device__ __forceinline__ TilePos first(int cta) const
    {
        const int q = (int)exact_div((uint32_t)cta, mul, shift), r = cta - q * d;
        return across ? TilePos{r, q} : TilePos{q, r};
    }
    // true where the next tile's rows are not `step` behind the last one's
    __device__ __forceinline__ bool next(TilePos &t) const
    {
        t.n += dn;
        t.m += dm;
        const bool wrap = t.m >= m_tiles;
        if (wrap) { t.m -= m_tiles; ++t.n; }
        return wrap || dn > 0;
    }
};
inline TileWalk make_tile_walk(const ConvProblem &p, int tile_rows, int m_tiles, int n_tiles, int grid, bool across)
{
    TileWalk w;
    const int total = m_tiles * n_tiles, rows = across ? grid / n_tiles : grid;       // row tiles from one of a CTA's tiles to its next
    w.m_tiles = m_tiles;
    w.tiles = across ? m_tiles / rows : total / grid;
    w.extra = across ? m_tiles % rows * n_tiles : total % grid;
    w.dn = across ? 0 : grid / m_tiles;
    w.dm = across ? rows : grid % m_tiles;
    w.d = across ? n_tiles : m_tiles;
    w.across = across;
    exact_div_params((uint32_t)w.d, w.mul, w.shift);
    w.step = make_tile_step(p, (uint32_t)tile_rows * (uint32_t)rows);
    return w;
}
struct RowCursor {
    uint32_t m;              // row of the implicit patch matrix
    int b, oh, ow;
    int base;                // word offset of the top-left input pixel (may be negative)
    uint32_t mask;           // taps inside the image; 0 for rows beyond M
};
__device__ __forceinline__ void row_locate(const ConvProblem &p, RowCursor &rc)
{
    const uint32_t ohw = (uint32_t)(p.OH * p.OW);
    rc.b = (int)exact_div(rc.m, p.ohw_mul, p.ohw_shift);
    const uint32_t rem = rc.m - (uint32_t)rc.b * ohw;
    rc.oh = (int)exact_div(rem, p.ow_mul, p.ow_shift);
    rc.ow = (int)(rem - (uint32_t)rc.oh * (uint32_t)p.OW);
}
__device__ __forceinline__ void row_step(const ConvProblem &p, const TileStep &s, RowCursor &rc)
{
    rc.m += s.rows;
    if (s.pointwise) return;
    rc.ow += s.dow;
    if (rc.ow >= p.OW) { rc.ow -= p.OW; ++rc.oh; }
    rc.oh += s.doh;
    if (rc.oh >= p.OH) { rc.oh -= p.OH; ++rc.b; }
    rc.b += s.db;
}
__device__ __forceinline__ uint32_t low_bits(int n) { return (1u << n) - 1u; }   // 0 <= n <= 31
__device__ __forceinline__ void row_window(const ConvProblem &p, const TileStep &s, RowCursor &rc)
{
    if (s.pointwise) {                                      // warp-uniform
        rc.base = (int)(rc.m * (uint32_t)p.cw);
        rc.mask = rc.m < (uint32_t)p.M ? 1u : 0u;
        return;
    }
    const int ih0 = rc.oh * p.stride - p.pad, iw0 = rc.ow * p.stride - p.pad;
    rc.base = ((rc.b * p.H + ih0) * p.W + iw0) * p.cw;
    // taps t with 0 <= iw0 + t < W and r with 0 <= ih0 + r < H (an empty range gives an empty mask)
    const int clo = min(max(-iw0, 0), p.kw), chi = max(min(p.W - iw0, p.kw), 0);
    const int rlo = min(max(-ih0, 0), p.kh), rhi = max(min(p.H - ih0, p.kh), 0);
    const uint32_t cols = low_bits(chi) & ~low_bits(clo);
    const uint32_t rows = s.pat & low_bits(rhi * p.kw) & ~low_bits(rlo * p.kw);
    rc.mask = rc.m < (uint32_t)p.M ? cols * rows : 0u;
}
template <int BYTES>
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const void *src, uint32_t nbytes)
{
    if (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(nbytes) : "memory");
    else if (BYTES == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(nbytes) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(nbytes) : "memory");
}
// Stages are 256 bits of K: eight words, 8 / GW units, two 16-byte halves `half` bytes apart in shared memory.
// A table entry is one word: the unit's word offset (27 bits) and its tap in the top five; tap 31, which no row mask
// contains, marks the zero padding of K.
constexpr int TAP_NONE = 31;
__device__ __forceinline__ void build_unit_table8(const ConvProblem &p, uint32_t tab_addr, int units, int gw, int tid, int nthreads)
{
    for (int u = tid; u < units; u += nthreads) {
        const int kword = u * gw;
        uint32_t ent = (uint32_t)TAP_NONE << 27;
        if (kword < p.kwords) {
            const int tap = p.cw_magic ? (int)__umulhi((uint32_t)kword, p.cw_magic) : kword, cj = kword - tap * p.cw;
            const int r = p.kw_magic ? (int)__umulhi((uint32_t)tap, p.kw_magic) : tap, t = tap - r * p.kw;
            ent = (uint32_t)((r * p.W + t) * p.cw + cj) | ((uint32_t)tap << 27);
        }
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(tab_addr + 4u * u), "r"(ent) : "memory");
    }
}
// Only the first `nunits` units are copied (warp-uniform; what lies beyond K's last word needs no copy when nobody reads it).
template <int GW>
__device__ __forceinline__ void gather_stage8(const uint32_t *x, const RowCursor &rc, uint32_t tab, uint32_t dst, uint32_t half, int nunits = 8)
{
    constexpr int U = 8 / GW;
    uint32_t ent[U];
    if (U == 2) {
        asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(ent[0]), "=r"(ent[1]) : "r"(tab));
    } else {
#pragma unroll
        for (int h = 0; h < U / 4; ++h)
            asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(ent[4 * h]), "=r"(ent[4 * h + 1]), "=r"(ent[4 * h + 2]), "=r"(ent[4 * h + 3]) : "r"(tab + 16u * h));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (u >= nunits) break;
        const bool ok = ((rc.mask >> (ent[u] >> 27)) & 1u) != 0u;
        const int idx = ok ? rc.base + (int)(ent[u] & 0x7FFFFFFu) : 0;
        constexpr int PER = 4 / GW;                         // units per 16-byte half
        cp_async_zfill<GW * 4>(dst + (u / PER) * half + (uint32_t)((u % PER) * GW * 4), x + idx, ok ? (uint32_t)(GW * 4) : 0u);
    }
}
// eight K words -> 32 tensor-memory columns (column 4e + j = word j of K word e)
__device__ __forceinline__ void expand_stage8(const uint4 &q0, const uint4 &q1, uint32_t (&v)[32])
{
    expand_a4(q0.x, &v[0]); expand_a4(q0.y, &v[4]); expand_a4(q0.z, &v[8]); expand_a4(q0.w, &v[12]);
    expand_a4(q1.x, &v[16]); expand_a4(q1.y, &v[20]); expand_a4(q1.z, &v[24]); expand_a4(q1.w, &v[28]);
}
// the first nk (1..8) words of a stage; a stage of at most four words has one 16-byte half and 16 columns
__device__ __forceinline__ void expand_store_stage8(uint32_t taddr, uint32_t src, uint32_t half, int nk)
{
    const uint4 q0 = ld_shared_v4(src);
    if (nk > 4) {                                           // warp-uniform
        uint32_t v[32];
        expand_stage8(q0, ld_shared_v4(src + half), v);
        tc_st32_nowait(taddr, v);
    } else {
        uint32_t v[16];
        expand_a4(q0.x, &v[0]); expand_a4(q0.y, &v[4]); expand_a4(q0.z, &v[8]); expand_a4(q0.w, &v[12]);
        tc_st16_nowait(taddr, v);
    }
}

// int32 output of one accumulator chunk: 32 rows (one per lane) x 32 consecutive columns, of which the first `ncols` exist.
// A lane storing its own row touches 32 rows per instruction; staged through shared memory the warp stores contiguous pieces
// of rows instead: four whole 128-byte rows per instruction where rows are 16-byte aligned, else one row of 32 integers
// (13208 x 473, K = 704: 40 -> 12 us).  `warp_tile`: I32_TILE_BYTES of shared memory owned by this warp; `dst0` points at (row0, first
// column), `ldc` is the row pitch in elements.  All 32 lanes must call it.
constexpr int I32_ROW_BYTES = 144;                         // 128 + 16: conflict-free both ways
constexpr int I32_TILE_BYTES = 32 * I32_ROW_BYTES;
__device__ __forceinline__ void store_int32_block(int32_t *dst0, long ldc, const int (&o)[32], uint32_t warp_tile,
                                                  long row0, long M, int lane, int ncols)
{
    const uint32_t mine = warp_tile + (uint32_t)(lane * I32_ROW_BYTES);
#pragma unroll
    for (int i4 = 0; i4 < 8; ++i4)
        st_shared_v4(mine + 16u * i4, (uint32_t)o[4 * i4], (uint32_t)o[4 * i4 + 1], (uint32_t)o[4 * i4 + 2], (uint32_t)o[4 * i4 + 3]);
    __syncwarp();
    if ((ldc & 3) == 0 && ncols >= 32) {                   // warp-uniform; the output is 16-byte aligned and chunks start at multiples of 32
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int r = (lane >> 3) + 4 * i;
            const uint4 v = ld_shared_v4(warp_tile + (uint32_t)(r * I32_ROW_BYTES + (lane & 7) * 16));
            if (row0 + r < M) *reinterpret_cast<uint4 *>(dst0 + (long)r * ldc + 4 * (lane & 7)) = v;
        }
    } else {
        const int rows = (int)min(32L, M - row0);
        int32_t *dst = dst0 + lane;
#pragma unroll 8
        for (int r = 0; r < 32; ++r, dst += ldc) {
            int v;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(warp_tile + (uint32_t)(r * I32_ROW_BYTES + 4 * lane)) : "memory");
            if (r < rows && lane < ncols) *dst = v;
        }
    }
    __syncwarp();
}

// Convolution-module epilogue (Section 4.2.1).
//
// Identity staging: an epilogue thread owns one output row and walks its 32-channel chunks in order.  The 64 bytes of
// fp16 identity values of a chunk are copied with cp.async into the row's slot of a small ring in shared memory,
// ID_AHEAD chunks before they are needed (across tile boundaries), so the loads are in flight while the MMAs run
// and while earlier chunks are computed.  Rows are ID_ROW_BYTES apart (64 + 16: conflict-free 16-byte accesses
// across a warp, both one row per lane and four lanes per row).
// (A variant that turns each 32 x 32 block through shared memory so that a lane owns a channel - parameters in
// registers, contiguous 64-byte requests, warp votes for the sign words - was measured at 0.55x the speed of this
// one: its 2-byte accesses and 32 votes per block cost more than the strided 16-byte accesses here.)
constexpr int ID_AHEAD = 2;
constexpr int ID_SLOTS = ID_AHEAD + 1;
constexpr int ID_ROW_BYTES = 80;
constexpr int ID_RING_BYTES = ID_SLOTS * BM * ID_ROW_BYTES;      // 30720

// Queue the copy of one chunk for the 32 rows of this warp (always commits a group, empty when there is nothing to
// copy).  The warp copies cooperatively: lane l fetches 16-byte part l % 4 of rows l / 4 + 8 i, so that one
// instruction touches 8 rows x 64 contiguous bytes instead of 32 rows x 16 bytes; `warp_slot` is the slot of the
// warp's first row, `row0` that row.  After cp.async.wait_group a __syncwarp makes all lanes' copies visible.
__device__ __forceinline__ void module_prefetch(const ConvProblem &p, uint32_t warp_slot, long row0, int n0, int lane)
{
    if (p.identity) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = (lane >> 2) + 8 * i;
            const long row = row0 + r;
            const bool ok = row < p.M;
            cp_async16(warp_slot + (uint32_t)(r * ID_ROW_BYTES + (lane & 3) * 16),
                       p.identity + (ok ? row * p.C_out + n0 + 8 * (lane & 3) : 0), ok);
        }
    }
    cp_async_commit();
}

// One chunk: 32 consecutive output channels n0 .. n0+31 of the warp's 32 output rows, lane = row.
//   t = dot * scale + shift;  u = t + identity;  r = u >= 0 ? u : slope * u;  y = fp16(r);  bit = (y + next_bias >= 0)
// one fp32 operation per step, each rounded to nearest (no fused multiply-add), the sign taken of the stored
// fp16 value.  Reads the identity values from the row's staging slot, writes the 32 fp16 values back into the
// same slot, from where the warp stores them cooperatively (same 8 rows x 64 bytes per instruction), and returns
// the 32 sign bits of the lane's row (bit i = channel n0 + i).  The channel count is a multiple of 32, so every
// 8-channel group is 16-byte aligned.  All 32 lanes must call it.
template <bool HAS_ID, bool HAS_NB>
__device__ __forceinline__ uint32_t module_chunk_t(const ConvProblem &p, const float (&dot)[32], uint32_t slot_addr, int n0)
{
    uint32_t bits = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) {                           // 8 channels per group
        uint4 idv = make_uint4(0u, 0u, 0u, 0u);
        if (HAS_ID) idv = ld_shared_v4(slot_addr + 16u * g);
        const uint32_t idw[4] = {idv.x, idv.y, idv.z, idv.w};
        uint32_t ow[4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int n = n0 + 8 * g + 4 * h;
            const float4 sc = __ldg(reinterpret_cast<const float4 *>(p.bn_scale + n));
            const float4 sh = __ldg(reinterpret_cast<const float4 *>(p.bn_shift + n));
            const float4 sl = __ldg(reinterpret_cast<const float4 *>(p.slope + n));
            float4 nb = make_float4(0.f, 0.f, 0.f, 0.f);
            if (HAS_NB) nb = __ldg(reinterpret_cast<const float4 *>(p.next_bias + n));
            const float scs[4] = {sc.x, sc.y, sc.z, sc.w}, shs[4] = {sh.x, sh.y, sh.z, sh.w};
            const float sls[4] = {sl.x, sl.y, sl.z, sl.w}, nbs[4] = {nb.x, nb.y, nb.z, nb.w};
#pragma unroll
            for (int q = 0; q < 2; ++q) {                   // two channels at a time: paired fp16 <-> fp32 conversions
                const int c = 8 * g + 4 * h + 2 * q;
                const float2 idf = __half22float2(*reinterpret_cast<const __half2 *>(&idw[2 * h + q]));
                float r[2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    float t = __fmul_rn(dot[c + e], scs[2 * q + e]);       // dot: an exact integer
                    t = __fadd_rn(t, shs[2 * q + e]);
                    const float u = HAS_ID ? __fadd_rn(t, e ? idf.y : idf.x) : t;
                    r[e] = (u >= 0.0f) ? u : __fmul_rn(sls[2 * q + e], u);
                }
                const __half2 y2 = __floats2half2_rn(r[0], r[1]);      // round to nearest even, element-wise
                ow[2 * h + q] = *reinterpret_cast<const uint32_t *>(&y2);
                const float2 yf = __half22float2(y2);
                bits |= (__fadd_rn(yf.x, nbs[2 * q]) >= 0.0f ? 1u : 0u) << c;
                bits |= (__fadd_rn(yf.y, nbs[2 * q + 1]) >= 0.0f ? 1u : 0u) << (c + 1);
            }
        }
        st_shared_v4(slot_addr + 16u * g, ow[0], ow[1], ow[2], ow[3]);
    }
    return bits;
}
__device__ __forceinline__ uint32_t module_chunk(const ConvProblem &p, const float (&dot)[32], uint32_t warp_slot,
                                                 long row0, int n0, int lane)
{
    const uint32_t slot_addr = warp_slot + (uint32_t)(lane * ID_ROW_BYTES);
    __syncwarp();                                           // the cooperative copies of all lanes have landed
    uint32_t bits;
    if (p.identity) bits = p.next_bias ? module_chunk_t<true, true>(p, dot, slot_addr, n0) : module_chunk_t<true, false>(p, dot, slot_addr, n0);
    else bits = p.next_bias ? module_chunk_t<false, true>(p, dot, slot_addr, n0) : module_chunk_t<false, false>(p, dot, slot_addr, n0);
    __syncwarp();                                           // the rows of all lanes are staged
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = (lane >> 2) + 8 * i;
        const long row = row0 + r;
        const uint4 v = ld_shared_v4(warp_slot + (uint32_t)(r * ID_ROW_BYTES + (lane & 3) * 16));
        if (row < p.M) *reinterpret_cast<uint4 *>(p.y_real + row * p.C_out + n0 + 8 * (lane & 3)) = v;
    }
    __syncwarp();                                           // the slot may be refilled
    return bits;
}

}  // namespace tc
}  // namespace bcnn
