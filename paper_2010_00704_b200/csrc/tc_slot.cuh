// Helpers of the pipelines without a control warp (conv_tc_pw.cu, conv_tc_pn.cu, conv_tc_c3.cu, conv_tc_mod.cu; the waits: stem.cu): tensor-memory loads that do not wait, the
// register pin that keeps uses behind the wait, the short-sleep bounded mbarrier wait, and the sign-bit gathering
// from packed 16-bit accumulator halves.
#pragma once
#include "tc_common.cuh"

namespace bcnn {
namespace tc {

// 64 accumulator columns of this warp's 32 rows as packed 16-bit halves: register i = columns 2i (low) and 2i + 1.
// The loads below do NOT wait: several are issued in a row, then tc_wait_ld(), then pin_regs() on every destination
// array - an empty volatile asm that takes the registers as read-write operands, so that no use of them can be
// scheduled ahead of the wait.
__device__ __forceinline__ void tc_ld64_pack16(uint32_t taddr, uint32_t (&v)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr) : "memory");
}
// 32 columns -> 16 registers.
__device__ __forceinline__ void tc_ld32_pack16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.pack::16b.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void pin_regs(uint32_t (&v)[16])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                      "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]) :: "memory");
}
__device__ __forceinline__ void pin_regs(uint32_t (&v)[32])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                      "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                      "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                      "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31]) :: "memory");
}

// Waits of this engine: hand-overs are on the critical path of a slot's cycle, so the waiter sleeps only briefly
// between polls (a failed try_wait returns at once: measured, polling without any sleep more than doubled the
// instructions the SM executes; the shared helpers' 100 ns is a fifth of a slot's cycle here).
// Bounded by elapsed clock cycles (about two seconds), checked every 64 polls together with the CTA's abort flag.
constexpr long long PW_WAIT_CYCLES = 4000000000LL;
constexpr uint32_t PW_SLEEP_NS = 32;
template <uint32_t SLEEP = PW_SLEEP_NS>
static __device__ __noinline__ bool pw_wait_slow(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err, int code)
{
    const long long t0 = clock64();
    for (uint32_t it = 1;; ++it) {
        __nanosleep(SLEEP);
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0u) {
            if (*abort_flag) return false;
            if (clock64() - t0 > PW_WAIT_CYCLES) break;
        }
    }
    *abort_flag = 1;
    if (err) atomicCAS(err, 0, code);
    return false;
}
// whole-warp wait (every lane polls; the verdict is a vote).  SLEEP: nanoseconds between polls - short for hand-overs on
// a pipeline's critical path, longer for roles with slack (a polling warp takes issue slots from the warps that work).
template <uint32_t SLEEP = PW_SLEEP_NS>
__device__ __forceinline__ bool pw_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err, int code)
{
    bool ok = mbar_try_wait(bar, parity);
    if (__all_sync(0xffffffffu, ok)) return true;
    if (!ok) ok = pw_wait_slow<SLEEP>(bar, parity, abort_flag, err, code);
    return __all_sync(0xffffffffu, ok);
}

// The wait of a lane that issues MMAs: no sleep, nothing but the question while it is answered with no (one lane of one warp asks).
__device__ __forceinline__ bool issuer_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *err, int code)
{
    for (uint32_t it = 0; !mbar_try_wait(bar, parity); ++it) {
        if ((it & 4095u) != 4095u) continue;
        if (*abort_flag) return false;
        if (it > (1u << 25)) {                 // some seconds
            *abort_flag = 1;
            if (err) atomicCAS(err, 0, code);
            return false;
        }
    }
    return true;
}

// Per-channel constants by an MMA, and sums that fit 16 bits.  A tile's first MMA (not accumulating) multiplies a constant
// activation tile with a constant row per channel and leaves BIAS + c in the accumulator: the first K block of 32 has one
// product 4 * 6 at scale 2^16 = BIAS, the second, at scale 4, adds up to the integer c.  BIAS = 1.5 * 2^20 keeps every
// following sum in one binade, so the low 16 mantissa bits are 8 (c + dot) in two's complement: the epilogue loads packed
// 16-bit halves (two columns per register, half the loads) and gathers sign bits with byte permutes, instead of two fp32
// operations and a quarter of a 16-byte shared load per column.  Holds for |c + dot| < 4096 and |c| <= CONST_MAX
// (thresholds are clamped: both are at most 2 K + 1), i.e. K <= CONST_MAX_K; checked exact on the GPU against popcounts.
// Tensor memory: CB_COLS columns - unit scales (4 columns serve instructions up to N = 128), the constant tile's scales, the
// constant tile.
constexpr int CONST_MAX = 2591, CONST_MAX_K = (CONST_MAX - 1) / 2;
constexpr int CB_COLS = 16, CB_COL = 512 - CB_COLS, CB_SCALE = CB_COL + 4, CB_A = CB_COL + 8;
// the block, in this warp's 32 lanes (the four warps of a group cover all lanes); returns once it is written
__device__ __forceinline__ void write_const_block(uint32_t t_lane)
{
    constexpr uint32_t sc = (127u + 16u) | ((127u + 2u) << 8) | ((127u + 16u) << 16) | ((127u + 2u) << 24);
    const uint32_t scales[8] = {SF_ONES, SF_ONES, SF_ONES, SF_ONES, sc, sc, sc, sc};
    // element 0 = 4; elements 32 .. 59 = 4, 60 and 61 = 1/2
    const uint32_t a[8] = {0x6u, 0u, 0u, 0u, 0x66666666u, 0x66666666u, 0x66666666u, 0x00116666u};
    tc_st8_nowait(t_lane + (uint32_t)CB_COL, scales);
    tc_st8_nowait(t_lane + (uint32_t)CB_A, a);
    tc_wait_st();
}
// first 32 bytes of row `row` of a constant weight tile (128-byte swizzled rows): 16 * digit for up to 28 elements - six as
// often as it fits (96), then what is left down to below 8 - and 2 * digit for two more
// (BIAS = false: the first block is zero, the MMA writes c alone)
template <bool BIAS = true>
__device__ __forceinline__ void store_const_row(int c, uint32_t row_addr, int xr)
{
    const uint32_t a = (uint32_t)(c < 0 ? -c : c), neg = c < 0 ? 0x88888888u : 0u;
    const uint32_t full = min(a / 96u, 26u);
    uint32_t rem = a - 96u * full;
    const uint32_t t = rem >> 3, c1 = t < 4u ? t : (t < 6u ? 4u : (t < 8u ? 5u : 6u));     // digit codes: 0 .. 6 = 0, 1/2, 1, 3/2, 2, 3, 4
    rem -= c1 < 4u ? 8u * c1 : (c1 == 4u ? 32u : (c1 == 5u ? 48u : 64u));
    const uint32_t c2 = rem >> 3, r3 = rem & 7u;                                             // rem < 32
    const uint32_t c3 = r3 < 4u ? r3 : (r3 < 6u ? 4u : 5u), c4 = r3 == 5u || r3 == 7u ? 1u : 0u;
    uint32_t o[4];
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q) {
        const uint32_t n = full <= 8u * q ? 0u : full - 8u * q;
        uint32_t w = n >= 8u ? 0x77777777u : 0x77777777u & ((1u << (4u * n)) - 1u);
        if ((full >> 3) == q) w |= c1 << (4u * (full & 7u));
        if (((full + 1u) >> 3) == q) w |= c2 << (4u * ((full + 1u) & 7u));
        if (q == 3) w |= (c3 << 16) | (c4 << 20);
        o[q] = w ^ neg;
    }
    st_shared_v4(row_addr + (uint32_t)((0 ^ xr) << 4), BIAS ? 0x7u : 0u, 0u, 0u, 0u);
    st_shared_v4(row_addr + (uint32_t)((1 ^ xr) << 4), o[0], o[1], o[2], o[3]);
}
// the constant MMA: accumulator = BIAS + c
__device__ __forceinline__ void tc_mma_const(uint32_t d_tmem, uint32_t tmem, uint32_t c_lo, uint32_t desc_hi, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
        "setp.ne.b32 p, 0, 0;\n\t"
        "mov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], db, %4, [%5], [%6], p;\n\t}"
        ::"r"(d_tmem), "r"(tmem + (uint32_t)CB_A), "r"(c_lo), "r"(desc_hi), "r"(idesc), "r"(tmem + (uint32_t)CB_SCALE), "r"(tmem + (uint32_t)CB_COL)
        : "memory");
}

// Output word of a 32-column block from its 16 packed registers: bit = (accumulator >= 0).  PRMT in sign-replication
// mode turns the two halves of two registers into four bytes 0x00 / 0xFF; step s keeps bit s of every byte.
__device__ __forceinline__ uint32_t sign_word(const uint32_t *r)
{
    uint32_t w = 0;
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        uint32_t d;
        asm("prmt.b32 %0, %1, %2, 0xFDB9;" : "=r"(d) : "r"(r[s]), "r"(r[8 + s]));    // sign bytes of r[s].b1, r[s].b3, r[8+s].b1, r[8+s].b3
        w |= ~d & (0x01010101u << s);
    }
    return w;
}

// Accumulator column c of a 32-column block holds this channel of the block (the order sign_word gathers bits in).
__host__ __device__ constexpr int channel_of_column(int c)
{
    return c < 16 ? ((c & 1) ? 8 + (c >> 1) : (c >> 1)) : ((c & 1) ? 24 + ((c - 16) >> 1) : 16 + ((c - 16) >> 1));
}

}  // namespace tc
}  // namespace bcnn
