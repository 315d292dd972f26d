// Streaming tcgen05 engine: wide layers, long K, small layers, the plain GEMMs, on PREPARED weights and (below) on raw ones.
//
// The weights of a layer never change between calls.  bcnn_prepare_weights expands their sign bits ONCE per layer into a
// caller-owned buffer - signed 4-bit codes, K-major, rows padded to 128 and K to 256, then K - 2 popc(W_n) per row; half
// the bytes that bcnn_prepared_weights_bytes asks for - and the kernel's weight operand arrives by TMA: one
// cp.async.bulk.tensor per ring stage (a 128-byte x BN-row box = 256 bits of K, 128-byte swizzle - exactly the
// shared-memory tile the MMA descriptor describes) issued by a loader warp, completing on the stage's mbarrier.  No warp
// touches a weight.
//
// Arithmetic: 4-bit operands (tc_common.cuh), fp32 accumulators that hold exact integers:
//   sum a*g = accumulator + cst_n                          cst_n = K - 2 popc(G_n)   (from the prepared buffer)
//   packed output: accumulator + (cst_n - thr_n) >= 0      thr clamped to +-(K + 1)
// so there are no per-row constants, and the per-column ones are added by the epilogue from a small table.
//
//   warp 0        issuer: one lane waits for a stage, issues its MMAs and their commits
//   warps 1-4     epilogue (256-wide tiles, and int32 128-wide ones of prepared weights: 1-8, two teams with half of the columns each): build the
//                 column table (where the columns change), tcgen05.ld, add + sign bits (or int32), store
//   G groups of 4 activation warps: implicit-im2col gather (cp.async), expansion, tcgen05.st into the ring in tensor memory
//   loader warp   weight tiles by TMA into the ring in shared memory
// Every mbarrier wait is bounded and reports through the device error word.
//
// 256-wide tiles have one accumulator buffer.  Packed ones, and those of two blocks, hand it over in halves of 128 columns: a tile's last two
// stages are multiplied half by half, and so are the next one's first two, so that each half is read while the other is worked on; int32 outputs
// of a pair leave it as 16-bit numbers (K <= 32767) and go to memory beside the next tile's MMAs.  Int32 tiles of one block are handed over whole, and
// each team's 128 consecutive columns go to memory one after the other.  Large products run on pairs of blocks (cta_group::2).
//
// RAW WEIGHTS (packed bits, new on each call): in each group as many weight warps as 32-row pieces of the CTA's weight tile expand them into
// the ring, instead of the loader.  A pair of CTAs is what pays there, each expands half of the weight rows: 4096 x 4096 x 4608
// packed 56 -> 36.8 us (0.41 us a stage against 0.28 of the pipe: the eight warps of a group have 250 issue slots of work per stage and its latencies),
// 8192 x 8192 x 9216 328 -> 220, and the short set-up: 2070 x 64 x 288 4.3 -> 3.0, 34 x 3712 x 608 5.5 -> 3.5.
//
// What bounds it.  Long products: power.  A 256-bit stage of a 256-wide tile takes 553 cycles of a pair (512 of the pipe), at a clock
// that falls from 1965 to 1600 .. 1750 MHz.  Narrow tiles: the issuer - a stage of four instructions with its wait and its commit costs it 300
// to 400 cycles beside busy warps, whatever the width (128: 256 of the pipe); and what a launch does once, which is why set-up is short, its
// divisions are the host's, and each role waits for the previous kernel as late as it can (0.7 us of a small layer's 4.3).
// Before and after, us: 3x3 128 -> 128 at M = 784 4.3 -> 3.3, at M = 200704 18.9 -> 17.2; 256 -> 256 at M = 50176 15.4 -> 13.1; 512 -> 512 /2 at M = 25088
// 23.5 -> 21.6; 1x1 256 -> 256 at M = 196 3.1 -> 2.3; 1000 x 4000 x 2304 8.4 -> 7.3; 8192 x 8192 x 512 52.6 -> 33.8.
#include "tc_slot.cuh"
#include "tensor_map.cuh"
#include <climits>

namespace bcnn {

namespace {

using namespace tc;

constexpr int PF = 3;                     // packed-word stages in flight per producer thread
constexpr int MAX_SMEM = 227 * 1024 - 512;

constexpr int ERR_PRODUCER_TIMEOUT = 131;
constexpr int ERR_MMA_TIMEOUT = 132;
constexpr int ERR_EPILOGUE_TIMEOUT = 133;
constexpr int ERR_LOADER_TIMEOUT = 134;

// where the weights are raw: the operand whose bits are signed and counted, hence what the constants belong to
constexpr int RAW_COLUMNS = 1, RAW_ROWS = 2;

// BN: output channels of a tile; MODE: 0 int32, 1 packed output; G: activation producer groups of four warps; TEAMS: epilogue
// teams of four warps, each with its share of a tile's columns; WHOLE: a 256-wide tile handed over in one piece, each team 128
// consecutive columns, which go to memory one after the other
template <int BN, int MODE, int G, int TEAMS, bool PAIR, int RAW = 0, bool WHOLE = false> struct Cfg {
    static constexpr int EPI_WARPS = 4 * TEAMS;
    static constexpr int NBUF = BN == 256 ? 1 : (BN == 128 ? 2 : 4);     // accumulator buffers
    static constexpr int A_COL0 = NBUF * BN;                              // first column of the activation ring
    static constexpr int STAGES = !PAIR && BN == 256 ? (MODE == 0 ? 4 : 5) : 7;
    static constexpr int CTAS = PAIR ? 2 : 1, TILE_ROWS = CTAS * BM;      // CTAs of a tile, its rows
    static constexpr int WW = RAW ? BN / CTAS / 32 : 0;                   // raw weights: a group's weight warps, a row per thread
    static constexpr int GROUP_WARPS = 4 + WW;
    static constexpr int PROD_THREADS = G * 32 * GROUP_WARPS;
    static constexpr int FIRST_PRODUCER_WARP = 1 + EPI_WARPS;
    static constexpr int LOADER_WARP = FIRST_PRODUCER_WARP + G * GROUP_WARPS;
    static constexpr int THREADS = 32 * (LOADER_WARP + (RAW ? 0 : 1));
    static constexpr int EC = BN / TEAMS;                                 // columns of a team
    static constexpr bool SPLIT = BN == 256 && !WHOLE;                    // one accumulator, handed over in halves of 128 columns
    static constexpr int PIECES = SPLIT ? 2 : 1, PC = EC / PIECES;        // pieces of a team's columns, columns of a piece
    static constexpr int MMA_N = SPLIT ? BN / 2 : BN;                     // columns of an instruction
    static constexpr int W_BYTES = BN / CTAS * ROWB;                      // one ring stage of weights
    // a producer's next copies ahead of the wait for its oldest (three stages in flight), or behind its store (two, and the store's latency
    // hidden).  us, ahead and behind: 128 wide 5x5 160 -> 128 at M = 336336 87.7 and 89.9, 128 -> 128 at 200704 17.1 and 17.2; 256 wide
    // 256 -> 256 at 50176 13.2 and 13.0
    static constexpr bool EARLY = BN < 256 && !RAW;
    static constexpr int SF_COL = 512 - (int)SF_COLS;                     // unit scales
    static constexpr int BITS_BYTES = PF * PROD_THREADS * 32;
    static constexpr int TABLE_BYTES = EPI_WARPS * EC * 4;                // one column table per epilogue warp
    // raw weights: tiles whose bit counts are kept - those with an accumulator, those in the ring, and one per group that has counted but
    // waits for a slot; a count per row of the operand that is signed
    static constexpr bool SIGNED_A = RAW == RAW_ROWS;
    static_assert(!PAIR || RAW != RAW_COLUMNS, "a pair's column constants would have to be exchanged");
    static constexpr int SLOTS = STAGES + NBUF + G, POP_ROWS = SIGNED_A ? BM : BN;
    static constexpr int POP_BYTES = RAW ? SLOTS * G * POP_ROWS * 4 : 0;
    static_assert(A_COL0 + STAGES * 32 <= SF_COL, "tensor memory budget");
    static_assert(STAGES >= G, "a producer group must not lap the ring (parity waits)");
};

// ---- two CTAs on one tile of 256 rows (cta_group::2): the even CTA's issuer multiplies for both, each brings its own 128 rows of
// activations and half of the weight rows, each keeps the accumulators of its own rows.
template <bool PAIR> __device__ __forceinline__ void commit(uint32_t bar)
{
    if (PAIR)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((uint16_t)3) : "memory");
    else
        tc_commit(bar);
}
template <bool PAIR> __device__ __forceinline__ void mma_f4(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t desc_hi, uint32_t idesc, uint32_t sf, uint32_t accumulate)
{
    if (PAIR)
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\t"
            "setp.ne.b32 p, %6, 0;\n\t"
            "mov.b64 db, {%2, %3};\n\t"
            "tcgen05.mma.cta_group::2.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], db, %4, [%5], [%5], p;\n\t}"
            ::"r"(d_tmem), "r"(a_tmem), "r"(b_lo), "r"(desc_hi), "r"(idesc), "r"(sf), "r"(accumulate) : "memory");
    else
        tc_mma_f4_ts(d_tmem, a_tmem, b_lo, desc_hi, idesc, sf, accumulate);
}
__device__ __forceinline__ void add_row(uint32_t (&v)[32], float c)
{
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__fadd_rn(__uint_as_float(v[i]), c));
}
__device__ __forceinline__ uint32_t in_even_cta(uint32_t addr)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(addr));
    return r;
}
// A warp of either CTA to a barrier of the even one, whose issuer starts MMAs behind it.  The arrive releases at block scope only, and that is
// enough, because nothing but the signal crosses: what it announces is used on the multiprocessor that made it, by that one's tensor
// core - its activations and its accumulators in its tensor memory, its half of the weights in its shared memory - and each has been completed
// for that unit before the arrive: stores and reads of tensor memory by tcgen05.wait and fence::before_thread_sync, expanded weights by a
// fence.proxy.async of every lane that stored, both before the __syncwarp in front of this.  No thread reads the other CTA's memory: its own
// counts and constants only.  (.release.cluster waits for all of a warp's memory operations, the int32 stores and the gather's copies too, and
// took twice the time.)
__device__ __forceinline__ void arrive_in_cluster(uint32_t bar, uint32_t pred)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t@q mbarrier.arrive.shared::cluster.b64 _, [%0];\n\t}" ::"r"(bar), "r"(pred) : "memory");
}
__device__ __forceinline__ void cluster_barrier()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename C>
__host__ __device__ constexpr int smem_bytes(int ktab_words, int mode)
{
    return 1024 + C::STAGES * C::W_BYTES + C::BITS_BYTES + C::TABLE_BYTES + C::POP_BYTES + ktab_words * 4 + 16 +
           (mode == 0 ? C::EPI_WARPS * I32_TILE_BYTES + 16 : 0);
}

// RAW: the weights are packed bits, expanded on the way by warps that count a row's bits as they go.  RAW_COLUMNS: weights signed and activations
// plain as above, K - 2 popc(W_n) per column.  RAW_ROWS: the other way round,
//   sum a*g = accumulator + K - 2 popc(a):
// a constant per row, for pairs of CTAs (which would have to exchange column constants) and where the activation warps have the time.  A signed
// word is seven operations and its count, a plain one five: us with columns and rows, 3x3/2 2048 -> 32 at M = 162288 184 and 206, 1x1 96 -> 352
// at 18177 (one stage) 7.7 and 8.8, 300 x 4000 x 9216 on 128-wide tiles 18.6 and 17.0.
template <int BN, int MODE, int G, int TEAMS, bool PAIR, int RAW, bool WHOLE>
__global__ void __launch_bounds__(Cfg<BN, MODE, G, TEAMS, PAIR, RAW, WHOLE>::THREADS, 1)
conv_tc_pre_kernel(const ConvProblem p, const int32_t *cst, const __grid_constant__ CUtensorMap wmap, const int ktab_words, const TileWalk walk)
{
    using C = Cfg<BN, MODE, G, TEAMS, PAIR, RAW, WHOLE>;
    constexpr int EPI_WARPS = C::EPI_WARPS, EC = C::EC;
    constexpr bool FUSED = MODE == 1, COLUMN_COUNTS = RAW == RAW_COLUMNS;       // column constants from counts of the weights' bits
    static_assert(!COLUMN_COUNTS || !C::SPLIT, "one piece: the counts are read once per tile");
    constexpr int NBUF = C::NBUF;
    constexpr int STAGES = C::STAGES;

    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * 8 + 2 * 4];
    __shared__ uint32_t tmem_base_smem;
    __shared__ int abort_flag_smem;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int ktiles = (p.kwords + 7) >> 3;
    const int unit = PAIR ? (int)(blockIdx.x >> 1) : (int)blockIdx.x, rank = PAIR ? (int)(blockIdx.x & 1u) : 0;      // of a pair, the CTA within it
    const int my_tiles = walk.tiles_of(unit);
    const int total_items = my_tiles * ktiles;
    // (256-wide tiles) stages at a tile's start and end that are multiplied half by half: while the second half's last MMAs run, the
    // epilogue takes the first half, and it takes the second half while the next tile's first MMAs run on the first.  Two of each
    // leave the ring room for the stages that follow.
    const int split_a = min(2, ktiles >> 1), split_b = min(2, ktiles - split_a);

    const uint32_t wring = (smem_u32(smem_raw) + 1023u) & ~1023u;         // [STAGES][BN / CTAS rows][128 B], by TMA or (raw weights) by warps
    const uint32_t bits_ring = wring + STAGES * C::W_BYTES;               // [PF][2][PROD_THREADS][16 B]
    const uint32_t tables = bits_ring + C::BITS_BYTES;                    // [EPI_WARPS][EC] column constants
    const uint32_t pops = tables + C::TABLE_BYTES;                        // [SLOTS][G][POP_ROWS] bit counts
    const uint32_t ktab_addr = pops + C::POP_BYTES;                       // unit table of the gather
    const uint32_t i32_tiles = (ktab_addr + (uint32_t)ktab_words * 4u + 15u) & ~15u;   // int32 output: store staging tiles
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (8 + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (16 + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (20 + b); };
    volatile int *abort_flag = &abort_flag_smem;

    if (tid < 24) {
        // full: the warps of the stage's group + the loader's arrive (+ its bytes); accumulator free: the epilogue warps
        // (of both CTAs, whose MMAs the even one issues)
        mbar_init(bar0 + 8u * tid, tid < 8 ? C::GROUP_WARPS * C::CTAS + (RAW ? 0 : 1) : (tid >= 20 ? EPI_WARPS * C::CTAS : 1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) abort_flag_smem = 0;
    if (warp == 0) {
        if (PAIR) {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
        } else {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
    }
    const int gwidth = gather_width(p.cw);
    build_unit_table8(p, ktab_addr, ktiles * (8 / gwidth), gwidth, tid, C::THREADS);
    if (!RAW && tid == 32 * C::LOADER_WARP) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&wmap)) : "memory");
    tc_fence_before();
    if (PAIR) cluster_barrier();               // the other CTA's barriers exist
    else __syncthreads();
    tc_fence_after();
    pdl_trigger();
    // (the roles that touch global memory wait for the previous kernel behind their own set-up)
    const uint32_t tmem_base = tmem_base_smem;

    if (warp == 0) {
        // ------------------------------------------------------------------ issuer (no memory instructions)
        constexpr uint32_t idesc = PAIR ? make_idesc_f4(C::MMA_N) + (1u << 27) : make_idesc_f4(C::MMA_N);      // M = 256 or 128
        const uint64_t desc0 = make_desc(0);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
        const uint32_t b_lo0 = (uint32_t)desc0 | ((wring & 0x3FFFFu) >> 4);      // + slot * (W_BYTES / 16)
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t a_tmem0 = tmem_u + (uint32_t)C::A_COL0;                   // + slot * 32 columns
        const uint32_t sf = tmem_u + (uint32_t)C::SF_COL;
        // A stage's MMAs for all columns, or for half h of a split tile: two K words per instruction, four instructions - but for the last
        // stage's zero tail, a branch of its own.  What a stage costs its issuer is the bound of narrow tiles: in a loop alone on its
        // multiprocessor 172 cycles with a wait, 257 with a test in front of each instruction, 400 with a vote and a reconvergence, and 256 or 128
        // is what the pipe takes for 128 or 64 columns.
        const int tail = (p.kwords - 8 * (ktiles - 1) + 1) >> 1;                // instructions of the last stage
        auto four = [&](int slot, int kt, uint32_t d, int h) {
            const uint32_t a_t = a_tmem0 + (uint32_t)slot * 32u;
            const uint32_t b_lo = b_lo0 + (uint32_t)slot * (C::W_BYTES >> 4) + (uint32_t)h * (C::W_BYTES >> 5);
            mma_f4<PAIR>(d, a_t, b_lo, desc_hi, idesc, sf, kt > 0 ? 1u : 0u);
            mma_f4<PAIR>(d, a_t + 8u, b_lo + 2u, desc_hi, idesc, sf, 1u);
            mma_f4<PAIR>(d, a_t + 16u, b_lo + 4u, desc_hi, idesc, sf, 1u);
            mma_f4<PAIR>(d, a_t + 24u, b_lo + 6u, desc_hi, idesc, sf, 1u);
        };
        auto multiply = [&](int slot, int kt, uint32_t d_tmem, int h) {
            const uint32_t d = d_tmem + (uint32_t)(h * C::MMA_N);
            if (kt < ktiles - 1 || tail == 4) {
                four(slot, kt, d, h);
            } else {
                const uint32_t a_t = a_tmem0 + (uint32_t)slot * 32u;
                const uint32_t b_lo = b_lo0 + (uint32_t)slot * (C::W_BYTES >> 4) + (uint32_t)h * (C::W_BYTES >> 5);
#pragma unroll 1
                for (uint32_t i = 0; i < (uint32_t)tail; ++i) mma_f4<PAIR>(d, a_t + 8u * i, b_lo + 2u * i, desc_hi, idesc, sf, kt > 0 || i > 0 ? 1u : 0u);
            }
        };
        auto second_half = [&](int slot, int kt, int n) {                        // n stages from (slot, kt), each handed back
            for (int j = 0; j < n; ++j) {
                multiply(slot, kt + j, tmem_u, 1);
                commit<PAIR>(empty_bar(slot));
                if (++slot == STAGES) slot = 0;
            }
        };
        // One lane runs the whole loop and does its own waits: one that is satisfied costs a hundred cycles behind MMAs in the queue, and
        // while the ring is ahead of the MMAs all are.
        if (rank == 0 && elect_one()) {
            int s = 0, buf = 0;
            uint32_t ring_phase = 0, buf_phase = 1;      // first use of every accumulator buffer: free
            bool ok = true;
            auto wait = [&](uint32_t bar, uint32_t parity) {
                ok = issuer_wait(bar, parity, abort_flag, p.err, ERR_MMA_TIMEOUT);
                tc_fence_after();
                return ok;
            };
            // the ring's next stage: its slot, or -1 after a time-out
            auto take = [&]() {
                const int slot = wait(full_bar(s), ring_phase) ? s : -1;
                if (++s == STAGES) { s = 0; ring_phase ^= 1u; }
                return slot;
            };
            for (int ti = 0; ti < my_tiles; ++ti) {
                if (!wait(tempty_bar(buf), buf_phase)) break;
                if (C::SPLIT) {
                    const int s0 = s;
                    int kt = 0, slot = 0;
                    for (; kt < split_a && (slot = take()) >= 0; ++kt) multiply(slot, kt, tmem_u, 0);
                    if (!ok || !wait(tempty_bar(1), buf_phase)) break;
                    second_half(s0, 0, split_a);
#pragma unroll 1
                    for (; kt < ktiles - split_b && (slot = take()) >= 0; ++kt) {
                        four(slot, kt, tmem_u, 0);
                        four(slot, kt, tmem_u + (uint32_t)C::MMA_N, 1);
                        commit<PAIR>(empty_bar(slot));
                    }
                    const int s_last = s;
                    for (; ok && kt < ktiles && (slot = take()) >= 0; ++kt) multiply(slot, kt, tmem_u, 0);
                    if (!ok) break;
                    commit<PAIR>(tfull_bar(0));
                    second_half(s_last, ktiles - split_b, split_b);
                    commit<PAIR>(tfull_bar(1));
                } else {
                    const uint32_t d_tmem = tmem_u + (uint32_t)(buf * BN);
                    int kt = 0, slot = 0;
#pragma unroll 1
                    for (; kt < ktiles - 1 && (slot = take()) >= 0; ++kt) {
                        four(slot, kt, d_tmem, 0);
                        commit<PAIR>(empty_bar(slot));
                    }
                    if (ok && (slot = take()) >= 0) {
                        multiply(slot, kt, d_tmem, 0);
                        commit<PAIR>(empty_bar(slot));
                    }
                    if (!ok) break;
                    commit<PAIR>(tfull_bar(buf));
                }
                if (++buf == NBUF) { buf = 0; buf_phase ^= 1u; }
            }
        }
        __syncwarp();
    } else if (!RAW && warp >= C::LOADER_WARP) {
        // ------------------------------------------------------------------ loader: weight tiles by TMA
        // item (tile, stage) -> ring slot item % STAGES.  A pair: this CTA's 64 rows of every 128 of the tile; the even CTA expects both
        // CTAs' bytes, and both complete on its barrier.
        int s = 0, it = 0;
        uint32_t phase = 1;                           // first pass through the ring: slots are free
        bool ok = true;
        TilePos at = walk.first(unit);
        pdl_wait();
        // (a tile's coordinates outside of its stages: this warp's loop is what bounds long K on narrow tiles - 3x3 768 -> 64 at M = 487500
        // 158 us with one loop over all items, 140 as it is)
        for (int ti = 0; ti < my_tiles && ok; ++ti, walk.next(at)) {
            const int row = at.n * (PAIR ? BN / 128 : BN);
            for (int kt = 0; kt < ktiles; ++kt) {
                ok = mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_LOADER_TIMEOUT);
                if (!ok) break;
                if (lane == 0) {
                    const uint32_t dst = wring + (uint32_t)s * C::W_BYTES;
                    if (rank == 0) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full_bar(s)), "r"((uint32_t)(C::CTAS * C::W_BYTES)) : "memory");
                    if (PAIR)
                        asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3, %4, %5}], [%6];"
                                     ::"r"(dst), "l"(reinterpret_cast<uint64_t>(&wmap)), "r"(kt * ROWB), "r"(0), "r"(rank), "r"(row), "r"(in_even_cta(full_bar(s))) : "memory");
                    else
                        asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                     ::"r"(dst), "l"(reinterpret_cast<uint64_t>(&wmap)), "r"(kt * ROWB), "r"(row), "r"(full_bar(s)) : "memory");
                }
                __syncwarp();
                ++it;
                if (++s == STAGES) { s = 0; phase ^= 1u; }
            }
        }
        // The odd CTA: the commits that hand its last slots back come from the other multiprocessor, and its barriers stay until they are in.  (The last
        // accumulator, which the epilogue waits for, is committed behind them, but on a barrier of its own.)
        if (PAIR && rank != 0) {
            for (int i = 0; i < STAGES && ok; ++i) {
                ok = mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_LOADER_TIMEOUT);
                if (++s == STAGES) { s = 0; phase ^= 1u; }
            }
        }
        // after a time-out elsewhere: copies still in flight must land before the CTA's shared memory goes away
        if (*abort_flag && rank == 0) {
            for (int j = it > STAGES ? it - STAGES : 0; j < it; ++j)
                mbar_wait_warp(full_bar(j % STAGES), (uint32_t)(j / STAGES) & 1u, abort_flag, nullptr, 0);
        }
        // (the odd CTA's copies complete on the other's barrier: it gives them a millisecond)
        if (PAIR && *abort_flag && rank != 0)
            for (int i = 0; i < 1000; ++i) __nanosleep(1000);
    } else if (warp <= EPI_WARPS) {
        // ------------------------------------------------------------------ epilogue
        const int quad = warp & 3;                 // tensor-memory lane quadrant this warp may read
        const int erow = quad * 32 + lane, team = (warp - 1) >> 2;
        constexpr int PC = C::PC, PIECES = C::PIECES, CH = PC / 32;             // chunks of 32 columns of a piece
        const uint32_t i32_tile = i32_tiles + (uint32_t)(warp - 1) * I32_TILE_BYTES;
        // column c of this warp's table: piece c / PC, column h * 128 + team * PC + c % PC of the tile (or team * EC + c)
        const uint32_t table = tables + (uint32_t)((warp - 1) * EC * 4);
        const bool narrow = p.K <= 32767;          // int32 outputs fit 16 bits
        bool alive = true;
        int buf = 0, table_n = -1;
        uint32_t buf_phase = 0;
        const int owords = p.C_out >> 5;
        auto store_words = [&](const uint32_t (&words)[CH], int em, int n0) {
            if (em < p.M) {
                uint32_t *dst = static_cast<uint32_t *>(p.out) + (long)em * owords + (n0 >> 5);
                if (PC >= 128 && (owords & 3) == 0 && n0 + PC <= p.C_out) {
    #pragma unroll
                    for (int c4 = 0; c4 + 3 < CH; c4 += 4) *reinterpret_cast<uint4 *>(dst + c4) = make_uint4(words[c4], words[c4 + 1], words[c4 + 2], words[c4 + 3]);
                } else if ((owords & 1) == 0 && n0 + PC <= p.C_out) {
    #pragma unroll
                    for (int c2 = 0; c2 < CH; c2 += 2) *reinterpret_cast<uint2 *>(dst + c2) = make_uint2(words[c2], words[c2 + 1]);
                } else {
    #pragma unroll
                    for (int ch = 0; ch < CH; ++ch)
                        if (n0 + ch * 32 < p.C_out) dst[ch] = words[ch];
                }
            }
        };
        TilePos at = walk.first(unit);
        const uint32_t tempty0 = PAIR ? in_even_cta(tempty_bar(0)) : tempty_bar(0);
        pdl_wait();
        for (int ti = 0; ti < my_tiles; ++ti, walk.next(at)) {
            const int n_base = at.n * BN + team * PC;                           // first column of this team's first piece
            const int em = at.m * C::TILE_ROWS + rank * BM + erow;
            // the column constants, built while the tile's MMAs run, anew only where the columns change; every warp keeps its own table,
            // so the four warps need no barrier among themselves.  Where the weights' bits are counted on the way the counts come with
            // the tile: then only what belongs to the thresholds is fetched here.
            constexpr int PER = EC / 32;
            int cc[COLUMN_COUNTS ? PER : 1];
            const bool new_columns = at.n != table_n;
            if (new_columns) {
                table_n = at.n;
                __syncwarp();
                auto constant = [&](int c) {
                    const int n = n_base + (c / PC) * (BN / 2) + c % PC;
                    int v = 0;
                    if (n < p.C_out) {
                        if (!RAW) v = __ldg(cst + n);
                        if (COLUMN_COUNTS) v = p.K;
                        if (FUSED) v -= max(min(__ldg(p.thr + n), p.K + 1), -p.K - 1);       // beyond that bound the decision is constant
                    }
                    return v;
                };
                if constexpr (COLUMN_COUNTS) {
#pragma unroll
                    for (int i = 0; i < PER; ++i) cc[i] = constant(lane + 32 * i);
                } else {
#pragma unroll 1
                    for (int c = lane; c < EC; c += 32) asm volatile("st.shared.b32 [%0], %1;" ::"r"(table + 4u * c), "r"(table_entry<MODE>(constant(c))) : "memory");
                }
                __syncwarp();
            }
            // the bits of row r of the signed operand: the counts of the groups that had a stage of the tile
            auto counted = [&](int r) {
                const uint32_t at_pop = pops + (uint32_t)((ti % C::SLOTS) * G * C::POP_ROWS + r) * 4u;
                const int first = (ti * ktiles) % G;
                int n_bits = 0;
#pragma unroll
                for (int g = 0; g < G; ++g) {
                    if ((g >= first ? g - first : g - first + G) < ktiles) {
                        int v;
                        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(at_pop + (uint32_t)(g * C::POP_ROWS) * 4u) : "memory");
                        n_bits += v;
                    }
                }
                return n_bits;
            };
            const long row0 = (long)em - lane;
            uint32_t packed[MODE == 0 ? PIECES : 1][CH][16];                    // int32 outputs of a 256-wide tile, two to a register
#pragma unroll
            for (int h = 0; h < PIECES; ++h) {
                const int n0 = n_base + h * (BN / 2), b = C::SPLIT ? h : buf;
                if (alive) alive = pw_wait<100>(tfull_bar(b), buf_phase, abort_flag, p.err, ERR_EPILOGUE_TIMEOUT);
                alive = __all_sync(0xffffffffu, alive && !*abort_flag);
                if (!alive) break;
                tc_fence_after();
                const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(C::SPLIT ? h * (BN / 2) + team * PC : buf * BN + team * EC);
                // all reads of this accumulator (half) are complete: hand it back
                auto hand_back = [&]() {
                    tc_fence_before();
                    __syncwarp();
                    if (PAIR) arrive_in_cluster(tempty0 + 8u * b, lane == 0 ? 1u : 0u);
                    else if (lane == 0) mbar_arrive(tempty0 + 8u * b);
                };
                float row_cst = 0.f;
                if (C::SIGNED_A) row_cst = (float)(p.K - 2 * counted(erow));
                if (COLUMN_COUNTS && new_columns) {
#pragma unroll
                    for (int i = 0; i < PER; ++i)
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(table + 4u * (lane + 32 * i)), "r"(table_entry<MODE>(cc[i] - 2 * counted(team * EC + lane + 32 * i))) : "memory");
                    __syncwarp();
                }
                if (FUSED && C::SIGNED_A) {
                    uint32_t words[CH];
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) {
                        uint32_t v[32];
                        tc_ld32(t_addr + 32u * ch, v);
                        if (ch == CH - 1) hand_back();
                        add_row(v, row_cst);
                        words[ch] = threshold_word(v, table + 4u * (h * PC + 32 * ch));
                    }
                    store_words(words, em, n0);
                } else if (FUSED) {
                    uint32_t words[CH];
#pragma unroll
                    for (int c2 = 0; c2 < CH; c2 += 2) {                        // 64 columns in registers at a time
                        uint32_t v[2][32];
                        tc_ld32_nowait(t_addr + 32u * c2, v[0]);
                        tc_ld32_nowait(t_addr + 32u * c2 + 32u, v[1]);
                        tc_wait_ld();
                        pin_regs(v[0]);
                        pin_regs(v[1]);
                        if (c2 + 2 == CH) hand_back();
                        threshold_words(v, table + 4u * (h * PC + 32 * c2), words[c2], words[c2 + 1]);
                    }
                    store_words(words, em, n0);
                } else if (C::SPLIT && narrow) {
                    // out of the accumulator at once, 16 bits each; to memory below, beside the next tile's MMAs
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) {
                        uint32_t v[32];
                        int o[32];
                        tc_ld32(t_addr + 32u * ch, v);
                        if (ch == CH - 1) hand_back();
                        if (C::SIGNED_A) add_row(v, row_cst);
                        biased_ints(v, table + 4u * (h * PC + 32 * ch), o);
#pragma unroll
                        for (int i = 0; i < 16; ++i) packed[h][ch][i] = __byte_perm((uint32_t)o[2 * i], (uint32_t)o[2 * i + 1], 0x5410);
                    }
                } else {
#pragma unroll 1
                    for (int ch = 0; ch < CH; ++ch) {
                        uint32_t v[32];
                        int o[32];
                        if (n0 + 32 * ch < p.C_out) {          // warp-uniform
                            tc_ld32(t_addr + 32u * ch, v);
                            if (C::SIGNED_A) add_row(v, row_cst);
                            biased_ints(v, table + 4u * (h * PC + 32 * ch), o);
                            store_int32_block(static_cast<int32_t *>(p.out) + row0 * p.C_out + n0 + 32 * ch, p.C_out, o, i32_tile, row0, p.M, lane, p.C_out - n0 - 32 * ch);
                        }
                    }
                    hand_back();
                }
            }
            if (!alive) break;
            if (MODE == 0 && C::SPLIT && narrow) {
#pragma unroll
                for (int h = 0; h < PIECES; ++h) {
#pragma unroll
                    for (int ch = 0; ch < CH; ++ch) {
                        const int col0 = n_base + h * (BN / 2) + 32 * ch;
                        if (col0 < p.C_out) {                  // warp-uniform
                            int o[32];
#pragma unroll
                            for (int i = 0; i < 16; ++i) {
                                o[2 * i] = (int)(short)(packed[h][ch][i] & 0xffffu);
                                o[2 * i + 1] = (int)packed[h][ch][i] >> 16;
                            }
                            store_int32_block(static_cast<int32_t *>(p.out) + row0 * p.C_out + col0, p.C_out, o, i32_tile, row0, p.M, lane, p.C_out - col0);
                        }
                    }
                }
            }
            if (++buf == NBUF) { buf = 0; buf_phase ^= 1u; }
        }
    } else {
        // ------------------------------------------------------------------ activation producers
        // Group g takes items g, g + G, ... of the CTA's flattened (tile, stage) list: a thread copies its row's 128
        // bits of K into its staging slot (PF items ahead), then expands the oldest staged item into the ring slot.
        // (raw weights: the group's other warps do the same with a weight row per thread, into the ring in shared memory)
        const int ptid = tid - 32 * C::FIRST_PRODUCER_WARP, pwarp = warp - C::FIRST_PRODUCER_WARP;
        const int grp = pwarp / C::GROUP_WARPS, wi = pwarp - grp * C::GROUP_WARPS;
        const bool is_w = RAW && wi >= 4;
        const int quad = warp & 3;                               // tensor-memory lane quadrant this warp may write
        const int row = is_w ? (wi - 4) * 32 + lane : quad * 32 + lane;      // of the weight tile, of the activation tile
        // the weight row's output channel within the tile (a pair: this CTA's 64 of every 128)
        const int wcol = PAIR ? (row >> 6) * 128 + rank * 64 + (row & 63) : row;
        const uint32_t *wrow = p.w;
        bool wok = false;
        constexpr uint32_t HALF_BYTES = C::PROD_THREADS * 16u, SLOT_BYTES = 2u * HALF_BYTES;
        const uint32_t bits0 = bits_ring + (uint32_t)ptid * 16u, bits_end = bits0 + PF * SLOT_BYTES;
        const uint32_t st_addr0 = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::A_COL0;
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        const TileStep &step = walk.step;

        int l_kt = grp;
        int l_left = total_items > grp ? (int)((unsigned)(total_items - grp + G - 1) / (unsigned)G) : 0;
        TilePos at = walk.first(unit);
        const uint32_t full0 = PAIR ? in_even_cta(full_bar(0)) : full_bar(0);
        RowCursor rc;
        rc.m = (uint32_t)(at.m * C::TILE_ROWS + rank * BM + row);
        rc.base = 0;
        rc.mask = 0;
        if (!is_w) row_locate(p, rc);
        auto tile_ready = [&]() {            // what a tile's stages need of its row
            if (is_w) {
                const int n = at.n * BN + wcol;
                wok = n < p.C_out;
                wrow = p.w + (long)(wok ? n : 0) * p.kwords;
            } else {
                row_window(p, step, rc);
            }
        };
        auto next_tile = [&]() {             // the CTA's next tile
            if (is_w) {
                walk.next(at);
            } else if (walk.next(at)) {
                rc.m = (uint32_t)(at.m * C::TILE_ROWS + rank * BM + row);
                row_locate(p, rc);
            } else {
                row_step(p, step, rc);
            }
        };
        while (l_kt >= ktiles) { l_kt -= ktiles; next_tile(); }
        tile_ready();
        uint32_t l_dst = bits0;
        // the scales are in place before this group's first arrival, which every MMA waits for
        if (grp == 0 && !is_w) write_unit_scales(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::SF_COL);
        auto issue_load = [&]() {
            if (is_w) {
                if ((p.kwords & 3) == 0) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int kword = l_kt * 8 + 4 * q;
                        const bool ok = wok && kword < p.kwords;
                        cp_async_zfill<16>(l_dst + q * HALF_BYTES, ok ? wrow + kword : p.w, ok ? 16u : 0u);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int kword = l_kt * 8 + e;
                        const bool ok = wok && kword < p.kwords;
                        cp_async_zfill<4>(l_dst + (e >> 2) * HALF_BYTES + 4u * (e & 3), ok ? wrow + kword : p.w, ok ? 4u : 0u);
                    }
                }
            } else if (gwidth == 4) gather_stage8<4>(p.x, rc, ktab_addr + (uint32_t)l_kt * 8u, l_dst, HALF_BYTES);
            else if (gwidth == 2) gather_stage8<2>(p.x, rc, ktab_addr + (uint32_t)l_kt * 16u, l_dst, HALF_BYTES);
            else gather_stage8<1>(p.x, rc, ktab_addr + (uint32_t)l_kt * 32u, l_dst, HALF_BYTES);
            l_dst += SLOT_BYTES;
            if (l_dst == bits_end) l_dst = bits0;
            --l_left;
            l_kt += G;
            if (l_kt >= ktiles) {
                do { l_kt -= ktiles; next_tile(); } while (l_kt >= ktiles);
                tile_ready();
            }
        };
        pdl_wait();
#pragma unroll 1
        for (int i = 0; i < PF - 1; ++i) {
            if (l_left > 0) issue_load();
            cp_async_commit();
        }
        uint32_t c_src = bits0;
        int s = grp;                          // ring slot (G <= STAGES) and its parity
        uint32_t phase = 1;                   // first pass through the ring: slots are free
        int c_kt = grp, c_ti = 0, n_bits = 0; // raw weights: the stage within its tile, the tile, the row's bits so far
        int it = grp;
#pragma unroll 1
        for (; it < total_items; it += G) {
            if (C::EARLY) {
                if (l_left > 0) issue_load();
                cp_async_commit();
                cp_async_wait<PF - 1>();
            } else {
                cp_async_wait<PF - 2>();
            }
            const uint4 q0 = ld_shared_v4(c_src), q1 = ld_shared_v4(c_src + HALF_BYTES);
            c_src += SLOT_BYTES;
            if (c_src == bits_end) c_src = bits0;
            // a signed row's bits, and their count left for the epilogue at the group's last stage of the tile
            auto count = [&](const uint32_t (&wds)[8]) {
#pragma unroll
                for (int e = 0; e < 8; ++e) n_bits += __popc(wds[e]);
                while (c_kt >= ktiles) { c_kt -= ktiles; ++c_ti; }
                if (c_kt + G >= ktiles) {
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(pops + (uint32_t)(((c_ti % C::SLOTS) * G + grp) * C::POP_ROWS + row) * 4u), "r"(n_bits) : "memory");
                    n_bits = 0;
                }
                c_kt += G;
            };
            if (is_w) {
                const uint32_t wds[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
                if (COLUMN_COUNTS) count(wds);
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) break;
                const uint32_t row_addr = wring + (uint32_t)s * C::W_BYTES + (uint32_t)row * ROWB;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    uint32_t v[4];
                    if (COLUMN_COUNTS) {
                        const uint4 o = expand_w4(wds[e]);
                        v[0] = o.x; v[1] = o.y; v[2] = o.z; v[3] = o.w;
                    } else {
                        expand_a4(wds[e], v);
                    }
                    st_shared_v4(row_addr + (uint32_t)((e ^ (row & 7)) << 4), v[0], v[1], v[2], v[3]);
                }
                if (!C::EARLY) {
                    if (l_left > 0) issue_load();
                    cp_async_commit();
                }
                fence_async_proxy();          // generic stores -> the MMAs
            } else {
                uint32_t v[32];
                if (C::SIGNED_A) {
                    const uint32_t wds[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const uint4 o = expand_w4(wds[e]);
                        v[4 * e] = o.x; v[4 * e + 1] = o.y; v[4 * e + 2] = o.z; v[4 * e + 3] = o.w;
                    }
                    count(wds);
                } else {
                    expand_stage8(q0, q1, v);
                }
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) break;
                tc_fence_after();             // the MMAs that read this slot are complete (their commit released it)
                tc_st32_nowait(st_addr0 + (uint32_t)s * 32u, v);
                if (!C::EARLY) {              // the next copies are issued while the store completes
                    if (l_left > 0) issue_load();
                    cp_async_commit();
                }
                tc_wait_st();
                tc_fence_before();
            }
            __syncwarp();
            if (PAIR) arrive_in_cluster(full0 + 8u * s, lane0);
            else mbar_arrive_pred(full0 + 8u * s, lane0);
            s += G;
            if (s >= STAGES) { s -= STAGES; phase ^= 1u; }
        }
        if (PAIR && RAW && rank != 0 && wi == 0 && it >= total_items) {      // as the loader above, which raw weights have not: the ring's next pass, but for its work
#pragma unroll 1
            for (; it < total_items + STAGES; it += G) {
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) break;
                s += G;
                if (s >= STAGES) { s -= STAGES; phase ^= 1u; }
            }
        }
        cp_async_wait<0>();
    }

    tc_fence_before();
    if (PAIR) cluster_barrier();               // nothing of the other CTA's refers to this one's memory any more
    else __syncthreads();
    if (warp == 0) {
        if (PAIR) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
        else asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// One weight word -> its 32 signed 4-bit codes (expand_w4), 16 bytes of a K-major row of k_pad / 2 bytes; padded rows and K
// words are zero.
__global__ void __launch_bounds__(256)
prepare_weights_kernel(const uint32_t *w, uint8_t *wexp, int32_t *cst, int N, int kwords, int n_pad, int k_pad)
{
    pdl_trigger();
    pdl_wait();
    const int kw_pad = k_pad / 32;
    const long total = (long)n_pad * kw_pad;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long)gridDim.x * blockDim.x) {
        const int kw = (int)(i % kw_pad), n = (int)(i / kw_pad);
        const bool live = n < N && kw < kwords;
        *reinterpret_cast<uint4 *>(wexp + i * 16) = live ? expand_w4(__ldg(w + (long)n * kwords + kw)) : make_uint4(0u, 0u, 0u, 0u);
    }
    for (long n = (long)blockIdx.x * blockDim.x + threadIdx.x; n < n_pad; n += (long)gridDim.x * blockDim.x) {
        int pop = 0;
        if (n < N)
            for (int kw = 0; kw < kwords; ++kw) pop += __popc(__ldg(w + n * kwords + kw));
        cst[n] = n < N ? kwords * 32 - 2 * pop : 0;
    }
}

int ktab_words_for(const ConvProblem &p) { return ((p.kwords + 7) >> 3) * (8 / gather_width(p.cw)); }

// int32 rows that are no whole number of 32-byte sectors: the sectors at the tile columns' borders and at the ends of the rows are written
// by two tiles.  With a column of tiles finished before the next is begun they leave the second-level cache half written and come back
// (300000 x 218 x 384: 57 MB read where the operands are 14; 314286 x 364 x 64 191 -> 117 us across the columns, 126000 x 507 x 576 120 -> 74,
// 150000 x 756 x 128 163 -> 113, 30912 x 4305 x 864 250 -> 166).  Not where the output stays in the cache (6157 x 645 x 224 7.8 -> 8.4), where K is long
// enough to be the time - blocks beside one another then fetch as many weight columns (94316 x 299 x 4320 79 -> 85) - or where the last column is so
// empty that its blocks idle (178587 x 135 x 96 33 -> 42).  A grid that is a multiple of the columns may leave an eighth of the blocks idle.
bool walk_across(const ConvProblem &p, int bn, long units)
{
    const long n_tiles = ((long)p.C_out + bn - 1) / bn;
    return p.mode == 0 && (p.C_out & 7) != 0 && n_tiles > 1 && n_tiles <= units && 8 * (units % n_tiles) <= units && p.kwords <= 56 &&
           (long)p.M * p.C_out >= 1L << 25 && 10L * p.C_out >= 7 * n_tiles * bn;
}

// pw.wexp == nullptr where the weights are raw (RAW)
template <int BN, int MODE, int G, int TEAMS, bool PAIR, int RAW = 0, bool WHOLE = false>
int launch_bn(const ConvProblem &p0, const PreparedWeights &pw, cudaStream_t stream)
{
    using C = Cfg<BN, MODE, G, TEAMS, PAIR, RAW, WHOLE>;
    ConvProblem p = p0;
    p.err = device_error_word();
    const long units = sm_count() / C::CTAS;
    const long m_tiles = ((long)p.M + C::TILE_ROWS - 1) / C::TILE_ROWS;
    const long n_tiles = ((long)p.C_out + BN - 1) / BN;
    const long total = m_tiles * n_tiles;
    if (total >= (1L << 31)) return BCNN_ERR_UNSUPPORTED;
    const bool across = !PAIR && BN > 64 && walk_across(p, BN, units);
    const long rows = across ? (m_tiles < units / n_tiles ? m_tiles : units / n_tiles) : 0;
    const int grid = (int)(across ? rows * n_tiles : total < units ? total : units);
    const int ktw = ktab_words_for(p);
    const int smem = smem_bytes<C>(ktw, MODE);
    if (smem > MAX_SMEM) return BCNN_ERR_UNSUPPORTED;
    CUtensorMap wmap = {};
    if constexpr (!RAW) {
        EncodeTiledFn encode = encode_tiled_fn();
        if (!encode) return BCNN_ERR_CUDA;
        // rows of k_pad / 2 bytes; for a pair as (128 rows, half of them, row)
        const cuuint64_t pitch = (cuuint64_t)pw.k_pad / 2;
        const cuuint64_t dims[4] = {pitch, PAIR ? 64u : (cuuint64_t)pw.n_pad, 2, (cuuint64_t)pw.n_pad / 128};
        const cuuint64_t strides[3] = {pitch, 64 * pitch, 128 * pitch};
        const cuuint32_t box[4] = {(cuuint32_t)ROWB, PAIR ? 64u : (cuuint32_t)BN, 1, PAIR ? (cuuint32_t)BN / 128 : 1};
        const cuuint32_t estr[4] = {1, 1, 1, 1};
        if (encode(&wmap, CU_TENSOR_MAP_DATA_TYPE_UINT8, PAIR ? 4 : 2, const_cast<uint8_t *>(pw.wexp), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BCNN_ERR_CUDA;
    }
    auto k = conv_tc_pre_kernel<BN, MODE, G, TEAMS, PAIR, RAW, WHOLE>;
    if (!allow_smem((const void *)k, MAX_SMEM)) return BCNN_ERR_CUDA;
    return launch<C::CTAS>(k, (unsigned)(grid * C::CTAS), C::THREADS, smem, stream, p, pw.cst, wmap, ktw, make_tile_walk(p, C::TILE_ROWS, (int)m_tiles, (int)n_tiles, grid, across));
}

}  // namespace

void prepared_layout(int C_out, int K, PreparedWeights &pw, size_t &bytes)
{
    pw.n_pad = (C_out + 127) / 128 * 128;
    pw.k_pad = (K + 255) / 256 * 256;
    // the buffer's size is part of the interface: a byte per weight, of which the 4-bit codes take at most half
    bytes = (size_t)pw.n_pad * ((K + 127) / 128 * 128) + (size_t)pw.n_pad * 4;
    pw.wexp = nullptr;
    pw.cst = nullptr;
}

int launch_prepare_weights(const uint32_t *w, void *prepared, int C_out, int K, cudaStream_t stream)
{
    PreparedWeights pw;
    size_t bytes;
    prepared_layout(C_out, K, pw, bytes);
    uint8_t *wexp = static_cast<uint8_t *>(prepared);
    int32_t *cst = reinterpret_cast<int32_t *>(wexp + (size_t)pw.n_pad * pw.k_pad / 2);
    const long total = (long)pw.n_pad * (pw.k_pad / 32);
    const int blocks = (int)((total + 255) / 256 < 1184 ? (total + 255) / 256 : 1184);
    return launch(prepare_weights_kernel, blocks, 256, 0, stream, w, wexp, cst, C_out, K / 32, pw.n_pad, pw.k_pad);
}

// ---- the variant that allocates nothing -------------------------------------------------------------------------
// Some callers cannot hand the library a buffer for the prepared weights because they cannot allocate device memory
// at all at the point where they call: code that runs inside somebody else's memory plan (an inference server whose
// arena is sized before the model's layers are known, a plug-in that only ever receives its input and output
// tensors), or code running while allocation is forbidden or would synchronise the device.  For them the prepared
// form lives in this array: it is part of the library's image, so every GPU that loads the library holds these
// STATIC_PREPARED_BYTES until the process exits.  The host-side name of a __device__ array is only a stand-in; the
// kernels need its device address, fetched once per device with cudaGetSymbolAddress.
constexpr size_t STATIC_PREPARED_BYTES = (size_t)4 << 20;
static __device__ __align__(256) unsigned char g_static_prepared[STATIC_PREPARED_BYTES];

size_t static_prepared_capacity() { return STATIC_PREPARED_BYTES; }

// Device address of the array on the current device (nullptr on failure); looked up on a device's first call.
static void *static_prepared_address()
{
    static void *cache[64] = {nullptr};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    if (!cache[dev]) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_static_prepared) != cudaSuccess) return nullptr;
        cache[dev] = ptr;
    }
    return cache[dev];
}

int launch_conv_tc_pre_static(const ConvProblem &p, cudaStream_t stream)
{
    if (!conv_tc_pre_supports(p)) return BCNN_ERR_UNSUPPORTED;
    PreparedWeights pw;
    size_t bytes = 0;
    prepared_layout(p.C_out, p.K, pw, bytes);
    if (bytes > STATIC_PREPARED_BYTES) return BCNN_ERR_WORKSPACE;
    void *scratch = static_prepared_address();
    if (!scratch) return BCNN_ERR_CUDA;
    // the expansion rewrites every byte of the layout it uses (padding rows and K words as zeros), so nothing of an
    // earlier call's contents is ever read
    const int st = launch_prepare_weights(p.w, scratch, p.C_out, p.K, stream);
    if (st != BCNN_OK) return st;
    return launch_conv_tc_pre(p, scratch, stream);
}

bool conv_tc_pre_supports(const ConvProblem &p)
{
    if (p.mode != 0 && p.mode != 1) return false;
    if (p.mode == 1 && (p.C_out % 32 != 0)) return false;
    if (p.kh * p.kw > 31) return false;                       // one validity bit per tap
    if ((long)p.B * p.H * p.W * p.cw >= (1L << 31)) return false;     // rows address the input by 32-bit word offsets
    if (smem_bytes<Cfg<256, 1, 2, 2, false>>(ktab_words_for(p), 1) > MAX_SMEM) return false;      // (the widths below need no more, but for one)
    if ((long)p.kh * p.W * p.cw >= (1L << 27)) return false;  // a unit's word offset within the window
    return p.K <= (1 << 20);                                  // sums up to 4 K + 2 stay exact in fp32
}

// How a product is cut up: columns of a tile, two blocks on one, a tile handed over in one piece, the operand whose bits are counted.
namespace {
struct StreamPlan {
    int bn;
    bool pair, whole;
    int raw;
};

// Expected time of a plan, ns: a start, a term per tile of the longest block and one per 256-bit stage of it - by how the gather goes: four, two, one
// word at a time - and int32 outputs by the million, those beyond 30 million of rows of no whole sectors once more.  Fitted to 3929 drawn layers and
// products with every variant timed, and 3070 more with int32 rows; within 7 to 12 % (one standard deviation).
struct Rates {
    int bn, ctas, packed, raw, across;
    long start, tile, stage[3], out, ragged;
};
constexpr Rates RATES[] = {
    {64, 1, 1, 0, 0, 1950, 430, {190, 212, 274}, 0, 0},        {128, 1, 1, 0, 0, 2080, 590, {201, 217, 287}, 0, 0},
    {256, 1, 1, 0, 0, 1930, 1110, {296, 301, 330}, 0, 0},      {256, 2, 1, 0, 0, 2380, 1200, {283, 289, 324}, 0, 0},
    {64, 1, 0, 0, 0, 2740, 373, {165, 176, 231}, 706, 788},    {128, 1, 0, 0, 0, 3720, 128, {188, 168, 223}, 785, 857},
    {128, 1, 0, 0, 1, 3340, 1414, {194, 163, 215}, 143, 413},  {256, 1, 0, 0, 0, 3450, 1053, {305, 292, 318}, 635, 726},
    {256, 1, 0, 0, 1, 2510, 3663, {306, 290, 312}, 101, 330},  {256, 2, 0, 0, 0, 5350, 1409, {240, 226, 265}, 913, 574},
    {64, 1, 1, RAW_COLUMNS, 0, 2210, 415, {282, 307, 363}, 0, 0}, {128, 1, 1, RAW_COLUMNS, 0, 2330, 594, {388, 460, 519}, 0, 0},
    {128, 1, 1, RAW_ROWS, 0, 2350, 689, {390, 459, 529}, 0, 0},   {256, 2, 1, RAW_ROWS, 0, 2620, 1275, {405, 498, 557}, 0, 0},
    {64, 1, 0, RAW_COLUMNS, 0, 2840, 480, {259, 290, 341}, 750, 0}, {128, 1, 0, RAW_COLUMNS, 0, 3250, 330, {340, 416, 467}, 1030, 0},
    {128, 1, 0, RAW_ROWS, 0, 3220, 298, {354, 429, 500}, 993, 0}, {256, 2, 0, RAW_ROWS, 0, 6080, 1742, {384, 536, 600}, 1248, 0},
};

long estimate(const ConvProblem &p, const StreamPlan &plan)
{
    const int ctas = plan.pair ? 2 : 1, gw = gather_width(p.cw);
    const long units = sm_count() / ctas, rows = ((long)p.M + ctas * BM - 1) / (ctas * BM), columns = ((long)p.C_out + plan.bn - 1) / plan.bn, kt = (p.kwords + 7) >> 3;
    const int across = !plan.raw && !plan.pair && plan.bn > 64 && walk_across(p, plan.bn, units) ? 1 : 0;
    const long tiles = across ? (rows + units / columns - 1) / (units / columns) : (rows * columns + units - 1) / units, outputs = (long)p.M * p.C_out;
    for (const Rates &r : RATES)
        if (r.bn == plan.bn && r.ctas == ctas && r.packed == (p.mode == 1) && r.raw == plan.raw && r.across == across)
            return r.start + tiles * (r.tile + kt * r.stage[gw == 4 ? 0 : gw == 2 ? 1 : 2]) + outputs / 1000 * r.out / 1000 +
                   ((p.C_out & 7) != 0 && outputs > 30000000 ? (outputs - 30000000) / 1000 * r.ragged / 1000 : 0);
    return LONG_MAX;
}

StreamPlan prepared_plan(const ConvProblem &p)
{
    // Tile width: 256, 128 or 64 columns.  Narrow tiles spread a small layer over more multiprocessors and shorten its epilogue, but
    // every tile expands its activation rows again.  By the estimates above; the choice takes 0.6 % longer than the best width in the mean where the output
    // is packed, 2.6 % where it is int32.
    //   packed, us at 64 / 128 / 256: 3x3 256 -> 256 at M = 50176 25.3, 15.5, 13.2; M = 196 4.0, 4.3, 5.6; 512 -> 512 at M = 12544 26.4, 15.2, 14.8;
    //   3x3 128 -> 128 at M = 6272 3.9, 3.6, 4.7; 1x1 64 -> 3264 at 13320 37.4, 32.0, 22.4; int32: 5x5 128 -> 7216 at M = 572 22.2, 15.0, 11.9; 3x3 384 -> 859
    //   at 4680 21.2, 11.7, 10.9; 1x1 224 -> 645 at 6157 8.2, 7.8, 6.9; 384 -> 218 at 10000 6.8, 6.7, 7.5
    const int sms = sm_count();
    const long m_tiles = ((long)p.M + BM - 1) / BM, kt = (p.kwords + 7) / 8, outputs = (long)p.M * p.C_out;
    const bool packed = p.mode == 1;
    auto tiles_of = [&](int bn) { return m_tiles * (((long)p.C_out + bn - 1) / bn); };
    auto waves_of = [&](int bn) { return (tiles_of(bn) + sms - 1) / sms; };
    static_assert(smem_bytes<Cfg<64, 1, 2, 1, false>>(0, 1) <= smem_bytes<Cfg<256, 1, 2, 2, false>>(0, 1) && smem_bytes<Cfg<128, 1, 2, 1, false>>(0, 1) <= smem_bytes<Cfg<256, 1, 2, 2, false>>(0, 1) &&
                  smem_bytes<Cfg<64, 0, 2, 1, false>>(0, 0) <= smem_bytes<Cfg<256, 1, 2, 2, false>>(0, 1) && smem_bytes<Cfg<128, 0, 3, 2, false>>(0, 0) <= smem_bytes<Cfg<256, 1, 2, 2, false>>(0, 1) &&
                  smem_bytes<Cfg<256, 1, 2, 2, true>>(0, 1) <= smem_bytes<Cfg<256, 1, 2, 2, false>>(0, 1),
                  "what conv_tc_pre_supports vouches for is the packed 256-wide variant's shared memory");
    const StreamPlan narrow = {64, false, false, 0}, medium = {128, false, false, 0};
    if (p.C_out <= 64) return narrow;                     // (a wide tile would be part empty)
    // Two multiprocessors on a tile of 256 x 256: half the weight bytes from L2 and into shared memory.  That pays where the tensor pipe is
    // kept busy for long - what limits such a product is power, the clock falls to 1.6 GHz (seconds of 16384 x 16384 x 9216 in a row: int32
    // 978 -> 877 us, packed 774 -> 745; 25088 x 512 x 4608 33.1 -> 30.7 and 23.1 -> 22.7; 16384 x 16384 x 2304 packed 231 -> 218) - and costs a hand-over between
    // the two elsewhere (50176 x 256 x 2304, three waves: 13.2 -> 14.0)
    const bool long_k = waves_of(256) >= 3 && p.K >= 4096;
    const StreamPlan pair = {256, true, false, 0};
    if (packed) {
        // tiles that start at the same time wait for one another's rows: 7 ns each
        auto cost = [&](const StreamPlan &s) { return estimate(p, s) + 7 * (tiles_of(s.bn) < sms ? tiles_of(s.bn) : sms); };
        const StreamPlan wide = {256, false, false, 0};
        const long c64 = cost(narrow), c128 = cost(medium), c256 = p.C_out > 128 ? cost(wide) : LONG_MAX;
        if (c64 < c128 && c64 <= c256) return narrow;
        return c128 <= c256 ? medium : waves_of(256) >= 8 || long_k ? pair : wide;
    }
    // int32.  A 256-wide tile of one block goes to memory in one piece, whole pieces of 128 columns at a time (0.79 of the time in halves, in the mean over 238
    // products); in halves only between two blocks, where its stores run beside the next tile's long K.  It needs its store staging tiles besides what
    // conv_tc_pre_supports vouches for: a K beyond 274 176 bits with an odd number of words per pixel, 548 352 with an even one, runs on narrower tiles.
    static_assert(smem_bytes<Cfg<256, 0, 2, 2, true>>(0, 0) <= smem_bytes<Cfg<256, 0, 2, 2, false, 0, true>>(0, 0), "and the tile of two blocks");
    const bool fits256 = p.C_out > 128 && smem_bytes<Cfg<256, 0, 2, 2, false, 0, true>>(ktab_words_for(p), 0) <= MAX_SMEM;
    const StreamPlan whole = {256, false, true, 0};
    // Rows of no whole sectors, more of them than the second-level cache holds, in one column of tiles: no neighbour has to fill them (us, tiles of 128 and
    // whole: 300000 x 218 x 384 109 and 71, 500000 x 146 x 768 149 and 108, 31405 x 138 x 3200 21.0 and 16.4; 300000 x 243 x 64, one stage, 83 and 98; of 64
    // and 128: 744810 x 90 x 128 172 and 74)
    if ((p.C_out & 7) != 0 && p.C_out <= 128 && outputs >= 1L << 25) return medium;
    if ((p.C_out & 7) != 0 && p.C_out <= 256 && fits256 && !long_k &&
        ((outputs >= 1L << 24 && (kt > 1 || p.C_out < 232)) || (kt >= 10 && outputs >= 1L << 22)))
        return whole;
    // One stage: the stores are the time, and over several waves 64-wide tiles of half-full columns take longer than the estimate has it (us at 64 and
    // 128: 5301 x 860 x 32, four waves, 9.0 and 7.5; 25435 x 120 x 64 6.7 and 6.0)
    const long c64 = kt == 1 && waves_of(64) > 2 ? LONG_MAX : estimate(p, narrow), c128 = estimate(p, medium);
    const long c256 = fits256 ? estimate(p, whole) / 20 * 21 : LONG_MAX, c_pair = fits256 && (waves_of(256) >= 8 || long_k) ? estimate(p, pair) : LONG_MAX;
    if (c64 <= c128 && c64 <= c256 && c64 <= c_pair) return narrow;
    if (c128 <= c256 && c128 <= c_pair) return medium;
    return c256 <= c_pair ? whole : pair;
}

// ---- raw weights: the streaming engine's packed and int32 outputs
StreamPlan raw_plan(const ConvProblem &p)
{
    const bool packed = p.mode == 1;
    // As for prepared weights, fitted to 20 products (packed, us at 64 / 128 / a pair's 256 columns: 4096 x 4096 x 4608 85.6, 53.1, 37.8; 2048 x
    // 2048 x 4608 26.3, 17.6, 13.6; 300 x 4000 x 9216 25.2, 17.0, 19.6; 1024 x 1024 x 4608 8.7, 10.3, 12.2; 20 x 64 x 960 3.5, 4.3, 5.5; int32: 4096 x 4096 x 4608 89.7, 56.7,
    // 53.4; 12544 x 512 x 4608 39.9, 27.4, 29.6; 34 x 3712 x 608 4.2, 5.4, 10.5)
    const int sms = sm_count(), ktw = ktab_words_for(p);
    const long kt = (p.kwords + 7) / 8;
    auto cost = [&](int rows, int bn, int units, long start, long wave, long stage) {
        const long tiles = (((long)p.M + rows - 1) / rows) * ((p.C_out + bn - 1) / bn);
        return start + (tiles + units - 1) / units * (wave + kt * stage);
    };
    const long c64 = cost(BM, 64, sms, 2500, packed ? 450 : 700, 300), c128 = cost(BM, 128, sms, 3000, packed ? 700 : 1200, 360);
    const bool fits = smem_bytes<Cfg<256, 0, 2, 2, true, RAW_ROWS>>(ktw, 0) <= MAX_SMEM;
    const long c256 = fits ? cost(2 * BM, 256, sms / 2, packed ? 3900 : 6500, packed ? 900 : 4900, 415) : LONG_MAX;
    if (c64 <= c128 && c64 <= c256) return {64, false, false, RAW_COLUMNS};
    if (c128 <= c256) return {128, false, false, kt < 8 ? RAW_COLUMNS : RAW_ROWS};
    return {256, true, false, RAW_ROWS};
}

// the kernels for prepared weights and for raw ones
template <int MODE>
int launch_plan(const StreamPlan &plan, const ConvProblem &p, const PreparedWeights &pw, cudaStream_t stream)
{
    if (plan.raw) {
        if (plan.bn == 64) return launch_bn<64, MODE, 2, 1, false, RAW_COLUMNS>(p, pw, stream);
        if (plan.bn == 128) return plan.raw == RAW_COLUMNS ? launch_bn<128, MODE, 2, 1, false, RAW_COLUMNS>(p, pw, stream) : launch_bn<128, MODE, 2, 1, false, RAW_ROWS>(p, pw, stream);
        return launch_bn<256, MODE, 2, 2, true, RAW_ROWS>(p, pw, stream);
    }
    if (plan.bn == 64) return launch_bn<64, MODE, 2, 1, false>(p, pw, stream);
    if (plan.bn == 128) return launch_bn<128, MODE, MODE == 0 ? 3 : 2, MODE == 0 ? 2 : 1, false>(p, pw, stream);
    return plan.pair ? launch_bn<256, MODE, 2, 2, true>(p, pw, stream) : launch_bn<256, MODE, 2, 2, false, 0, MODE == 0>(p, pw, stream);
}

// the gather's table at its longest fits beside every raw variant
template <int BN, int G, int TEAMS, bool PAIR, int RAW>
constexpr bool raw_fits() { return smem_bytes<Cfg<BN, 0, G, TEAMS, PAIR, RAW>>(MAX_RAW_KTAB, 0) <= MAX_SMEM && smem_bytes<Cfg<BN, 1, G, TEAMS, PAIR, RAW>>(MAX_RAW_KTAB, 1) <= MAX_SMEM; }
static_assert(raw_fits<64, 2, 1, false, RAW_COLUMNS>() && raw_fits<128, 2, 1, false, RAW_COLUMNS>() && raw_fits<128, 2, 1, false, RAW_ROWS>() && raw_fits<256, 2, 2, true, RAW_ROWS>(),
              "what conv_tc_i8_supports vouches for");

}  // namespace

int launch_conv_tc_pre(const ConvProblem &p, const void *prepared, cudaStream_t stream)
{
    if (!conv_tc_pre_supports(p)) return BCNN_ERR_UNSUPPORTED;
    PreparedWeights pw;
    size_t bytes;
    prepared_layout(p.C_out, p.K, pw, bytes);
    pw.wexp = static_cast<const uint8_t *>(prepared);
    pw.cst = reinterpret_cast<const int32_t *>(pw.wexp + (size_t)pw.n_pad * pw.k_pad / 2);
    const StreamPlan plan = prepared_plan(p);
    return p.mode == 1 ? launch_plan<1>(plan, p, pw, stream) : launch_plan<0>(plan, p, pw, stream);
}

// ---- raw weights: the streaming engine's packed and int32 outputs
int launch_conv_tc_raw(const ConvProblem &p, cudaStream_t stream)
{
    const StreamPlan plan = raw_plan(p);
    return p.mode == 1 ? launch_plan<1>(plan, p, PreparedWeights{}, stream) : launch_plan<0>(plan, p, PreparedWeights{}, stream);
}

long conv_tc_stream_estimate(const ConvProblem &p, bool raw) { return estimate(p, raw ? raw_plan(p) : prepared_plan(p)); }

// Columns of a tile, blocks on one, 1 where it is handed over whole, the operand whose bits are counted (0: none), 256-bit stages, the most tiles
// of a block.
void conv_tc_stream_plan(const ConvProblem &p, bool raw, int (&out)[6])
{
    const StreamPlan plan = raw ? raw_plan(p) : prepared_plan(p);
    const long ctas = plan.pair ? 2 : 1, units = sm_count() / ctas, tiles = ((long)p.M + ctas * BM - 1) / (ctas * BM) * (((long)p.C_out + plan.bn - 1) / plan.bn);
    out[0] = plan.bn;
    out[1] = (int)ctas;
    out[2] = plan.whole ? 1 : 0;
    out[3] = plan.raw;
    out[4] = (p.kwords + 7) >> 3;
    out[5] = (int)((tiles + units - 1) / units);
}

}  // namespace bcnn
