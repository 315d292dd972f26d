// Wide pointwise engine: binary 1x1 convolutions (stride 1, no padding) and plain GEMMs with K = 128, 256 or 512 bits
// and a multiple of 128 output channels, packed output - the deeper binary 1x1 convolutions of the paper's network (Section
// 4.2.1; Table 1: 256 and 512 channels at 56 x 56 ... 14 x 14).  A 128-row tile of such a layer is only 8 or 16 words of
// K per row and a few hundred tensor-pipe cycles per 128 output channels: the engines that cut the output channels
// into slices and walk the rows once per slice expand every activation row once per slice and pay a pipeline's
// start-up per slice and tile.
//
// Here a tile's activations are expanded ONCE and multiplied against all the weight slices the CTA keeps in shared
// memory (RS = 1 or 2 slices of 128 output channels, expanded once per CTA; the CTAs form C_out / 128 / RS groups and each
// group walks all row tiles).
//   * A row tile is a contiguous block of x (128 rows x K / 8 bytes): one bulk asynchronous copy (cp.async.bulk) per tile
//     into a ring in shared memory, two loader warps taking alternate tiles.
//   * Tensor memory: two accumulators and a ring of activation UNITS of eight K words (32 columns; four words for K = 128); a
//     tile is one unit, or two for K = 512 (filled by two producer groups).  Four producer groups of four warps (thread = row: two
//     16-byte shared-memory loads, 40 logic operations, one tensor-memory store).
//   * A tile's output channels are cut into PARTS of 128 (one slice each).  Two issuer warps walk the tiles in order and take
//     alternate parts, each with its own accumulator and epilogue group: per part an issuer waits for its accumulator, issues
//     the constant MMA (the constant rows of the slices sit side by side in one operand tile) and the K / 64 MMAs, and
//     commits on the part's "done" barrier.  One issuer's waits, fence and commit between two parts take about as long as
//     a short part's MMAs run; with two, one's MMAs run during the other's bookkeeping.
//   * The producers that reuse a unit wait for the last part of each issuer of the tile that used it.
// Arithmetic: 4-bit operands (tc_common.cuh), fp32 accumulators that hold exact integers, the per-channel constants
// K - 2 popc(G) - threshold written by a first MMA so that the epilogue needs 16 bits and a sign (tc_slot.cuh; the weight
// rows are laid out in that gathering's column order).
// "Done" numbers d = tile * parts + part use barrier d % 64.  A parity wait is only right while the waiter starts waiting
// for completion k after k - 1 and before k + 1: the epilogue group of d takes its barrier's completions in turn, and
// its issuer cannot get past part d + 2 (it needs the accumulator of d back), let alone to d + 64; the producers that
// wait for d are those of a tile at most seven tiles later, which both issuers issue before the tile of d + 64 (a tile
// has at most four parts).
// Every mbarrier wait is bounded and reports through the device error word.
#include "tc_slot.cuh"

namespace bcnn {

namespace {

using namespace tc;

constexpr int ERR_PN_LOADER_TIMEOUT = 151;       // loader: no free ring stage
constexpr int ERR_PN_PRODUCER_TIMEOUT = 152;     // producer: the tile's rows did not arrive
constexpr int ERR_PN_ISSUER_TIMEOUT = 153;       // issuer: a tile's activations were not filled
constexpr int ERR_PN_EPILOGUE_TIMEOUT = 154;     // epilogue: a slice's MMAs did not complete
constexpr int ERR_PN_UNIT_TIMEOUT = 155;         // producer: the unit's previous MMAs did not complete
constexpr int ERR_PN_ACC_TIMEOUT = 156;          // issuer: an accumulator was not handed back

constexpr int NGRP = 2;                   // loader / epilogue groups
constexpr int NPG = 4;                    // producer groups of four warps
constexpr int RD = 4;                     // row tiles in a loader's ring
constexpr int BN = 128;                   // output channels per weight slice (rows of a weight tile)
constexpr int NB = 64, NAF = 8;
constexpr int MAX_TILES = 7;              // row tiles in the ring of units
constexpr int NISS = 2;                   // issuer warps (parts alternate)
constexpr int MAX_NACC = 4;
constexpr int FIRST_LOADER_WARP = 2, FIRST_PRODUCER_WARP = 4, FIRST_EPILOGUE_WARP = 4 + 4 * NPG;
constexpr int WARPS = 4 + 4 * NPG + 4 * NGRP;
constexpr int THREADS = 32 * WARPS;
constexpr int W_TILE_BYTES = BN * ROWB;   // one 256-bit stage of one slice's expanded weights

struct PnPlan {
    int rs;            // resident slices per CTA (1 or 2)
    int ng;            // CTA groups = slices / rs
    int m_tiles;
};

// UPT: units per tile; UWORDS: K words per unit (8; 4 for K = 128)
template <int UPT, int UWORDS>
__global__ void __launch_bounds__(THREADS, 1)
conv_tc_pn_kernel(const ConvProblem p, const PnPlan plan)
{
    constexpr int KWORDS = UWORDS * UPT, KT = (KWORDS + 7) / 8, U_COLS = 4 * UWORDS;
    constexpr int TILE_BYTES = BM * KWORDS * 4;
    constexpr int NBARS = 2 * NGRP * RD + NAF + NB + MAX_NACC;
    // an accumulator per issuer / epilogue group; beside them seven tiles (three for K = 512)
    constexpr int NACC = 2, NU0 = (CB_COL - NACC * BN) / U_COLS / UPT * UPT, NUNIT = NU0 < MAX_TILES ? NU0 : MAX_TILES;
    constexpr int A_COL0 = NACC * BN;
    static_assert(NUNIT / UPT <= MAX_TILES && MAX_TILES < NAF, "ring of tile-full barriers");

    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[NBARS];
    __shared__ uint32_t tmem_base_smem;
    __shared__ int abort_flag_smem;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int RS = plan.rs, PARTS = plan.rs;               // resident slices = parts per tile
    // CTA group cg keeps the slices cg * RS .. cg * RS + RS - 1; the CTAs of a group share the row tiles
    const int cg = (int)blockIdx.x % plan.ng, idx = (int)blockIdx.x / plan.ng, per_group = (int)gridDim.x / plan.ng;
    const int my_tiles = idx < plan.m_tiles ? (plan.m_tiles - 1 - idx) / per_group + 1 : 0;
    auto row_tile = [&](int n) { return idx + n * per_group; };

    const uint32_t wexp = (smem_u32(smem_raw) + 1023u) & ~1023u;          // [RS][KT][128 rows][128 B] expanded weights
    const uint32_t cexp = wexp + (uint32_t)(RS * KT) * W_TILE_BYTES;      // [128 rows][128 B]: 32-byte piece s = constant row of slice s
    const uint32_t pops = cexp + W_TILE_BYTES;                            // [RS][BN] bit counts
    const uint32_t ring = pops + (uint32_t)(RS * BN) * 4u;                // [NGRP][RD] row tiles
    const uint32_t bar0 = smem_u32(bars);
    auto load_full = [&](int gr, int s) { return bar0 + 8u * (gr * RD + s); };
    auto load_empty = [&](int gr, int s) { return bar0 + 8u * (NGRP * RD + gr * RD + s); };
    auto a_full = [&](int s) { return bar0 + 8u * (2 * NGRP * RD + s); };
    auto tile_done = [&](int s) { return bar0 + 8u * (2 * NGRP * RD + NAF + s); };
    auto acc_free = [&](int s) { return bar0 + 8u * (2 * NGRP * RD + NAF + NB + s); };
    volatile int *abort_flag = &abort_flag_smem;

    if (tid == 0) {
        for (int s = 0; s < NGRP * RD; ++s) {
            mbar_init(load_full(0, s), 1);              // the loader's arrive (+ the copy's bytes)
            mbar_init(load_empty(0, s), 4 * UPT);       // the producer warps that read the stage
        }
        for (int s = 0; s < NAF; ++s) mbar_init(a_full(s), 4 * UPT);    // the producer warps that fill the tile's units
        for (int s = 0; s < NB; ++s) mbar_init(tile_done(s), 1);        // the issuer's commit
        for (int s = 0; s < MAX_NACC; ++s) mbar_init(acc_free(s), 4);   // the four warps of the epilogue group that reads it
        abort_flag_smem = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_wait();
    // The loader warps start now: the first row tiles arrive while the other warps expand the weights (these kernels
    // run for 10 - 40 us; the weights' expansion and the first copy's latency are 1.5 - 2 us each).  The other warps meet
    // at a named barrier of their own; everybody meets again at the end.
    const bool is_loader = warp >= FIRST_LOADER_WARP && warp < FIRST_PRODUCER_WARP;
    auto sync_workers = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(THREADS - 64) : "memory"); };
    if (!is_loader) {
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int i = tid < 64 ? tid : tid - 64; i < RS * BN; i += THREADS - 64) asm volatile("st.shared.b32 [%0], %1;" ::"r"(pops + 4u * i), "r"(0) : "memory");
    sync_workers();
    // ---- one-off: the resident slices' expanded weights and constants; MMA row `row` of slice s carries channel ch.  Eight
    // lanes take the words of one 256-bit stage; a row's bit count is collected in shared memory.  WU words in flight per thread.
    constexpr int WU = 4, NW = THREADS - 64;                              // (threads 64 .. 127 are the loaders)
    const int wt = tid < 64 ? tid : tid - 64, wtotal = RS * BN * KWORDS;
    for (int i0 = wt; i0 < wtotal; i0 += WU * NW) {
        uint32_t w[WU];
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int i = i0 + u * NW, e = i % KWORDS, rw = i / KWORDS, row = rw % BN;
            const int ch = (cg * RS + rw / BN) * BN + (row & ~31) + channel_of_column(row & 31);
            w[u] = i < wtotal && ch < p.C_out ? __ldg(p.w + (long)ch * KWORDS + e) : 0u;
        }
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int i = i0 + u * NW, e = i % KWORDS, rw = i / KWORDS, row = rw % BN, s = rw / BN;
            if (i >= wtotal) break;                                       // (warp-uniform: wtotal is a multiple of 32)
            const int ch = (cg * RS + s) * BN + (row & ~31) + channel_of_column(row & 31);
            const bool have = ch < p.C_out;
            expand_store_w4(w[u], have, wexp + (uint32_t)(s * KT + (e >> 3)) * W_TILE_BYTES + (uint32_t)row * ROWB, row & 7, e & 7);
            int pop = __popc(w[u]);
            pop += __shfl_xor_sync(0xffffffffu, pop, 1);
            pop += __shfl_xor_sync(0xffffffffu, pop, 2);
            if (KWORDS >= 8) pop += __shfl_xor_sync(0xffffffffu, pop, 4);
            if (KWORDS >= 8 ? (e & 7) == 0 : (e & 3) == 0) asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(pops + 4u * rw), "r"(pop) : "memory");
        }
    }
    tc_fence_before();
    sync_workers();
    tc_fence_after();
    for (int rw = wt; rw < RS * BN; rw += NW) {
        const int row = rw % BN, s = rw / BN, ch = (cg * RS + s) * BN + (row & ~31) + channel_of_column(row & 31);
        int pop;
        asm volatile("ld.shared.b32 %0, [%1];" : "=r"(pop) : "r"(pops + 4u * rw) : "memory");
        const bool have = ch < p.C_out;
        const int t = have ? __ldg(p.thr + ch) : 0;
        // K - 2 popc - thr (thr clamped to +-(K + 1)); 32-byte piece s of the row: XOR with s * 2 in 16-byte units
        store_const_row(have ? p.K - 2 * pop - max(min(t, p.K + 1), -p.K - 1) : 0, cexp + (uint32_t)row * ROWB, (row & 7) ^ (2 * s));
    }
    if (warp >= FIRST_PRODUCER_WARP && warp < FIRST_PRODUCER_WARP + 4) write_const_block(tmem_base_smem + ((uint32_t)((warp & 3) * 32) << 16));
    fence_async_proxy();
    tc_fence_before();
    sync_workers();
    tc_fence_after();
    pdl_trigger();
    }
    const uint32_t tmem_base = is_loader ? 0u : tmem_base_smem;

    if (warp < NISS) {
        // ------------------------------------------------------------------ MMA issuer of the parts d = warp (mod 2), in order.
        // (One issuer's waits, fence and commit between two parts take about as long as a part's MMAs run: with two
        // issuers one's MMAs run during the other's bookkeeping.)
        constexpr uint32_t idesc = make_idesc_f4(BN);
        const uint64_t desc0 = make_desc(wexp);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32), b_lo = (uint32_t)desc0;
        const uint32_t c_lo = (uint32_t)make_desc(cexp);
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t sf = tmem_u + (uint32_t)CB_COL;
        bool ok = true;
        for (int n = 0; n < my_tiles && ok; ++n) {
            if (!pw_wait(a_full(n % NAF), (uint32_t)(n / NAF) & 1u, abort_flag, p.err, ERR_PN_ISSUER_TIMEOUT)) break;
            for (int j = warp; j < PARTS; j += NISS) {
                const int d = n * PARTS + j;                                      // "done" number
                const int acc = d % NACC;
                if (d >= NACC) {                  // the epilogue has read the accumulator's previous contents
                    ok = pw_wait(acc_free(acc), (uint32_t)(d / NACC - 1) & 1u, abort_flag, p.err, ERR_PN_ACC_TIMEOUT);
                    if (!ok) break;
                }
                tc_fence_after();
                if (elect_one()) {
                    const uint32_t d_t = tmem_u + (uint32_t)(acc * BN);
                    const uint32_t w_lo = b_lo + (uint32_t)(j * KT) * (W_TILE_BYTES >> 4);
                    tc_mma_const(d_t, tmem_u, c_lo + 2u * j, desc_hi, idesc);          // accumulator = the constants of slice j
#pragma unroll
                    for (int h = 0; h < UPT; ++h) {
                        const uint32_t a_t = tmem_u + (uint32_t)(A_COL0 + ((n * UPT + h) % NUNIT) * U_COLS);
#pragma unroll
                        for (int t = 0; t < UWORDS / 2; ++t)
                            tc_mma_f4_ts(d_t, a_t + 8u * t, w_lo + (uint32_t)(h * (W_TILE_BYTES >> 4) + 2 * t), desc_hi, idesc, sf, 1u);
                    }
                    tc_commit(tile_done(d % NB));
                }
                __syncwarp();
            }
        }
    } else if (warp < FIRST_PRODUCER_WARP) {
        // ------------------------------------------------------------------ loader of group warp - 2: one row tile per bulk copy
        const int grp = warp - FIRST_LOADER_WARP;
        int stage = 0;
        uint32_t phase = 1;                       // first pass through the ring: the stages are free
        int issued = 0;
        for (int n = grp; n < my_tiles; n += NGRP) {
            if (!pw_wait<256>(load_empty(grp, stage), phase, abort_flag, p.err, ERR_PN_LOADER_TIMEOUT)) break;
            if (lane == 0) {
                const long row0 = (long)row_tile(n) * BM;
                const long rows = min((long)BM, (long)p.M - row0);                // rows beyond M keep whatever the stage held
                const uint32_t bytes = (uint32_t)rows * KWORDS * 4u;              // a multiple of 32
                const uint32_t dst = ring + (uint32_t)(grp * RD + stage) * TILE_BYTES;
                const uint32_t *src = p.x + row0 * KWORDS;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(load_full(grp, stage)), "r"(bytes) : "memory");
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(dst), "l"(src), "r"(bytes), "r"(load_full(grp, stage)) : "memory");
            }
            __syncwarp();
            ++issued;
            if (++stage == RD) { stage = 0; phase ^= 1u; }
        }
        // after a time-out elsewhere: copies still in flight must land before the CTA's shared memory goes away
        if (*abort_flag) {
            const int first = issued > RD ? issued - RD : 0;
            for (int q = first; q < issued; ++q)
                pw_wait(load_full(grp, q % RD), (uint32_t)(q / RD) & 1u, abort_flag, nullptr, 0);
        }
    } else if (warp >= FIRST_EPILOGUE_WARP) {
        // ------------------------------------------------------------------ epilogue group (warp - first) / 4: "done" numbers d = group (mod 2)
        const int quad = warp & 3;
        const int grp = (warp - FIRST_EPILOGUE_WARP) >> 2;
        const int r = quad * 32 + lane;                           // row of the tile
        const uint32_t t_lane0 = tmem_base + ((uint32_t)(quad * 32) << 16);
        const int owords = p.C_out >> 5;
        const int total = my_tiles * PARTS;
        for (int d = grp; d < total; d += 2) {
            const int n = d / PARTS, j = d - n * PARTS, acc = d % NACC;
            const uint32_t t_lane = t_lane0 + (uint32_t)(acc * BN);
            if (!pw_wait<64>(tile_done(d % NB), (uint32_t)(d / NB) & 1u, abort_flag, p.err, ERR_PN_EPILOGUE_TIMEOUT)) break;
            tc_fence_after();
            uint32_t words[4];
            uint32_t rr[2][32];
#pragma unroll
            for (int h = 0; h < 2; ++h) tc_ld64_pack16(t_lane + (uint32_t)(h * 64), rr[h]);
            tc_wait_ld();
#pragma unroll
            for (int h = 0; h < 2; ++h) pin_regs(rr[h]);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_free(acc));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                words[2 * h] = sign_word(rr[h]);
                words[2 * h + 1] = sign_word(rr[h] + 16);
            }
            const long m = (long)row_tile(n) * BM + r;
            if (m < p.M) {
                *reinterpret_cast<uint4 *>(static_cast<uint32_t *>(p.out) + m * owords + (cg * PARTS + j) * 4) = make_uint4(words[0], words[1], words[2], words[3]);
            }
        }
    } else {
        // ------------------------------------------------------------------ producer group (warp - first) / 4
        // thread = row of the tile = tensor-memory lane.  The group fills unit h (K words 8 h .. 8 h + 7) of the tiles
        // n0, n0 + step, ...
        const int quad = warp & 3;
        const int grp = (warp - FIRST_PRODUCER_WARP) >> 2;
        const int h = UPT == 2 ? (grp & 1) : 0;
        const int n0 = UPT == 2 ? (grp >> 1) : grp, step = UPT == 2 ? NPG / 2 : NPG;
        const int r = quad * 32 + lane;
        const uint32_t my_off = (uint32_t)(r * KWORDS * 4 + h * UWORDS * 4);
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)A_COL0;
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        for (int n = n0; n < my_tiles; n += step) {
            const int lg = n & 1, stage = (n >> 1) % RD;
            if (!pw_wait<64>(load_full(lg, stage), (uint32_t)((n >> 1) / RD) & 1u, abort_flag, p.err, ERR_PN_PRODUCER_TIMEOUT)) break;
            const uint32_t src = ring + (uint32_t)(lg * RD + stage) * TILE_BYTES + my_off;
            const uint4 q0 = ld_shared_v4(src);
            uint4 q1 = q0;
            if (UWORDS == 8) q1 = ld_shared_v4(src + 16u);
            uint32_t v[32];                       // expanded before the wait for the unit
            expand_stage8(q0, q1, v);             // (four words: the second half is dropped)
            // the MMAs of the tile that used this ring position last have read it (nothing to wait for the first time round)
            const int u = n * UPT + h;
            if (u >= NUNIT) {
                const int dm = (u - NUNIT) / UPT * PARTS + PARTS - 1;         // that tile's last "done" numbers: one per issuer
                if (PARTS >= 2 && !pw_wait<64>(tile_done((dm - 1) % NB), (uint32_t)((dm - 1) / NB) & 1u, abort_flag, p.err, ERR_PN_UNIT_TIMEOUT)) break;
                if (!pw_wait<64>(tile_done(dm % NB), (uint32_t)(dm / NB) & 1u, abort_flag, p.err, ERR_PN_UNIT_TIMEOUT)) break;
            }
            tc_fence_after();
            const uint32_t taddr = t_lane + (uint32_t)((u % NUNIT) * U_COLS);
            if constexpr (UWORDS == 8) tc_st32_nowait(taddr, v);
            else tc_st16_nowait(taddr, reinterpret_cast<const uint32_t (&)[16]>(v[0]));
            // the stage may be refilled: its words have left through registers (handing it back right behind the loads
            // let a refill that hit L2 overtake them, on a CTA's first tiles: a few rows wrong in one launch of fifteen)
            __syncwarp();
            mbar_arrive_pred(load_empty(lg, stage), lane0);
            tc_wait_st();
            tc_fence_before();
            __syncwarp();
            mbar_arrive_pred(a_full(n % NAF), lane0);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

// Resident slices per CTA.  One: the fewest weights to expand at the start (0.8 us per K = 256 slice, 1.4 us per K = 512 slice),
// but every group expands all the rows; two share a row tile's expansion.  Two win once a CTA would walk more than a dozen row
// tiles with one (256 x 256 at M = 802816: 39 -> 28 us, at 200704: 13.4 -> 11.3; 512 x 512 at M = 200704: 28.4 -> 23.9, at 50176:
// 11.0 -> 11.5); four never do (one issuer pair cannot use them).
int pn_resident_slices(int slices, int m_tiles, int sms) { return slices % 2 == 0 && (long)m_tiles * slices > 12L * sms ? 2 : 1; }

template <int UPT, int UWORDS>
int launch_pn(const ConvProblem &p0, cudaStream_t stream)
{
    constexpr int KWORDS = UWORDS * UPT, KT = (KWORDS + 7) / 8, TILE_BYTES = BM * KWORDS * 4;
    ConvProblem p = p0;
    p.err = device_error_word();
    PnPlan plan;
    const int slices = p.C_out / BN;
    plan.m_tiles = (p.M - 1) / BM + 1;
    const int sms = sm_count();
    plan.rs = pn_resident_slices(slices, plan.m_tiles, sms);
    plan.ng = slices / plan.rs;
    const int smem = 1024 + (plan.rs * KT + 1) * W_TILE_BYTES + plan.rs * BN * 4 + NGRP * RD * TILE_BYTES + 128;
    if (smem > 227 * 1024 - 1024) return BCNN_ERR_UNSUPPORTED;
    int per_group = sms / plan.ng;
    if (per_group > plan.m_tiles) per_group = plan.m_tiles;
    if (per_group < 1) per_group = 1;
    void (*k)(const ConvProblem, const PnPlan) = conv_tc_pn_kernel<UPT, UWORDS>;
    const int ask = smem < 120 * 1024 ? 120 * 1024 : smem;          // one CTA per SM (it takes all of tensor memory)
    if (!allow_smem((const void *)k, 227 * 1024 - 1024)) return BCNN_ERR_CUDA;
    return launch(k, (unsigned)(per_group * plan.ng), THREADS, ask, stream, p, plan);
}

}  // namespace

bool conv_tc_pn_supports(const ConvProblem &p)
{
    if (p.mode != 1) return false;                               // packed output only
    if (!(p.kh == 1 && p.kw == 1 && p.stride == 1 && p.pad == 0)) return false;
    if (p.kwords != 4 && p.kwords != 8 && p.kwords != 16) return false;      // K = 128, 256 or 512
    return p.C_out % BN == 0 && p.C_out <= 16 * BN;
}

int launch_conv_tc_pn(const ConvProblem &p, cudaStream_t stream)
{
    if (!conv_tc_pn_supports(p)) return BCNN_ERR_UNSUPPORTED;
    return p.kwords == 4 ? launch_pn<1, 4>(p, stream) : (p.kwords == 8 ? launch_pn<1, 8>(p, stream) : launch_pn<2, 8>(p, stream));
}

}  // namespace bcnn
