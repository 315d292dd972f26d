// Short-K 3x3 engine: binary 3x3 convolutions (stride 1 or 2) on 32 or 64 input channels with up to 128 output
// channels, packed output - the stem / down-sampling shaped layers and the first 3x3 layers of the backbone, where a
// 128-row tile is nine or eighteen 32-bit words of K per row and the weight-stationary engine spends most of its
// instructions on the gather (a table look-up, a mask test and a 4-byte cp.async per K word).
//
// The implicit im2col is done by TMA:
//   * an output tile is a TH x TW = 8 x 16 patch of output pixels of one image (128 rows of the patch matrix);
//   * its input halo - ((TH-1) s + 3) rows x ((TW-1) s + 3) pixels x C_in bits - arrives by ONE tiled TMA copy
//     (cp.async.bulk.tensor.3d over the packed input seen as [B][H][W * C_in / 32 words]) into a ring in shared
//     memory.  Out-of-image rows and pixels are the copy's zero fill = the -1 padding: no tap masks anywhere.  The
//     copy's first word must be 16-byte aligned, so the box starts up to three pixels left of the halo (XOFF);
//   * a producer thread (= one output pixel) reads its nine pixels' words from the halo tile at compile-time offsets,
//     expands them and stores them to tensor memory: per K word one shared-memory load and five logic operations.
// Arithmetic: 4-bit operands (tc_common.cuh), fp32 accumulators that hold exact integers, the per-channel constants written by
// a first MMA so that the epilogue needs 16 bits and a sign (tc_slot.cuh).
//
// One commit per tile.  Tensor memory holds NACC accumulators and a ring of NUNIT activation UNITS: the nine taps of
// 32 input channels of one tile, 40 columns (ten words of K: two per MMA, the tenth meets zero weights).  A tile is one unit
// for C_in = 32 and two for C_in = 64 (K order: channel word, then tap).  Two issuer warps take alternate tiles (an issuer's
// waits, its 5 or 10 instructions and its commit take about as long as a tile's MMAs run; 128 output channels: a half of every
// tile each, 3x3 64 -> 128 /2 at M = 200704 15.2 us with one issuer, 14.2 with two; four issuers on alternate tiles gain
// nothing): wait until the tile's units are
// full and its accumulator free, issue the tile's MMAs and ONE commit on the tile's "done" barrier, which the epilogue
// (accumulator ready) and the producers (units free again) wait on.
// Four producer groups of four warps fill ONE unit of every tile they take:
//   * C_in = 64: groups 2 j and 2 j + 1 fill the two units of the tiles n = j (mod 2);
//   * C_in = 32: group j fills the tiles n = j (mod 4).
// Two loader warps and two epilogue groups take alternate tiles.
// The "done" barriers form a ring of NB = 16 (tile n -> barrier n % 16), a multiple of NACC and more than the tiles in
// flight.
// A parity wait on an mbarrier is only right while the waiter starts waiting for completion k after completion k - 1 and
// before completion k + 1.  Tile m's "done" is completion m / NB of its barrier; its waiters are the epilogue of tile m and
// the producers of tile m + D, D = NUNIT / CW <= NB / 2, which reuse its units.  A producer group's tiles are an even number
// apart, so its wait before this one was for an earlier tile of the same issuer, and an issuer's tiles complete in order:
// completion k - 1 has happened.  Tile m + NB cannot be done before the waiter is through: the fills of the tiles from
// m + 2 D on need tile m + D (or a later one of its issuer) done, hence filled; NB being a multiple of NACC, it also needs the
// accumulator of tile m back from the epilogue.
// A launch's set-up - barriers by a thread each, divisions by the host, every role's wait for the previous kernel behind its own
// set-up - is half a microsecond of a small layer: 3x3 32 -> 64 /2 at M = 3136 3.0 -> 2.8 us, at M = 200704 6.15 -> 5.85; 64 -> 64 at M = 3136 3.6 -> 3.3.
// Every mbarrier wait is bounded and reports through the device error word.
#include "tc_slot.cuh"
#include "tensor_map.cuh"

namespace bcnn {

namespace {

using namespace tc;

constexpr int ERR_C3_LOADER_TIMEOUT = 141;       // loader: no free ring stage
constexpr int ERR_C3_PRODUCER_TIMEOUT = 142;     // producer: the tile's halo did not arrive
constexpr int ERR_C3_ISSUER_TIMEOUT = 143;       // issuer: a tile's activations were not filled
constexpr int ERR_C3_EPILOGUE_TIMEOUT = 144;     // epilogue: the tile's MMAs did not complete
constexpr int ERR_C3_UNIT_TIMEOUT = 145;         // producer: the unit's previous MMAs did not complete
constexpr int ERR_C3_ACC_TIMEOUT = 146;          // issuer: an accumulator was not handed back

constexpr int TH = 8, TW = 16;            // output tile (TH * TW = 128 = tensor-memory lanes)
constexpr int NGRP = 2;                   // epilogue groups (alternate tiles)
constexpr int NLD = 2;                    // loader warps (alternate tiles: n & 1, n >> 1; four with half the ring each: 34.9 -> 36.3 us on the first 3x3/2 layer)
static_assert(NLD == 2, "tile n: loader n & 1, its tile n >> 1");
constexpr int NPG = 4;                    // producer groups of four warps
constexpr int RD = 6;                     // halo tiles in a loader's ring
constexpr int TAPS = 9, UWORDS = 10;      // K words of a unit: the nine taps and a zero
constexpr int U_COLS = 4 * UWORDS;        // columns of a unit
constexpr int NB = 16;                    // ring of "tile done" barriers
constexpr int NAF = 8;                    // ring of "tile full" barriers (at most eight tiles are being filled)
constexpr int MAX_NUNIT = 8, MAX_NACC = 4;

// CW: words per input pixel (1, 2) = units per tile; BN: accumulator columns per tile (32, 64, 128 >= C_out).
template <int CW, int BN> struct C3Cfg {
    static constexpr int KW = TAPS * CW;                    // words of K per row
    static constexpr int KT = (UWORDS * CW + 7) / 8;        // 256-bit stages of the expanded weights
    // 128 output channels run as two halves of 64 against the same activation units, each with its accumulator, issuer and
    // epilogue group; the units are free again when both halves are done
    static constexpr int NH = BN == 128 ? 2 : 1;            // halves
    static constexpr int AW = BN / NH;                      // accumulator columns
    static constexpr int NACC = NH == 2 ? 2 : 4;            // accumulators (NH == 2: one per half)
    static constexpr int NISS = 2;                          // issuer warps: alternate tiles, or a half each
    static constexpr int NU0 = (CB_COL - NACC * AW) / U_COLS;
    static constexpr int NUNIT = NU0 >= MAX_NUNIT ? MAX_NUNIT : NU0 / CW * CW;   // 8 (32 columns), 6 (64), 8 (128)
    static constexpr int A_COL0 = NACC * AW;
    static_assert(A_COL0 + NUNIT * U_COLS <= CB_COL, "tensor memory budget");
    static_assert(NUNIT >= 2 * CW && NUNIT / CW <= NAF && 2 * (NUNIT / CW) <= NB && NB % NACC == 0 && NACC <= MAX_NACC && NACC % NISS == 0, "barrier rings");
    // warps: issuers, two loaders, then the producer groups, then the epilogue groups (warp % 4 is the tensor-memory lane
    // quadrant of a warp: any four consecutive warps cover all of them)
    static constexpr int FIRST_LOADER_WARP = NISS;
    static constexpr int FIRST_PRODUCER_WARP = FIRST_LOADER_WARP + NLD;
    static constexpr int FIRST_EPILOGUE_WARP = FIRST_PRODUCER_WARP + 4 * NPG;
    static constexpr int WARPS = FIRST_EPILOGUE_WARP + 4 * NGRP;
    static constexpr int THREADS = 32 * WARPS;
    static constexpr int W_TILE_BYTES = BN * ROWB;
};

struct C3Geom {
    int stride, xoff;        // XOFF: pixels between the box's first pixel and the halo's
    int wbw, hb;             // box: words per row, rows
    int stage_bytes;         // hb * wbw * 4 rounded up to 128
    int tiles_x, tiles_y;    // tiles per image row / column of tiles
    int total_tiles;
    int tiles, extra;        // tiles of every CTA; CTAs that have one more
    uint32_t img_mul, img_shift, row_mul, row_shift;      // exact_div by the tiles of an image and of a row of tiles
    struct Step {
        int db, dty, dtx;    // images, rows of tiles and tiles
    } step[2];               // one and two of the CTA's tiles further
};

C3Geom c3_geometry(const ConvProblem &p)
{
    C3Geom g;
    g.stride = p.stride;
    const int A = 4 / p.cw;                                  // pixels per 16 bytes
    g.xoff = (A - p.pad % A) % A;
    const int wpx = ((TW - 1) * p.stride + 3 + g.xoff + A - 1) / A * A;
    g.wbw = wpx * p.cw;
    g.hb = (TH - 1) * p.stride + 3;
    g.stage_bytes = (g.hb * g.wbw * 4 + 127) / 128 * 128;
    g.tiles_x = (p.OW + TW - 1) / TW;
    g.tiles_y = (p.OH + TH - 1) / TH;
    g.total_tiles = p.B * g.tiles_x * g.tiles_y;
    return g;
}
// what depends on the grid: the divisions, done here
void c3_walk(C3Geom &g, unsigned grid)
{
    const unsigned per_img = (unsigned)(g.tiles_x * g.tiles_y);
    g.tiles = (int)((unsigned)g.total_tiles / grid);
    g.extra = (int)((unsigned)g.total_tiles % grid);
    exact_div_params(per_img, g.img_mul, g.img_shift);
    exact_div_params((uint32_t)g.tiles_x, g.row_mul, g.row_shift);
    for (int i = 0; i < 2; ++i) {
        const unsigned st = grid << i, rem = st % per_img;
        g.step[i] = {(int)(st / per_img), (int)(rem / (unsigned)g.tiles_x), (int)(rem % (unsigned)g.tiles_x)};
    }
}

template <int CW, int BN>
int c3_smem_bytes(const C3Geom &g)
{
    using C = C3Cfg<CW, BN>;
    return 1024 + (C::KT + 1) * C::W_TILE_BYTES + (BN * 4 + 127) / 128 * 128 + NLD * RD * g.stage_bytes + 128;
}

template <int CW, int BN>
__global__ void __launch_bounds__(C3Cfg<CW, BN>::THREADS, 1)
conv_tc_c3_kernel(const ConvProblem p, const C3Geom g, const __grid_constant__ CUtensorMap xmap)
{
    using C = C3Cfg<CW, BN>;
    constexpr int KT = C::KT, NACC = C::NACC, NUNIT = C::NUNIT, NH = C::NH, AW = C::AW;
    constexpr int NBARS = 2 * NLD * RD + NAF + NB + MAX_NACC;

    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[NBARS];
    __shared__ uint32_t tmem_base_smem;
    __shared__ int abort_flag_smem;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    // this CTA's tiles: blockIdx.x + n * gridDim.x, n = 0, 1, ...; tile n belongs to loader / epilogue group n % 2, uses
    // accumulator n % NACC, "full" barrier n % NAF, "done" barrier n % NB (two halves: both epilogue groups, accumulator =
    // half, "done" barrier (2 n + half) % NB); its unit h is the CTA's unit number n * CW + h,
    // in ring position (n * CW + h) % NUNIT
    const int my_tiles = g.tiles + ((int)blockIdx.x < g.extra ? 1 : 0);
    const int cn = min(BN, p.C_out);

    const uint32_t wexp = (smem_u32(smem_raw) + 1023u) & ~1023u;          // [KT][BN rows][128 B] expanded weights
    const uint32_t cexp = wexp + KT * C::W_TILE_BYTES;                    // [BN rows][128 B] constant rows (first 32 bytes)
    const uint32_t pops = cexp + C::W_TILE_BYTES;                         // [BN] bit counts
    const uint32_t ring = pops + (BN * 4 + 127) / 128 * 128;              // [NLD][RD] halo tiles
    const uint32_t bar0 = smem_u32(bars);
    auto load_full = [&](int gr, int s) { return bar0 + 8u * (gr * RD + s); };
    auto load_empty = [&](int gr, int s) { return bar0 + 8u * (NLD * RD + gr * RD + s); };
    auto a_full = [&](int s) { return bar0 + 8u * (2 * NLD * RD + s); };
    auto tile_done = [&](int s) { return bar0 + 8u * (2 * NLD * RD + NAF + s); };
    auto acc_free = [&](int s) { return bar0 + 8u * (2 * NLD * RD + NAF + NB + s); };
    volatile int *abort_flag = &abort_flag_smem;

    if (tid < NBARS) {
        // a stage loaded: the loader's arrive (+ the copy's bytes); free again: the producer warps that read it; a tile's units full: the
        // producer warps that fill them; done: the issuer's commit; an accumulator free: the four epilogue warps of the tile's group
        constexpr int E0 = NLD * RD, F0 = 2 * NLD * RD, D0 = F0 + NAF, A0 = D0 + NB;
        mbar_init(bar0 + 8u * tid, tid < E0 || (tid >= D0 && tid < A0) ? 1 : (tid >= A0 ? 4 : 4 * CW));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) abort_flag_smem = 0;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    for (int c = tid; c < BN; c += C::THREADS) asm volatile("st.shared.b32 [%0], %1;" ::"r"(pops + 4u * c), "r"(0) : "memory");
    if (tid == 32 * C::FIRST_LOADER_WARP) asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&xmap)) : "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    // The loader warps start now: the first halo tiles arrive while the other warps expand the weights (0.5 us of a small layer's
    // 4).  The other warps meet at a named barrier of their own; everybody meets again at the end.
    const bool is_loader = warp >= C::FIRST_LOADER_WARP && warp < C::FIRST_PRODUCER_WARP;
    const uint32_t tmem_base = tmem_base_smem;
    if (!is_loader) {
        constexpr int NW = C::THREADS - 32 * NLD, WTOTAL = KT * 8 * BN, WU = (WTOTAL + NW - 1) / NW;
        const int wt = tid < 32 * C::FIRST_LOADER_WARP ? tid : tid - 32 * NLD;
        auto sync_workers = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(NW) : "memory"); };
        // ---- one-off: expanded weights and the channels' bit counts.  K position e of the MMAs = channel word e / 10, tap e % 10
        // (global weight word tap * CW + channel word) -> stage e / 8, 16-byte piece e % 8; MMA row `row` carries channel ch.
        // All of a thread's words, and its threshold, are requested before the first is used.
        const int my_ch = (wt & ~31) + channel_of_column(wt & 31);
        pdl_wait();
        const int thr = wt < BN && my_ch < cn ? __ldg(p.thr + my_ch) : 0;
        uint32_t w[WU];
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int idx = wt + u * NW, e = idx % (KT * 8), row = idx / (KT * 8), tap = e % UWORDS, cword = e / UWORDS;
            const int ch = (row & ~31) + channel_of_column(row & 31);
            w[u] = idx < WTOTAL && tap < TAPS && cword < CW && ch < cn ? __ldg(p.w + (long)ch * C::KW + tap * CW + cword) : 0u;
        }
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int idx = wt + u * NW, e = idx % (KT * 8), row = idx / (KT * 8), tap = e % UWORDS, cword = e / UWORDS;
            const int ch = (row & ~31) + channel_of_column(row & 31);
            if (idx >= WTOTAL) break;
            const bool live = tap < TAPS && cword < CW && ch < cn;
            expand_store_w4(w[u], live, wexp + (uint32_t)(e >> 3) * C::W_TILE_BYTES + (uint32_t)row * ROWB, row & 7, e & 7);
            if (live) asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(pops + 4u * row), "r"(__popc(w[u])) : "memory");
        }
        if (warp >= C::FIRST_PRODUCER_WARP && warp < C::FIRST_PRODUCER_WARP + 4) write_const_block(tmem_base + ((uint32_t)((warp & 3) * 32) << 16));
        tc_fence_before();
        sync_workers();
        tc_fence_after();
        if (wt < BN) {                  // constants K - 2 popc - thr (thr clamped to +-(K + 1))
            int pop;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(pop) : "r"(pops + 4u * wt) : "memory");
            store_const_row(p.K - 2 * pop - max(min(thr, p.K + 1), -p.K - 1), cexp + (uint32_t)wt * ROWB, wt & 7);
        }
        fence_async_proxy();
        tc_fence_before();
        sync_workers();
        tc_fence_after();
    }

    // A role's tiles are a fixed number of tiles apart: image and tile coordinates follow by carries (two divisions per tile
    // were a third of an epilogue warp's time).
    struct TileCursor {
        int b, ty, tx, db, dty, dtx;
    };
    auto cursor = [&](int n0, int log_step) {
        const uint32_t t = blockIdx.x + (uint32_t)n0 * gridDim.x;
        TileCursor c;
        c.b = (int)exact_div(t, g.img_mul, g.img_shift);
        const uint32_t rem = t - (uint32_t)c.b * (uint32_t)(g.tiles_x * g.tiles_y);
        c.ty = (int)exact_div(rem, g.row_mul, g.row_shift);
        c.tx = (int)rem - c.ty * g.tiles_x;
        c.db = g.step[log_step].db;
        c.dty = g.step[log_step].dty;
        c.dtx = g.step[log_step].dtx;
        return c;
    };
    auto advance = [&](TileCursor &c) {
        c.tx += c.dtx;
        if (c.tx >= g.tiles_x) { c.tx -= g.tiles_x; ++c.ty; }
        c.ty += c.dty;
        if (c.ty >= g.tiles_y) { c.ty -= g.tiles_y; ++c.b; }
        c.b += c.db;
    };

    if (warp < C::NISS) {
        // ------------------------------------------------------------------ MMA issuer of tiles n = warp (mod NISS), or of
        // half `warp` of every tile, in order
        constexpr uint32_t idesc = make_idesc_f4(AW);
        constexpr uint32_t HALF_DESC = (uint32_t)(AW * ROWB) >> 4;               // weight rows of the second half
        const uint64_t desc0 = make_desc(wexp);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32), b_lo = (uint32_t)desc0;
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t sf = tmem_u + (uint32_t)CB_COL, c_lo = (uint32_t)make_desc(cexp);
        const uint32_t hf = NH == 2 ? __shfl_sync(0xffffffffu, (uint32_t)warp, 0) : 0u;
        const uint32_t w_lo = b_lo + hf * HALF_DESC;
        auto issue = [&](int n) {
            const uint32_t d_t = tmem_u + (uint32_t)((NH == 2 ? (int)hf : n % NACC) * AW);
            tc_mma_const(d_t, tmem_u, c_lo + hf * HALF_DESC, desc_hi, idesc);
#pragma unroll
            for (int h = 0; h < CW; ++h) {
                const uint32_t a_t = tmem_u + (uint32_t)(C::A_COL0 + ((n * CW + h) % NUNIT) * U_COLS);
#pragma unroll
                for (int t = 0; t < UWORDS / 2; ++t) {
                    const int e = h * UWORDS + 2 * t;
                    tc_mma_f4_ts(d_t, a_t + 8u * t, w_lo + (uint32_t)((e >> 3) * (C::W_TILE_BYTES >> 4) + (e & 7)),
                                 desc_hi, idesc, sf, 1u);
                }
            }
            tc_commit(tile_done((n * NH + (int)hf) % NB));
        };
        constexpr int N_STEP = NH == 2 ? 1 : C::NISS;
        // completion of acc_free to wait for: the epilogue has read the accumulator's previous tile
        auto previous = [&](int n) { return NH == 2 ? n - 1 : n / NACC - 1; };
        // One lane runs the loop where a tile is six short instructions, the whole warp, electing a lane per tile, where it is more of them or both
        // halves wait for one accumulator each (us, one lane and the warp: 32 -> 32 at M = 3211264 34.6 and 36.0; 32 -> 96 at 1130040 30.7 and 28.3;
        // 32 -> 128 at 1505280 38.4 and 35.8; 64 -> 64 /2 at 493950 16.4 and 15.2)
        if constexpr (CW == 1 && NH == 1) {
            if (elect_one()) {
                for (int n = warp; n < my_tiles; n += N_STEP) {
                    if (!issuer_wait(a_full(n % NAF), (uint32_t)(n / NAF) & 1u, abort_flag, p.err, ERR_C3_ISSUER_TIMEOUT)) break;
                    const int prev = previous(n);
                    if (prev >= 0 && !issuer_wait(acc_free(n % NACC), (uint32_t)prev & 1u, abort_flag, p.err, ERR_C3_ACC_TIMEOUT)) break;
                    tc_fence_after();
                    issue(n);
                }
            }
            __syncwarp();
        } else {
            for (int n = NH == 2 ? 0 : warp; n < my_tiles; n += N_STEP) {
                if (!pw_wait(a_full(n % NAF), (uint32_t)(n / NAF) & 1u, abort_flag, p.err, ERR_C3_ISSUER_TIMEOUT)) break;
                const int prev = previous(n);
                if (prev >= 0 && !pw_wait(acc_free(NH == 2 ? (int)hf : n % NACC), (uint32_t)prev & 1u, abort_flag, p.err, ERR_C3_ACC_TIMEOUT)) break;
                tc_fence_after();
                if (elect_one()) issue(n);
                __syncwarp();
            }
        }
    } else if (warp < C::FIRST_PRODUCER_WARP) {
        // ------------------------------------------------------------------ loader of a group: one halo tile per TMA copy
        const int grp = warp - C::FIRST_LOADER_WARP;
        int stage = 0;
        uint32_t phase = 1;                       // first pass through the ring: the stages are free
        int issued = 0;
        TileCursor tc = cursor(grp, 1);
        pdl_wait();
        for (int n = grp; n < my_tiles; n += NLD, advance(tc)) {
            if (!pw_wait<256>(load_empty(grp, stage), phase, abort_flag, p.err, ERR_C3_LOADER_TIMEOUT)) break;
            if (lane == 0) {
                const uint32_t dst = ring + (uint32_t)(grp * RD + stage) * (uint32_t)g.stage_bytes;
                const int x = (tc.tx * TW * g.stride - p.pad - g.xoff) * CW;     // words; a multiple of 4 by construction
                const int y = tc.ty * TH * g.stride - p.pad;
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(load_full(grp, stage)), "r"((uint32_t)(g.hb * g.wbw * 4)) : "memory");
                asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                             ::"r"(dst), "l"(reinterpret_cast<uint64_t>(&xmap)), "r"(x), "r"(y), "r"(tc.b), "r"(load_full(grp, stage)) : "memory");
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
    } else if (warp >= C::FIRST_EPILOGUE_WARP) {
        // ------------------------------------------------------------------ epilogue group (warp - first) / 4
        const int quad = warp & 3;
        const int grp = (warp - C::FIRST_EPILOGUE_WARP) >> 2;
        const int r = quad * 32 + lane;                           // row of the tile = output pixel (r / TW, r % TW)
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const int owords = p.C_out >> 5;
        // NH == 1: the group takes alternate tiles; NH == 2: the group takes its half (64 channels) of every tile
        TileCursor tc = cursor(NH == 2 ? 0 : grp, NH == 2 ? 0 : 1);
        for (int n = NH == 2 ? 0 : grp; n < my_tiles; n += NH == 2 ? 1 : NGRP, advance(tc)) {
            const int acc = NH == 2 ? grp : n % NACC;
            const int d = NH == 2 ? 2 * n + grp : n;                              // the tile's (half's) "done" number
            const int ch0 = NH == 2 ? 2 * grp : 0;                                // first output word of this accumulator
            if (!pw_wait<NH == 2 ? 64 : 128>(tile_done(d % NB), (uint32_t)(d / NB) & 1u, abort_flag, p.err, ERR_C3_EPILOGUE_TIMEOUT)) break;
            tc_fence_after();
            uint32_t words[AW / 32];
            if constexpr (AW == 32) {
                uint32_t v[16];
                tc_ld32_pack16(t_lane + (uint32_t)(acc * AW), v);
                tc_wait_ld();
                pin_regs(v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_free(acc));
                words[0] = sign_word(v);
            } else {
                uint32_t v[32];
                tc_ld64_pack16(t_lane + (uint32_t)(acc * AW), v);
                tc_wait_ld();
                pin_regs(v);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acc_free(acc));
                words[0] = sign_word(v);
                words[1] = sign_word(v + 16);
            }
            const int oh = tc.ty * TH + (r >> 4), ow = tc.tx * TW + (r & 15);
            if (oh < p.OH && ow < p.OW) {
                uint32_t *dst = static_cast<uint32_t *>(p.out) + (long)(((unsigned)tc.b * p.OH + oh) * p.OW + ow) * owords + ch0;
                if (AW == 64 && (owords & 1) == 0) {                  // (an even word count keeps the pair 8-byte aligned)
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(words[0], words[1 % (AW / 32)]);
                } else {
#pragma unroll
                    for (int ch = 0; ch < AW / 32; ++ch)
                        if (ch0 + ch < owords) dst[ch] = words[ch];
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ producer group (warp - first) / 4
        // thread = output pixel (ty, tx) of the tile = tensor-memory lane; its nine input pixels sit at rows
        // ty * s + kr, pixels tx * s + XOFF + kt of the halo tile.  The group fills unit h (channel word h of the nine
        // taps) of the tiles n0, n0 + step, ...
        const int quad = warp & 3;
        const int grp = (warp - C::FIRST_PRODUCER_WARP) >> 2;
        const int h = CW == 2 ? (grp & 1) : 0;
        const int n0 = CW == 2 ? (grp >> 1) : grp, step = CW == 2 ? NPG / 2 : NPG;
        const int r = quad * 32 + lane;
        const uint32_t my_off = (uint32_t)((((r >> 4) * g.stride) * g.wbw + ((r & 15) * g.stride + g.xoff) * CW + h) * 4);
        const uint32_t row_pitch = (uint32_t)(g.wbw * 4);
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::A_COL0;
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        for (int n = n0; n < my_tiles; n += step) {
            const int lg = n & 1, stage = (n >> 1) % RD;
            uint32_t wds[TAPS];
            if (!pw_wait<64>(load_full(lg, stage), (uint32_t)((n >> 1) / RD) & 1u, abort_flag, p.err, ERR_C3_PRODUCER_TIMEOUT)) break;
            const uint32_t src = ring + (uint32_t)(lg * RD + stage) * (uint32_t)g.stage_bytes + my_off;
#pragma unroll
            for (int tap = 0; tap < TAPS; ++tap)
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(wds[tap]) : "r"(src + (uint32_t)(tap / 3) * row_pitch + (uint32_t)((tap % 3) * CW * 4)) : "memory");
            // expanded before the wait for the unit (the unit's tenth word is not written: its weights are zero)
            uint32_t v[32], v4[4];
#pragma unroll
            for (int e = 0; e < 8; ++e) expand_a4(wds[e], &v[4 * e]);
            expand_a4(wds[8], v4);
            // the MMAs of the tile that used this ring position last have read it (nothing to wait for the first time round)
            const int u = n * CW + h;
            if (u >= NUNIT) {
                const int dm = (u - NUNIT) / CW * NH;                             // that tile's first "done" number
                if (!pw_wait<64>(tile_done(dm % NB), (uint32_t)(dm / NB) & 1u, abort_flag, p.err, ERR_C3_UNIT_TIMEOUT)) break;
                if (NH == 2 && !pw_wait<64>(tile_done((dm + 1) % NB), (uint32_t)((dm + 1) / NB) & 1u, abort_flag, p.err, ERR_C3_UNIT_TIMEOUT)) break;
            }
            tc_fence_after();
            const uint32_t taddr = t_lane + (uint32_t)((u % NUNIT) * U_COLS);
            tc_st32_nowait(taddr, v);
            tc_st4_nowait(taddr + 32u, v4);
            // the stage may be refilled: its words have left through registers (right behind the loads a refill could overtake them)
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

template <int CW, int BN>
int launch_c3(const ConvProblem &p0, cudaStream_t stream)
{
    using C = C3Cfg<CW, BN>;
    ConvProblem p = p0;
    p.err = device_error_word();
    C3Geom g = c3_geometry(p);
    const int smem = c3_smem_bytes<CW, BN>(g);
    if (smem > 227 * 1024 - 1024) return BCNN_ERR_UNSUPPORTED;
    const int sms = sm_count();
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return BCNN_ERR_CUDA;
    // the packed input as [B][H][W * CW] 32-bit words; box = wbw words x hb rows of one image; zero fill outside
    CUtensorMap xmap;
    const cuuint64_t dims[3] = {(cuuint64_t)p.W * CW, (cuuint64_t)p.H, (cuuint64_t)p.B};
    const cuuint64_t strides[2] = {(cuuint64_t)p.W * CW * 4, (cuuint64_t)p.H * p.W * CW * 4};
    const cuuint32_t box[3] = {(cuuint32_t)g.wbw, (cuuint32_t)g.hb, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    if (encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_UINT32, 3, const_cast<uint32_t *>(p.x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return BCNN_ERR_CUDA;
    const unsigned grid = (unsigned)(g.total_tiles < sms ? g.total_tiles : sms);
    c3_walk(g, grid);
    void (*k)(const ConvProblem, const C3Geom, const CUtensorMap) = conv_tc_c3_kernel<CW, BN>;
    const int ask = smem < 120 * 1024 ? 120 * 1024 : smem;          // one CTA per SM (it takes all of tensor memory)
    if (!allow_smem((const void *)k, 227 * 1024 - 1024)) return BCNN_ERR_CUDA;
    return launch(k, grid, C::THREADS, ask, stream, p, g, xmap);
}

}  // namespace

bool conv_tc_c3_supports(const ConvProblem &p)
{
    if (p.mode != 1) return false;                               // packed output only
    if (p.kh != 3 || p.kw != 3 || p.stride < 1 || p.stride > 2 || p.pad > 1) return false;
    if (p.cw != 1 && p.cw != 2) return false;
    if (p.C_out % 32 != 0 || p.C_out > 128) return false;
    if ((p.W * p.cw) % 4 != 0) return false;                     // image rows must be 16-byte multiples (TMA strides)
    if ((reinterpret_cast<uintptr_t>(p.x) & 15u) != 0) return false;   // TMA base address
    const long tiles = (long)p.B * ((p.OH + TH - 1) / TH) * ((p.OW + TW - 1) / TW);
    return tiles < (1L << 30);                                   // tile numbers are 32-bit on the device
}

int launch_conv_tc_c3(const ConvProblem &p, cudaStream_t stream)
{
    if (!conv_tc_c3_supports(p)) return BCNN_ERR_UNSUPPORTED;
    if (p.cw == 1) {
        if (p.C_out <= 32) return launch_c3<1, 32>(p, stream);
        if (p.C_out <= 64) return launch_c3<1, 64>(p, stream);
        return launch_c3<1, 128>(p, stream);
    }
    if (p.C_out <= 32) return launch_c3<2, 32>(p, stream);
    if (p.C_out <= 64) return launch_c3<2, 64>(p, stream);
    return launch_c3<2, 128>(p, stream);
}

}  // namespace bcnn
