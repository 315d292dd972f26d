// Streaming tcgen05 engine on weights that are expanded as they arrive: the module epilogue of layers that neither the module engine
// (pointwise) nor the weight-stationary engine takes; the packed and int32 outputs of such weights run on conv_tc_pre.cu.
// Arithmetic: 4-bit operands (tc_common.cuh), fp32 accumulators that hold exact integers,
// sum a*g = accumulator + K - 2 popc(G):  one constant per output channel, nothing per row.
//
// Persistent, warp-specialised; each CTA walks a static list of 128 x BN tiles.
//   warp 0          issuer: tcgen05.mma / commit only, waits on named barriers only (a memory
//                   instruction after tensor-core instructions would stall it)
//   warps 1-4       epilogue: tcgen05.ld, the module's steps, hand the accumulator back
//   G = 2 producer groups, each 4 activation warps + 4 weight warps, one thread per tile
//                   row; the groups take the ring's stages alternately so that one group gathers
//                   while the other expands.  Packed words are staged with cp.async (16 bytes per
//                   row half and stage, zero-fill out of range).
//                     activation rows -> TENSOR memory (tcgen05.st, 32 columns per stage): the
//                       MMA takes A from tensor memory, so shared memory carries only weights
//                     weight rows     -> shared memory, 128-byte-swizzled K-major tiles
//   last warp       control: does the issuer's mbarrier waits and releases it stage by stage
// A ring stage is 256 bits of K.  Tensor memory (512 columns): two accumulators of BN = 128 columns, 7 ring stages and the unit
// scales.  Column popcounts are taken from the words as they are
// expanded; each group leaves its partial constants for a tile in shared-memory slots.
// Every mbarrier wait is bounded and reports through the device error word.
#include "tc_common.cuh"

namespace bcnn {

namespace {

using namespace tc;

constexpr int EPI_WARPS = 4;
constexpr int G = 2;                      // producer groups
constexpr int PF = 3;                     // packed-word stages in flight per producer thread
constexpr int MAX_SMEM = 227 * 1024 - 512; // dynamic shared memory available beside the static part

constexpr int ERR_PRODUCER_TIMEOUT = 101;
constexpr int ERR_MMA_TIMEOUT = 102;
constexpr int ERR_EPILOGUE_TIMEOUT = 103;

constexpr int BN = 128;                   // output channels of a tile
struct Cfg {
    static constexpr int NBUF = 2;                                        // accumulator buffers
    static constexpr int A_COL0 = NBUF * BN;                              // first column of the activation ring
    static constexpr int STAGES = 7;
    static constexpr int GROUP_WARPS = 4 + BN / 32;
    static constexpr int GROUP_THREADS = 32 * GROUP_WARPS;
    static constexpr int PROD_THREADS = G * GROUP_THREADS;
    static constexpr int FIRST_PRODUCER_WARP = 1 + EPI_WARPS;
    static constexpr int CONTROL_WARP = FIRST_PRODUCER_WARP + G * GROUP_WARPS;
    static constexpr int THREADS = 32 * (CONTROL_WARP + 1);
    static constexpr int W_BYTES = BN * ROWB;                             // one ring stage of weights
    static constexpr int SF_COL = 512 - (int)SF_COLS;                     // unit scales
    static constexpr int BITS_BYTES = PF * PROD_THREADS * 32;
    static constexpr int SLOTS = STAGES + NBUF + 2;                       // per-tile constant slots
    static constexpr int SLOT_INTS = G * BN;
    static constexpr int CONST_BYTES = SLOTS * SLOT_INTS * 4;
    static constexpr int TABLE_BYTES = EPI_WARPS * BN * 4;                // column constants as fp32, one table per epilogue warp
    static_assert(A_COL0 + STAGES * 32 <= SF_COL, "tensor memory budget");
    static_assert(STAGES >= G, "a producer group must not lap the ring (parity waits)");
};

int smem_bytes(int ktab_words)
{
    using C = Cfg;
    return 1024 + C::STAGES * C::W_BYTES + C::BITS_BYTES + C::CONST_BYTES + C::TABLE_BYTES + ktab_words * 4 + ID_RING_BYTES + 16;
}

__global__ void __launch_bounds__(Cfg::THREADS, 1)
conv_tc_i8_kernel(const ConvProblem p, const int ktab_words)
{
    using C = Cfg;
    constexpr int NBUF = C::NBUF;
    constexpr int STAGES = C::STAGES;
    constexpr int SLOTS = C::SLOTS;

    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * 8 + 2 * 2];
    __shared__ uint32_t tmem_base_smem;
    __shared__ int abort_flag_smem;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int ktiles = (p.kwords + 7) >> 3;
    const int m_tiles = (p.M - 1) / BM + 1;                  // M >= 1; no overflow for M close to 2^31
    const int n_tiles = (p.C_out + BN - 1) / BN;
    const int total_tiles = m_tiles * n_tiles;
    const int my_tiles = ((int)blockIdx.x < total_tiles) ? (total_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int total_items = my_tiles * ktiles;

    const uint32_t wring = (smem_u32(smem_raw) + 1023u) & ~1023u;         // [STAGES][BN rows][128 B]
    const uint32_t bits_ring = wring + STAGES * C::W_BYTES;               // [PF][2][PROD_THREADS][16 B]
    const uint32_t consts = bits_ring + C::BITS_BYTES;                    // [SLOTS][G][BN] int32
    const uint32_t tables = consts + C::CONST_BYTES;                      // [EPI_WARPS][BN] fp32
    const uint32_t ktab_addr = tables + C::TABLE_BYTES;                   // unit table of the gather
    const uint32_t idring = (ktab_addr + (uint32_t)ktab_words * 4u + 15u) & ~15u;   // [ID_SLOTS][BM rows][80 B]
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (8 + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (16 + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (18 + b); };
    volatile int *abort_flag = &abort_flag_smem;

    if (tid == 0) {
        for (int s = 0; s < 8; ++s) {
            mbar_init(full_bar(s), C::GROUP_WARPS);      // every warp of the group that owns the stage
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), EPI_WARPS);
        }
        abort_flag_smem = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    const int gwidth = gather_width(p.cw);
    build_unit_table8(p, ktab_addr, ktiles * (8 / gwidth), gwidth, tid, C::THREADS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    pdl_wait();
    const uint32_t tmem_base = tmem_base_smem;

    if (warp == 0) {
        // ------------------------------------------------------------------ issuer (no memory instructions)
        constexpr uint32_t idesc = make_idesc_f4(BN);
        const uint64_t desc0 = make_desc(0);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
        const uint32_t b_lo0 = (uint32_t)desc0 | ((wring & 0x3FFFFu) >> 4);      // + slot * (W_BYTES / 16)
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);             // warp-uniform copy for the issuer
        const uint32_t a_tmem0 = tmem_u + (uint32_t)C::A_COL0;                   // + slot * 32 columns
        const uint32_t sf = tmem_u + (uint32_t)C::SF_COL;
        int s = 0, buf = 0;
        for (int ti = 0; ti < my_tiles; ++ti) {
            const uint32_t d_tmem = tmem_u + (uint32_t)(buf * BN);
            const uint32_t tfull = tfull_bar(buf);
            for (int kt = 0; kt < ktiles; ++kt) {
                const uint32_t a_t = a_tmem0 + (uint32_t)s * 32u;
                const uint32_t b_lo = b_lo0 + (uint32_t)s * (C::W_BYTES >> 4);
                const int nk = p.kwords - 8 * kt;                 // two K words per instruction; skip the zero tail
                const uint32_t ebar = empty_bar(s);
                asm volatile("bar.sync %0, 64;" ::"r"(1 + s) : "memory");
                tc_fence_after();
                // per instruction: 8 tensor-memory columns of A, +2 (16-byte units) in the B descriptor
                if (elect_one()) {
                    tc_mma_f4_ts(d_tmem, a_t, b_lo, desc_hi, idesc, sf, kt > 0 ? 1u : 0u);
                    if (nk > 2) tc_mma_f4_ts(d_tmem, a_t + 8u, b_lo + 2u, desc_hi, idesc, sf, 1u);
                    if (nk > 4) tc_mma_f4_ts(d_tmem, a_t + 16u, b_lo + 4u, desc_hi, idesc, sf, 1u);
                    if (nk > 6) tc_mma_f4_ts(d_tmem, a_t + 24u, b_lo + 6u, desc_hi, idesc, sf, 1u);
                    tc_commit(ebar);
                    if (kt == ktiles - 1) tc_commit(tfull);
                }
                __syncwarp();
                if (++s == STAGES) s = 0;
            }
            if (++buf == NBUF) buf = 0;
        }
    } else if (warp == C::CONTROL_WARP) {
        // ------------------------------------------------------------------ control: waits for the issuer
        // A stage is released (bar.arrive on 1 + slot) once its ring slot is full and, for a tile's
        // first stage, once the accumulator buffer is free.  The slot being full implies that the
        // issuer is past the previous use of the same named barrier.  After a time-out the remaining
        // stages are released without waiting so that the issuer always terminates.
        int s = 0, buf = 0;
        uint32_t ring_phase = 0, buf_phase = 1;      // first use of every accumulator buffer: free
        bool alive = true;
        for (int ti = 0; ti < my_tiles; ++ti) {
            if (lane == 0 && alive) alive = mbar_wait(tempty_bar(buf), buf_phase, abort_flag, p.err, ERR_MMA_TIMEOUT);
            for (int kt = 0; kt < ktiles; ++kt) {
                if (lane == 0 && alive) alive = mbar_wait(full_bar(s), ring_phase, abort_flag, p.err, ERR_MMA_TIMEOUT);
                // after a time-out: bar.sync, which pairs every release with one wait of the issuer (two bar.arrive in a
                // row on one barrier would complete it without the issuer)
                if (__shfl_sync(0xffffffffu, alive ? 1 : 0, 0)) asm volatile("bar.arrive %0, 64;" ::"r"(1 + s) : "memory");
                else asm volatile("bar.sync %0, 64;" ::"r"(1 + s) : "memory");
                if (++s == STAGES) { s = 0; ring_phase ^= 1u; }
            }
            if (++buf == NBUF) { buf = 0; buf_phase ^= 1u; }
        }
    } else if (warp <= EPI_WARPS) {
        // ------------------------------------------------------------------ epilogue
        const int quad = warp & 3;                 // tensor-memory lane quadrant this warp may read
        const int erow = quad * 32 + lane;
        bool alive = true;
        int buf = 0;
        uint32_t buf_phase = 0;
        // the identity values of this thread's row are staged ID_AHEAD live chunks ahead (a chunk is
        // live when its first channel exists), in ring slot (live chunk number) % ID_SLOTS
        const uint32_t id_warp = idring + (uint32_t)(quad * 32) * ID_ROW_BYTES;   // slot 0, the warp's first row
        int pf_ti = 0, pf_ch = 0, pf_slot = 0, cur_slot = 0;
        auto prefetch_next = [&]() {
            bool queued = false;
            while (pf_ti < my_tiles && !queued) {
                const int t = (int)blockIdx.x + pf_ti * (int)gridDim.x;
                const int nt = t / m_tiles, mt = t - nt * m_tiles;
                const int n = nt * BN + pf_ch * 32;
                if (n < p.C_out) {
                    module_prefetch(p, id_warp + (uint32_t)pf_slot * (BM * ID_ROW_BYTES), (long)mt * BM + quad * 32, n, lane);
                    queued = true;
                }
                if (++pf_ch == BN / 32) { pf_ch = 0; ++pf_ti; }
            }
            if (!queued) cp_async_commit();
            if (++pf_slot == ID_SLOTS) pf_slot = 0;
        };
        for (int a = 0; a < ID_AHEAD; ++a) prefetch_next();
        for (int ti = 0; ti < my_tiles; ++ti) {
            const int tile = (int)blockIdx.x + ti * (int)gridDim.x;
            const int n_tile = tile / m_tiles, m_tile = tile - n_tile * m_tiles;
            const int m0 = m_tile * BM, n0 = n_tile * BN;
            const int em = m0 + erow;
            // which producer groups took part in this tile (each leaves partial constants): both,
            // unless the tile is a single stage
            const int first_group = (ti * ktiles) & 1;
            const bool two = ktiles >= 2;
            const uint32_t slot = consts + (uint32_t)((ti % SLOTS) * C::SLOT_INTS * 4);
            const uint32_t part0 = slot + (uint32_t)(first_group * BN * 4);
            const uint32_t part1 = slot + (uint32_t)((first_group ^ 1) * BN * 4);
            if (alive) alive = mbar_wait(tfull_bar(buf), buf_phase, abort_flag, p.err, ERR_EPILOGUE_TIMEOUT);
            alive = __all_sync(0xffffffffu, alive && !*abort_flag);
            if (!alive) break;
            tc_fence_after();
            // the groups' partial constants -> this warp's table of fp32 addends
            const uint32_t table = tables + (uint32_t)(quad * BN * 4);
            for (int c = lane; c < BN; c += 32) {
                int v0, v1 = 0;
                asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v0) : "r"(part0 + 4u * c) : "memory");
                if (two) asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v1) : "r"(part1 + 4u * c) : "memory");
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(table + 4u * c), "r"(table_entry<2>(v0 + v1)) : "memory");
            }
            __syncwarp();
            const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * BN);
            uint32_t words[BN / 32];
#pragma unroll
            for (int ch = 0; ch < BN / 32; ++ch) {
                const int col0 = ch * 32;
                words[ch] = 0;
                if (n0 + col0 < p.C_out) {             // warp-uniform
                    uint32_t v[32];
                    tc_ld32(t_addr + (uint32_t)col0, v);
                    float dot[32];
#pragma unroll
                    for (int i4 = 0; i4 < 8; ++i4) {
                        const uint4 cc = ld_shared_v4(table + 4u * (col0 + 4 * i4));
                        dot[4 * i4 + 0] = __uint_as_float(fadd_bits(v[4 * i4 + 0], cc.x));
                        dot[4 * i4 + 1] = __uint_as_float(fadd_bits(v[4 * i4 + 1], cc.y));
                        dot[4 * i4 + 2] = __uint_as_float(fadd_bits(v[4 * i4 + 2], cc.z));
                        dot[4 * i4 + 3] = __uint_as_float(fadd_bits(v[4 * i4 + 3], cc.w));
                    }
                    prefetch_next();
                    cp_async_wait<ID_AHEAD>();                        // this chunk's copy has landed
                    words[ch] = module_chunk(p, dot, id_warp + (uint32_t)cur_slot * (BM * ID_ROW_BYTES), (long)em - lane, n0 + col0, lane);
                    if (++cur_slot == ID_SLOTS) cur_slot = 0;
                }
            }
            // all reads of this accumulator buffer are complete: hand it back
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty_bar(buf));
            if (++buf == NBUF) { buf = 0; buf_phase ^= 1u; }
            if (p.out != nullptr && em < p.M) {
                const int owords = p.C_out >> 5;
                uint32_t *dst = static_cast<uint32_t *>(p.out) + (long)em * owords + (n0 >> 5);
                if ((owords & 3) == 0 && n0 + BN <= p.C_out) {
                    *reinterpret_cast<uint4 *>(dst) = make_uint4(words[0], words[1], words[2], words[3]);
                } else {
#pragma unroll
                    for (int ch = 0; ch < BN / 32; ++ch)
                        if (n0 + ch * 32 < p.C_out) dst[ch] = words[ch];
                }
            }
        }
        cp_async_wait<0>();
    } else {
        // ------------------------------------------------------------------ producers
        const int pw = warp - C::FIRST_PRODUCER_WARP;            // producer warp index
        const int grp = pw / C::GROUP_WARPS, wi = pw - grp * C::GROUP_WARPS;
        const bool is_a = wi < 4;
        // activation warps are matched to tensor-memory lane quadrants (a warp may only touch
        // lanes 32 * (warp % 4) ...): the first four warps of a group have four distinct residues
        const int quad = warp & 3;
        const int row = is_a ? quad * 32 + lane : (wi - 4) * 32 + lane;   // row of the A or of the W tile
        const int ptid = tid - 32 * C::FIRST_PRODUCER_WARP;
        constexpr uint32_t HALF_BYTES = C::PROD_THREADS * 16u, SLOT_BYTES = 2u * HALF_BYTES;
        const uint32_t bits0 = bits_ring + (uint32_t)ptid * 16u, bits_end = bits0 + PF * SLOT_BYTES;
        const uint32_t st_addr0 = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::A_COL0;
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        const bool w16 = (p.kwords & 3) == 0;
        const TileStep step = make_tile_step(p, (uint32_t)BM * gridDim.x);

        // this thread's items: grp, grp + G, ... of the CTA's flattened (tile, stage) list
        // ---- load cursor: tile (n_tile, m_tile) and, per role, the activation row or the weight row
        int l_kt = grp;
        int l_left = total_items > grp ? (total_items - grp + G - 1) / G : 0;
        int l_n = (int)blockIdx.x / m_tiles, l_m = (int)blockIdx.x - l_n * m_tiles;
        RowCursor rc;
        rc.m = (uint32_t)l_m * BM + (uint32_t)row;
        rc.base = 0;
        rc.mask = 0;
        const uint32_t *wrow = p.w;
        bool wok = false;
        if (is_a) row_locate(p, rc);
        auto next_tile = [&]() {             // the CTA's next tile: gridDim.x further along (n_tile, m_tile)
            l_m += (int)gridDim.x;
            if (l_m < m_tiles) {
                if (is_a) row_step(p, step, rc);
            } else {
                do { l_m -= m_tiles; ++l_n; } while (l_m >= m_tiles);
                if (is_a) {
                    rc.m = (uint32_t)l_m * BM + (uint32_t)row;
                    row_locate(p, rc);
                }
            }
        };
        auto tile_ready = [&]() {            // per-tile values of the row after the cursor moved
            if (is_a) {
                row_window(p, step, rc);
            } else {
                const int n = l_n * BN + row;
                wok = n < p.C_out;
                wrow = p.w + (long)(wok ? n : 0) * p.kwords;
            }
        };
        while (l_kt >= ktiles) { l_kt -= ktiles; next_tile(); }
        tile_ready();
        uint32_t l_dst = bits0;
        auto issue_load = [&]() {
            if (is_a) {
                if (gwidth == 4) gather_stage8<4>(p.x, rc, ktab_addr + (uint32_t)l_kt * 8u, l_dst, HALF_BYTES);
                else if (gwidth == 2) gather_stage8<2>(p.x, rc, ktab_addr + (uint32_t)l_kt * 16u, l_dst, HALF_BYTES);
                else gather_stage8<1>(p.x, rc, ktab_addr + (uint32_t)l_kt * 32u, l_dst, HALF_BYTES);
            } else if (w16) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int kword = l_kt * 8 + 4 * h;
                    const bool ok = wok && kword < p.kwords;
                    cp_async_zfill<16>(l_dst + h * HALF_BYTES, ok ? wrow + kword : p.w, ok ? 16u : 0u);
                }
            } else {
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int kword = l_kt * 8 + e;
                    const bool ok = wok && kword < p.kwords;
                    cp_async_zfill<4>(l_dst + (e >> 2) * HALF_BYTES + 4u * (e & 3), ok ? wrow + kword : p.w, ok ? 4u : 0u);
                }
            }
            l_dst += SLOT_BYTES;
            if (l_dst == bits_end) l_dst = bits0;
            --l_left;
            l_kt += G;
            if (l_kt >= ktiles) {
                do { l_kt -= ktiles; next_tile(); } while (l_kt >= ktiles);
                tile_ready();
            }
        };

#pragma unroll 1
        for (int i = 0; i < PF - 1; ++i) {
            if (l_left > 0) issue_load();
            cp_async_commit();
        }

        // the scales are in place before this group's first arrival, which every MMA waits for
        if (grp == 0 && is_a) write_unit_scales(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::SF_COL);
        // ---- expand cursor
        uint32_t c_src = bits0;
        int c_ti = 0, c_kt = grp, pop = 0;
        int s = grp;                          // ring slot (G <= STAGES) and its parity
        uint32_t phase = 1;                   // first pass through the ring: slots are free
#pragma unroll 1
        for (int it = grp; it < total_items; it += G) {
            if (l_left > 0) issue_load();
            cp_async_commit();
            cp_async_wait<PF - 1>();
            const uint4 q0 = ld_shared_v4(c_src), q1 = ld_shared_v4(c_src + HALF_BYTES);
            c_src += SLOT_BYTES;
            if (c_src == bits_end) c_src = bits0;
            while (c_kt >= ktiles) { c_kt -= ktiles; ++c_ti; }
            if (is_a) {
                uint32_t v[32];               // column 4e + j = word j of K word e
                expand_stage8(q0, q1, v);
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) break;
                tc_fence_after();     // the MMAs that read this slot are complete (their commit released it)
                tc_st32(st_addr0 + (uint32_t)s * 32u, v);
                tc_fence_before();
            } else {
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) break;
                const uint32_t row_addr = wring + (uint32_t)s * C::W_BYTES + (uint32_t)row * ROWB;
                const int xr = row & 7;
                // rows and K words beyond the problem have no set bit here, and the codes of their -1 weights meet either
                // activations of clear bits or accumulator columns that nobody reads
                const uint32_t wds[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    expand_store_w4(wds[e], true, row_addr, xr, e);
                    pop += __popc(wds[e]);
                }
                if (c_kt + G >= ktiles) {
                    // this group's last stage of the tile: leave its partial constants for the epilogue.
                    //   K - 2 pg; the term that does not depend on the popcounts goes with the group of the tile's first stage
                    const int cst = -2 * pop + (((c_ti * ktiles) & 1) == grp ? p.K : 0);
                    const uint32_t part = consts + (uint32_t)(((c_ti % SLOTS) * C::SLOT_INTS + grp * BN + row) * 4);
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(part), "r"(cst) : "memory");
                    pop = 0;
                }
                fence_async_proxy();  // generic-proxy stores -> visible to the MMA (async proxy)
            }
            __syncwarp();
            mbar_arrive_pred(full_bar(s), lane0);
            s += G;
            if (s >= STAGES) { s -= STAGES; phase ^= 1u; }
            c_kt += G;
        }
        cp_async_wait<0>();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
    }
}

int ktab_words_for(const ConvProblem &p) { return (((p.kwords + 7) >> 3) * (8 / gather_width(p.cw)) + 3) & ~3; }

int launch_module(const ConvProblem &p0, cudaStream_t stream)
{
    ConvProblem p = p0;
    p.err = device_error_word();
    const int sms = sm_count();
    const long m_tiles = ((long)p.M + BM - 1) / BM;
    const long n_tiles = ((long)p.C_out + BN - 1) / BN;
    const long total = m_tiles * n_tiles;
    if (total >= (1L << 31)) return BCNN_ERR_UNSUPPORTED;
    const unsigned grid = (unsigned)(total < sms ? total : sms);
    const int ktw = ktab_words_for(p);
    const int smem = smem_bytes(ktw);
    if (smem > MAX_SMEM) return BCNN_ERR_UNSUPPORTED;
    if (!allow_smem((const void *)conv_tc_i8_kernel, MAX_SMEM)) return BCNN_ERR_CUDA;
    return launch(conv_tc_i8_kernel, grid, Cfg::THREADS, smem, stream, p, ktw);
}

}  // namespace

bool conv_tc_i8_supports(const ConvProblem &p)
{
    if (p.mode != 0 && (p.C_out % 32 != 0)) return false;
    if (p.kh * p.kw > 31) return false;                       // one validity bit per tap
    if ((long)p.B * p.H * p.W * p.cw >= (1L << 31)) return false;     // rows address the input by 32-bit word offsets
    if (ktab_words_for(p) > MAX_RAW_KTAB) return false;           // the K-word table of the gather must fit
    if ((long)p.kh * p.W * p.cw >= (1L << 27)) return false;  // a unit's word offset within the window
    return p.K <= (1 << 20);                                  // sums up to 4 K + 2 stay exact in fp32
}

int launch_conv_tc_i8(const ConvProblem &p, cudaStream_t stream)
{
    if (!conv_tc_i8_supports(p)) return BCNN_ERR_UNSUPPORTED;
    return p.mode == 2 ? launch_module(p, stream) : launch_conv_tc_raw(p, stream);
}

}  // namespace bcnn
