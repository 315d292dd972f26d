// Weight-stationary variant of the tcgen05 engine for layers with a short K: the expanded weights of up to
// 128 output channels fit in shared memory.  Wider layers run as slices of 128 (or 64) output channels: a CTA
// keeps one slice's weights, so the activations are expanded once per slice.
//
// Arithmetic.  4-bit operands (tc_common.cuh): every product with a set activation bit is +-2, accumulators are fp32 in
// tensor memory and hold exact integers, and with S = sum over set activation bits of the weight signs (acc = 2 S):
//   sum a*g = acc + K - 2 popc(G)          (a, g in {-1,+1})
// so the epilogue needs one constant per output channel, from a table in shared memory, and nothing per row.
// Differences to conv_tc_i8.cu, all aimed at short tiles (a 128 x 32 x 64 tile is one MMA instruction):
//   * the CTA expands its weight tile ONCE into shared memory and keeps it for all its
//     output tiles; only activations stream through the ring;
//   * the activation ring lives in TENSOR memory, not shared memory: producers write expanded rows
//     with tcgen05.st and the MMA takes its A operand from tensor memory.  A narrow MMA is bound by
//     operand fetch from shared memory (128 x 32 bytes of A per instruction whatever N is); with A in
//     tensor memory only the small weight slice is fetched;
//   * G producer groups of 128 threads take the ring's stages round-robin, so that G stages
//     are being gathered / expanded at any time (one thread's stage latency is several
//     hundred cycles, an MMA stage as little as 64);
//   * up to four accumulator buffers, so the epilogue of one tile overlaps the MMAs of the next ones;
//   * the warp that issues the MMAs waits only on named barriers; a separate control warp does the
//     mbarrier waits for it (a memory instruction after tensor-core instructions stalls the issuer);
//   * the implicit-im2col gather uses a per-K-word table (tap, word offset) and a per-row
//     tap-validity mask instead of divisions; out-of-image taps are zero-filled by cp.async.
// Every mbarrier wait is bounded and reports through the device error word.
#include "tc_common.cuh"

namespace bcnn {

namespace {

using namespace tc;

constexpr int EPI_WARPS = 4;              // warps of one epilogue team (one per tensor-memory lane quadrant)
constexpr int PF = 3;                     // packed-word stages in flight per producer thread
constexpr int MAX_SMEM = 227 * 1024;

constexpr int ERR_PRODUCER_TIMEOUT = 111;
constexpr int ERR_MMA_TIMEOUT = 112;
constexpr int ERR_EPILOGUE_TIMEOUT = 113;

// DUAL: two CTAs share an SM (two independent MMA issuers), each with half of tensor memory.
// TEAMS: epilogue teams of four warps; team t takes the tiles t, t + TEAMS, ... of the CTA (their accumulator
// buffers are then a fixed subset, so NBUF is a multiple of TEAMS).  Two teams serve the module epilogue, which is
// bound by the epilogue warps, and the 128-wide slices with one CTA per SM.
template <int BN, int G, bool DUAL, int TEAMS = 1> struct Cfg {
    static constexpr int FIRST_PRODUCER_THREAD = 32 * (1 + EPI_WARPS * TEAMS);
    static constexpr int PROD_THREADS = G * BM;
    // Tensor memory (512 columns): NBUF accumulator buffers of BN columns, then the activation ring,
    // one stage = 128 rows x 256 bits of K expanded to 128 bytes = 32 columns.
    static constexpr int TMEM_COLS = DUAL ? 256 : 512;
    static constexpr int NBUF = DUAL ? (BN == 128 ? 1 : 2) : (BN == 32 ? 4 : (BN == 64 ? 3 : 2));
    static constexpr int CONTROL_WARP = (FIRST_PRODUCER_THREAD + PROD_THREADS) / 32;
    static constexpr int THREADS = FIRST_PRODUCER_THREAD + PROD_THREADS + 32;
    static constexpr int A_COL0 = NBUF * BN;
    static constexpr int SF_COL = TMEM_COLS - (int)SF_COLS;      // unit scales
    static constexpr int STAGES = (SF_COL - A_COL0) / 32 > 8 ? 8 : (SF_COL - A_COL0) / 32;
    static constexpr int CTAS_PER_SM = DUAL ? 2 : 1;
    // registers are granted in blocks of 8 per thread: bound the pair of CTAs to 64 registers per thread
    static constexpr int BOUND_THREADS = DUAL ? 512 : THREADS;
    static_assert(A_COL0 + STAGES * 32 <= SF_COL, "tensor memory budget");
    static_assert(STAGES >= G, "a producer group must not lap the ring (parity waits)");
    static constexpr int W_TILE_BYTES = BN * ROWB;           // one K stage of the expanded weights
    static constexpr int HALF_BYTES = PROD_THREADS * 16;     // four K words of every producer thread
};

struct WsLayout {
    int ktiles;       // 256-bit K stages
    int halves;       // 16-byte halves staged per producer thread and ring slot
    int row_kt;       // > 0: producers work tile by tile (all row_kt stages of a row at once), see the producers
    int bits_bytes;   // staging ring of the packed words
    int smem;         // dynamic shared memory in bytes
};

template <int BN, int G, bool DUAL, int TEAMS = 1>
__host__ __device__ inline WsLayout ws_layout(int kwords, int mode)
{
    using C = Cfg<BN, G, DUAL, TEAMS>;
    WsLayout l;
    l.ktiles = (kwords + 7) >> 3;
    // Short K: a producer group takes whole tiles in turn instead of single stages, so the per-tile work
    // (row coordinates, tap mask, bookkeeping) is done once per row and tile.  A group then runs up to
    // (G - 1) * ktiles + 1 ring slots ahead of the slot it waits for; the parity waits need the ring
    // to be at least that deep.
    l.row_kt = (l.ktiles <= 2 && C::STAGES >= (G - 1) * l.ktiles + 1) ? l.ktiles : 0;
    l.halves = l.row_kt ? (kwords + 3) >> 2 : 2;
    l.bits_bytes = PF * C::HALF_BYTES * l.halves;
    l.smem = 1024 + l.ktiles * C::W_TILE_BYTES + l.bits_bytes + BN * 4 + l.ktiles * 32;
    if (mode == 2) l.smem += TEAMS * ID_RING_BYTES + 16;      // identity staging rings of the module epilogue
    if (mode == 0) l.smem += TEAMS * EPI_WARPS * I32_TILE_BYTES + 16;   // store staging tiles of the int32 epilogue
    // Tensor memory is shared out by the resident CTAs (all 512 columns, or 256 each for two): ask
    // for enough shared memory that no further CTA of this kernel fits on the SM (it would sit in
    // tcgen05.alloc until a neighbour exits).
    const int floor_bytes = DUAL ? 78 * 1024 : 120 * 1024;
    if (l.smem < floor_bytes) l.smem = floor_bytes;
    return l;
}

template <int BN, int G, bool DUAL, int MODE, int TEAMS = 1>
__global__ void __launch_bounds__(Cfg<BN, G, DUAL, TEAMS>::BOUND_THREADS, Cfg<BN, G, DUAL, TEAMS>::CTAS_PER_SM)
conv_tc_ws_kernel(const ConvProblem p)
{
    using C = Cfg<BN, G, DUAL, TEAMS>;
    static_assert(C::NBUF % TEAMS == 0, "a team's tiles must map to a fixed set of accumulator buffers");
    constexpr bool FUSED = MODE == 1, MODULE = MODE == 2;
    constexpr int NBUF = C::NBUF;
    constexpr int MAX_STAGES = 8;

    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 2 * 4];
    __shared__ uint32_t tmem_base_smem;
    __shared__ int abort_flag_smem;

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const WsLayout L = ws_layout<BN, G, DUAL, TEAMS>(p.kwords, MODE);
    const int ktiles = L.ktiles;
    constexpr int STAGES = C::STAGES;
    const int m_tiles = (p.M - 1) / BM + 1;                  // M >= 1; no overflow for M close to 2^31
    // N slices: a CTA keeps the weights of one slice of BN output channels and walks row tiles mb, mb + mstride, ...
    // (the grid is a multiple of the slice count)
    const int n_tiles = (p.C_out + BN - 1) / BN;
    const int n0 = ((int)blockIdx.x % n_tiles) * BN;
    const int cn = min(BN, p.C_out - n0);                     // channels of this slice
    const int mb = (int)blockIdx.x / n_tiles;
    const int mstride = (int)gridDim.x / n_tiles;
    const int my_tiles = (mb < m_tiles) ? (m_tiles - 1 - mb) / mstride + 1 : 0;
    const int total_items = my_tiles * ktiles;

    // shared-memory map (all 1024-byte aligned where the MMA reads)
    const uint32_t wexp = (smem_u32(smem_raw) + 1023u) & ~1023u;          // [ktiles][BN rows][128 B]
    const uint32_t bits_ring = wexp + (uint32_t)ktiles * C::W_TILE_BYTES; // [PF][halves][PROD_THREADS][16 B]
    const uint32_t colc_addr = bits_ring + (uint32_t)L.bits_bytes;                 // [BN] int32
    const uint32_t ktab_addr = colc_addr + BN * 4;                        // unit table of the gather: [ktiles * 8 / gw]
    const uint32_t idring = (ktab_addr + (uint32_t)ktiles * 32u + 15u) & ~15u;   // module epilogue only: [ID_SLOTS][BM rows][80 B]
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (MAX_STAGES + s); };
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * MAX_STAGES + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * MAX_STAGES + 4 + b); };
    volatile int *abort_flag = &abort_flag_smem;

    if (tid == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(full_bar(s), 4);          // the four warps of the group that owns the stage
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 4; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), EPI_WARPS);
        }
        abort_flag_smem = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"((uint32_t)C::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }

    const int gw = gather_width(p.cw);
    build_unit_table8(p, ktab_addr, ktiles * (8 / gw), gw, tid, C::THREADS);
    for (int c = tid; c < BN; c += C::THREADS) asm volatile("st.shared.b32 [%0], %1;" ::"r"(colc_addr + 4u * c), "r"(0) : "memory");
    pdl_wait();
    __syncthreads();
    // ---- one-off: expand the weight tile, count every row's set bits.  Eight lanes take the eight K words of one stage of
    // one row: coalesced loads, 128-byte rows stored without bank conflicts.
    // WU words of a thread are requested together (the expansion is otherwise one L2 latency per word).
    constexpr int WU = 8;
    const int wtotal = ktiles * BN * 8;                      // a multiple of 32: a warp's lanes stay together
    for (int i0 = tid; i0 < wtotal; i0 += WU * C::THREADS) {
        uint32_t w[WU];
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int idx = i0 + u * C::THREADS, row = (idx >> 3) / ktiles, kword = ((idx >> 3) - row * ktiles) * 8 + (idx & 7);
            w[u] = idx < wtotal && kword < p.kwords && row < cn ? __ldg(p.w + (long)(n0 + row) * p.kwords + kword) : 0u;
        }
#pragma unroll
        for (int u = 0; u < WU; ++u) {
            const int idx = i0 + u * C::THREADS, row = (idx >> 3) / ktiles, kt = (idx >> 3) - row * ktiles, e = idx & 7;
            if (idx >= wtotal) break;
            const bool live = kt * 8 + e < p.kwords && row < cn;           // rows / K words beyond the problem: zeros
            expand_store_w4(w[u], live, wexp + (uint32_t)kt * C::W_TILE_BYTES + (uint32_t)row * ROWB, row & 7, e);
            int pop = __popc(w[u]);
            pop += __shfl_xor_sync(0xffffffffu, pop, 1);
            pop += __shfl_xor_sync(0xffffffffu, pop, 2);
            pop += __shfl_xor_sync(0xffffffffu, pop, 4);
            if (e == 0) asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(colc_addr + 4u * row), "r"(pop) : "memory");
        }
    }
    fence_async_proxy();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    const uint32_t tmem_base = tmem_base_smem;

    if (warp == 0) {
        // ------------------------------------------------------------------ MMA issuer
        // This warp never touches memory: a load or an mbarrier wait issued after tensor-core
        // instructions holds the issuing thread until they have drained (measured: +230 cycles per
        // stage), a named barrier does not.  The control warp does the waiting and releases one
        // stage at a time through named barrier 1 + slot.  There is one issuer on purpose: the
        // producers' parity waits rely on the ring being consumed in order (a second issuer working on
        // the next tile lets a late slot fall two phases behind a waiting producer).
        constexpr uint32_t idesc = make_idesc_f4(BN);
        const uint64_t desc0 = make_desc(0);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32);
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);             // warp-uniform copy for the issuer
        const uint32_t a_tmem0 = tmem_u + (uint32_t)C::A_COL0;                   // + slot * 32 columns
        const uint32_t sf = tmem_u + (uint32_t)C::SF_COL;
        const uint32_t b_lo0 = (uint32_t)desc0 | ((wexp & 0x3FFFFu) >> 4);       // + kt * (W_TILE_BYTES / 16)
        int s = 0, buf = 0;
        for (int ti = 0; ti < my_tiles; ++ti) {
            const uint32_t d_tmem = tmem_u + (uint32_t)(buf * BN);
            const uint32_t tfull = tfull_bar(buf);
            for (int kt = 0; kt < ktiles; ++kt) {
                const uint32_t a_t = a_tmem0 + (uint32_t)s * 32u;
                const uint32_t b_lo = b_lo0 + (uint32_t)kt * (C::W_TILE_BYTES >> 4);
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
        // Stage `it` is released (bar.arrive on 1 + slot) once its ring slot is full and, for a tile's
        // first stage, once the accumulator buffer is free.  The slot being full implies that the
        // issuer is past the previous use of the same named barrier (it committed that slot's release).
        // After a time-out the remaining stages are released without waiting so that the issuer,
        // whose barrier wait has no time limit, always terminates; the error word tells the host.
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
    } else if (warp <= EPI_WARPS * TEAMS) {
        // ------------------------------------------------------------------ epilogue
        const int quad = warp & 3;
        const int erow = quad * 32 + lane;
        const int team = (warp - 1) >> 2;                        // takes the tiles team, team + TEAMS, ...
        const uint32_t i32_tile = idring + (uint32_t)(team * EPI_WARPS + quad) * I32_TILE_BYTES;   // int32 epilogue (shares the place of the module's rings)
        bool alive = true;
        // module epilogue: chunk q of this thread's row sequence = (tile q / nch, chunk q % nch); its identity values
        // are staged ID_AHEAD chunks ahead in ring slot q % ID_SLOTS
        const int nch = (cn + 31) >> 5;
        const uint32_t id_warp = idring + (uint32_t)team * ID_RING_BYTES + (uint32_t)(quad * 32) * ID_ROW_BYTES;   // slot 0, the warp's first row
        int pf_ti = team, pf_ch = 0, pf_slot = 0, cur_slot = 0;
        auto prefetch_next = [&]() {
            if (pf_ti < my_tiles) {
                const long row0 = (long)(mb + pf_ti * mstride) * BM + quad * 32;
                module_prefetch(p, id_warp + (uint32_t)pf_slot * (BM * ID_ROW_BYTES), row0, n0 + pf_ch * 32, lane);
                if (++pf_ch == nch) { pf_ch = 0; pf_ti += TEAMS; }
            } else {
                cp_async_commit();
            }
            if (++pf_slot == ID_SLOTS) pf_slot = 0;
        };
        if (MODULE)
            for (int a = 0; a < ID_AHEAD; ++a) prefetch_next();
        // the rows' bit counts -> the epilogue's column constants: K - 2 popc, for the packed output - thr
        // (a threshold beyond +-(K + 1) decides like that bound)
        for (int c = tid - 32; c < BN; c += 32 * EPI_WARPS * TEAMS) {
            int pop;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(pop) : "r"(colc_addr + 4u * c) : "memory");
            int cst = p.K - 2 * pop;
            if (FUSED) cst -= max(min(c < cn ? __ldg(p.thr + n0 + c) : 0, p.K + 1), -p.K - 1);
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(colc_addr + 4u * c), "r"(table_entry<MODE>(cst)) : "memory");
        }
        asm volatile("bar.sync 9, %0;" ::"n"(32 * EPI_WARPS * TEAMS) : "memory");
        for (int ti = team; ti < my_tiles; ti += TEAMS) {
            const int buf = ti % NBUF;                            // tiles use the accumulator buffers in turn
            const uint32_t buf_phase = (uint32_t)(ti / NBUF) & 1u;
            const int m_tile = mb + ti * mstride;
            const int em = m_tile * BM + erow;
            if (alive) alive = mbar_wait(tfull_bar(buf), buf_phase, abort_flag, p.err, ERR_EPILOGUE_TIMEOUT);
            alive = __all_sync(0xffffffffu, alive && !*abort_flag);
            if (!alive) break;
            tc_fence_after();
            const uint32_t t_addr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(buf * BN);
            uint32_t words[BN / 32];
#pragma unroll
            for (int ch = 0; ch < BN / 32; ++ch) {
                const int col0 = ch * 32;
                words[ch] = 0;
                if (col0 < cn) {                                      // warp-uniform
                    uint32_t v[32];
                    tc_ld32(t_addr + (uint32_t)col0, v);
                    if (FUSED) {
                        words[ch] = threshold_word(v, colc_addr + 4u * col0);
                    } else if (MODULE) {
                        float dot[32];
#pragma unroll
                        for (int i4 = 0; i4 < 8; ++i4) {
                            const uint4 c = ld_shared_v4(colc_addr + 4u * (col0 + 4 * i4));
                            dot[4 * i4] = __uint_as_float(fadd_bits(v[4 * i4], c.x));
                            dot[4 * i4 + 1] = __uint_as_float(fadd_bits(v[4 * i4 + 1], c.y));
                            dot[4 * i4 + 2] = __uint_as_float(fadd_bits(v[4 * i4 + 2], c.z));
                            dot[4 * i4 + 3] = __uint_as_float(fadd_bits(v[4 * i4 + 3], c.w));
                        }
                        prefetch_next();
                        cp_async_wait<ID_AHEAD>();                    // this chunk's copy has landed
                        words[ch] = module_chunk(p, dot, id_warp + (uint32_t)cur_slot * (BM * ID_ROW_BYTES), (long)em - lane, n0 + col0, lane);
                        if (++cur_slot == ID_SLOTS) cur_slot = 0;
                    } else {
                        int o[32];
                        biased_ints(v, colc_addr + 4u * col0, o);
                        const long row0 = (long)em - lane;
                        store_int32_block(static_cast<int32_t *>(p.out) + row0 * p.C_out + n0 + col0, p.C_out, o, i32_tile, row0, p.M, lane, cn - col0);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty_bar(buf));
            if ((FUSED || (MODULE && p.out != nullptr)) && em < p.M) {
                const int owords = p.C_out >> 5, swords = cn >> 5;      // words of a row, of this slice
                uint32_t *dst = static_cast<uint32_t *>(p.out) + (long)em * owords + (n0 >> 5);
                if (BN == 128 && swords == 4 && (owords & 3) == 0) {
                    *reinterpret_cast<uint4 *>(dst) = make_uint4(words[0], words[1], words[2], words[3]);
                } else if (BN >= 64 && swords == 2 && (owords & 1) == 0) {
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(words[0], words[1]);
                } else {
#pragma unroll
                    for (int ch = 0; ch < BN / 32; ++ch)
                        if (ch < swords) dst[ch] = words[ch];
                }
            }
        }
        if (MODULE) cp_async_wait<0>();
    } else {
        // ------------------------------------------------------------------ producers
        // Group g takes items g, g + G, ... of the CTA's flattened (tile, stage) list.  Per item a
        // thread copies its row's 256 bits of K into its staging slot (PF items ahead), then expands
        // the oldest staged item into the ring slot of tensor memory.
        const int ptid = tid - C::FIRST_PRODUCER_THREAD;
        const int grp = ptid >> 7;                               // group = 4 consecutive warps
        const int quad = warp & 3;                               // tensor-memory lane quadrant this warp may write
        const int row = quad * 32 + lane;                        // the four warps of a group cover rows 0..127
        constexpr uint32_t HALF_BYTES = C::HALF_BYTES;
        const uint32_t SLOT_BYTES = (uint32_t)L.halves * HALF_BYTES;
        const uint32_t bits0 = bits_ring + (uint32_t)ptid * 16u, bits_end = bits0 + PF * SLOT_BYTES;
        const uint32_t st_addr0 = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::A_COL0;
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        const TileStep step = make_tile_step(p, (uint32_t)(BM * mstride));
        // the scales are in place before this group's first arrival, which every MMA waits for
        if (grp == 0) write_unit_scales(tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)C::SF_COL);

        auto produce = [&](auto gw_tag) {
            constexpr int GW = decltype(gw_tag)::value;
            constexpr uint32_t TAB_STAGE = (8 / GW) * 4u;        // table bytes per stage
            // ---- load cursor
            RowCursor rc;
            rc.m = (uint32_t)mb * BM + (uint32_t)row;
            row_locate(p, rc);
            int l_kt = grp;
            int l_left = total_items > grp ? (total_items - grp + G - 1) / G : 0;
            while (l_kt >= ktiles) { l_kt -= ktiles; row_step(p, step, rc); }
            row_window(p, step, rc);
            uint32_t l_dst = bits0;
            auto issue = [&]() {
                gather_stage8<GW>(p.x, rc, ktab_addr + (uint32_t)l_kt * TAB_STAGE, l_dst, HALF_BYTES);
                l_dst += SLOT_BYTES;
                if (l_dst == bits_end) l_dst = bits0;
                --l_left;
                l_kt += G;
                if (l_kt >= ktiles) {
                    do { l_kt -= ktiles; row_step(p, step, rc); } while (l_kt >= ktiles);
                    row_window(p, step, rc);
                }
            };
#pragma unroll 1
            for (int n = 0; n < PF - 1; ++n) {
                if (l_left > 0) issue();
                cp_async_commit();
            }
            // ---- expand cursor
            uint32_t c_src = bits0;
            int s = grp;                          // ring slot (G <= STAGES) and its parity
            uint32_t phase = 1;                   // first pass through the ring: slots are free
#pragma unroll 1
            for (int it = grp; it < total_items; it += G) {
                if (l_left > 0) issue();
                cp_async_commit();
                cp_async_wait<PF - 1>();
                uint32_t v[32];               // column 4e + j = word j of K word e
                expand_stage8(ld_shared_v4(c_src), ld_shared_v4(c_src + HALF_BYTES), v);
                c_src += SLOT_BYTES;
                if (c_src == bits_end) c_src = bits0;
                if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) break;
                tc_fence_after();     // the MMAs that read this slot are complete (their commit released it)
                tc_st32(st_addr0 + (uint32_t)s * 32u, v);
                tc_fence_before();
                __syncwarp();
                mbar_arrive_pred(full_bar(s), lane0);
                s += G;
                if (s >= STAGES) { s -= STAGES; phase ^= 1u; }
            }
            cp_async_wait<0>();
        };
        // ---- short K: this group's items are the tiles grp, grp + G, ...; all stages of a row are staged
        // together (PF tiles ahead) and expanded one ring slot after the other
        auto produce_rows = [&](auto gw_tag, auto kt_tag) {
            constexpr int GW = decltype(gw_tag)::value;
            constexpr int KT = decltype(kt_tag)::value;
            constexpr uint32_t TAB_STAGE = (8 / GW) * 4u;
            const uint32_t TSLOT_BYTES = SLOT_BYTES;              // one staged tile: [halves][PROD_THREADS][16 B]
            const uint32_t tend = bits0 + PF * TSLOT_BYTES;
            const int nk_last = p.kwords - 8 * (KT - 1);          // K words of the row's last stage (1..8)
            const TileStep gstep = make_tile_step(p, (uint32_t)(BM * mstride * G));
            RowCursor rc;
            rc.m = (uint32_t)(mb + grp * mstride) * BM + (uint32_t)row;
            row_locate(p, rc);
            row_window(p, gstep, rc);
            int l_left = my_tiles > grp ? (my_tiles - grp + G - 1) / G : 0;
            uint32_t l_dst = bits0;
            auto issue = [&]() {
#pragma unroll
                for (int kt = 0; kt < KT; ++kt)
                    gather_stage8<GW>(p.x, rc, ktab_addr + (uint32_t)kt * TAB_STAGE, l_dst + (uint32_t)(2 * kt) * HALF_BYTES, HALF_BYTES,
                                      kt < KT - 1 ? 8 : ((nk_last + 3) & ~3) / GW);        // whole halves: what K lacks is zero-filled
                l_dst += TSLOT_BYTES;
                if (l_dst == tend) l_dst = bits0;
                --l_left;
                row_step(p, gstep, rc);
                row_window(p, gstep, rc);
            };
#pragma unroll 1
            for (int n = 0; n < PF - 1; ++n) {
                if (l_left > 0) issue();
                cp_async_commit();
            }
            uint32_t c_src = bits0;
            int s = grp * KT;                     // ring slot of the tile's first stage and its parity
            uint32_t phase = 1;
            while (s >= STAGES) { s -= STAGES; phase ^= 1u; }
#pragma unroll 1
            for (int ti = grp; ti < my_tiles; ti += G) {
                if (l_left > 0) issue();
                cp_async_commit();
                cp_async_wait<PF - 1>();
                bool alive = true;
#pragma unroll
                for (int kt = 0; kt < KT; ++kt) {
                    if (alive && !mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_PRODUCER_TIMEOUT)) alive = false;
                    if (alive) {
                        tc_fence_after();
                        expand_store_stage8(st_addr0 + (uint32_t)s * 32u, c_src + (uint32_t)(2 * kt) * HALF_BYTES, HALF_BYTES, kt < KT - 1 ? 8 : nk_last);
                        tc_wait_st();
                        tc_fence_before();
                        __syncwarp();
                        mbar_arrive_pred(full_bar(s), lane0);
                    }
                    if (++s == STAGES) { s = 0; phase ^= 1u; }
                }
                if (!alive) break;
                c_src += TSLOT_BYTES;
                if (c_src == tend) c_src = bits0;
                s += (G - 1) * KT;                // the other groups' tiles
                while (s >= STAGES) { s -= STAGES; phase ^= 1u; }
            }
            cp_async_wait<0>();
        };
        auto rows_by_kt = [&](auto gw_tag) {
            if (L.row_kt == 1) produce_rows(gw_tag, IntC<1>{});
            else produce_rows(gw_tag, IntC<2>{});
        };
        if (L.row_kt) {
            if (gw == 4) rows_by_kt(IntC<4>{});
            else if (gw == 2) rows_by_kt(IntC<2>{});
            else rows_by_kt(IntC<1>{});
        } else if (gw == 4) produce(IntC<4>{});
        else if (gw == 2) produce(IntC<2>{});
        else produce(IntC<1>{});
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)C::TMEM_COLS) : "memory");
    }
}

template <int BN, int G, bool DUAL, int TEAMS = 1>
int launch_ws(const ConvProblem &p0, cudaStream_t stream)
{
    ConvProblem p = p0;
    p.err = device_error_word();
    const int sms = sm_count();
    using C = Cfg<BN, G, DUAL, TEAMS>;
    const WsLayout L = ws_layout<BN, G, DUAL, TEAMS>(p.kwords, p.mode);
    const long m_tiles = ((long)p.M + BM - 1) / BM;
    const long slots = (long)sms * C::CTAS_PER_SM;
    const long n_tiles = (p.C_out + BN - 1) / BN;
    long per_slice = slots / n_tiles;                         // CTAs that share one slice of the weights
    if (per_slice < 1) return BCNN_ERR_UNSUPPORTED;
    if (per_slice > m_tiles) per_slice = m_tiles;
    const unsigned grid = (unsigned)(per_slice * n_tiles);
    void (*k)(const ConvProblem) = p.mode == 2 ? conv_tc_ws_kernel<BN, G, DUAL, 2, TEAMS>
                                   : (p.mode == 1 ? conv_tc_ws_kernel<BN, G, DUAL, 1, TEAMS> : conv_tc_ws_kernel<BN, G, DUAL, 0, TEAMS>);
    if (!allow_smem((const void *)k, DUAL ? 113 * 1024 : MAX_SMEM - 1024)) return BCNN_ERR_CUDA;
    return launch(k, grid, C::THREADS, L.smem, stream, p);
}

// The expanded weights, the packed-word staging ring and the tables must fit in shared memory
// (in half of it when two CTAs share an SM).
template <int BN, int G, bool DUAL, int TEAMS = 1>
bool fits(const ConvProblem &p)
{
    return ws_layout<BN, G, DUAL, TEAMS>(p.kwords, p.mode).smem <= (DUAL ? 113 * 1024 : MAX_SMEM - 1024);
}

}  // namespace

bool conv_tc_ws_supports(const ConvProblem &p)
{
    if (p.mode != 0 && (p.C_out % 32 != 0)) return false;
    if (p.kh * p.kw > 31 || p.K > (1 << 16)) return false;
    // rows address the input by 32-bit word offsets
    if ((long)p.B * p.H * p.W * p.cw >= (1L << 31) || (long)p.kh * p.W * p.cw >= (1L << 27)) return false;
    if (p.C_out <= 32) return fits<32, 4, false>(p);
    if (p.C_out <= 64) return fits<64, 4, false>(p);
    if (fits<128, 4, false>(p) || fits<128, 2, false>(p)) return p.C_out <= 128 * 64;
    // wider layers whose 128-channel slice of the weights does not fit: 64-channel slices
    return p.C_out > 128 && p.C_out <= 64 * 64 && fits<64, 4, false>(p);
}

// A wide layer whose K is too long for slices of 128 channels runs in slices of 64.
bool conv_tc_ws_narrow_slices(const ConvProblem &p)
{
    return p.C_out > 128 && !fits<128, 4, false, 2>(p) && !fits<128, 2, true>(p) && !fits<128, 2, false>(p);
}

// Expected time, ns: a start, the expansion of a slice's weights by K, and per row tile of the longest CTA a term and one per 256-bit stage by how
// the gather goes; int32 outputs by their number.  Fitted to 3530 drawn layers and products within 5 to 11 % (one standard deviation); slices of 64, which
// expand every row tile twice as often, to 94 products within 5 % (with the rates of 128 the estimate was 0.79 to 0.89 of their time).
long conv_tc_ws_estimate(const ConvProblem &p)
{
    struct Rates {
        long start, weights, tile, stage[3], out;
    };
    // up to 64 channels, up to 128, slices of 128, slices of 64; packed, int32
    static constexpr Rates RATES[2][4] = {
        {{4140, 210, 180, {154, 166, 215}, 0}, {4400, 500, 560, {135, 147, 173}, 0}, {4730, 346, 490, {195, 189, 230}, 0}, {4870, 276, 270, {161, 211, 299}, 0}},
        {{4450, 190, 141, {145, 161, 205}, 782}, {5670, 455, 543, {102, 131, 172}, 600}, {5100, 317, 1508, {173, 158, 205}, 268}, {5705, 273, 157, {186, 192, 330}, 173}}};
    const bool halved = conv_tc_ws_narrow_slices(p);
    const Rates &r = RATES[p.mode == 1 ? 0 : 1][p.C_out <= 64 ? 0 : p.C_out <= 128 ? 1 : halved ? 3 : 2];
    const long width = halved ? 64 : 128, slices = (p.C_out + width - 1) / width, ctas = sm_count() / slices > 0 ? sm_count() / slices : 1, kt = (p.kwords + 7) / 8;
    const long tiles = (((long)p.M + BM - 1) / BM + ctas - 1) / ctas;
    const int gw = gather_width(p.cw);
    return r.start + kt * r.weights + tiles * (r.tile + kt * r.stage[gw == 4 ? 0 : gw == 2 ? 1 : 2]) + (long)p.M * p.C_out / 1000 * r.out / 1000;
}

int launch_conv_tc_ws(const ConvProblem &p, cudaStream_t stream)
{
    if (!conv_tc_ws_supports(p)) return BCNN_ERR_UNSUPPORTED;
    // module epilogue: bound by the epilogue warps, so two teams of them, one producer group and two CTAs per SM;
    // layers wider than 64 channels run as 64-channel slices (two accumulator buffers are needed for two teams)
    if (p.mode == 2) {
        if (p.C_out <= 32 && fits<32, 1, true, 2>(p)) return launch_ws<32, 1, true, 2>(p, stream);
        if (p.C_out > 32 && fits<64, 1, true, 2>(p)) return launch_ws<64, 1, true, 2>(p, stream);
        if (p.C_out > 32 && p.C_out <= 32 * 64 && fits<32, 1, true, 2>(p)) return launch_ws<32, 1, true, 2>(p, stream);   // long K: 32-channel slices
    }
    // narrow layers: the per-stage cost of issuing MMAs exceeds their execution time, so two CTAs
    // per SM (two issuers) when the resident weights leave room for it
    if (p.C_out <= 32) return fits<32, 2, true>(p) ? launch_ws<32, 2, true>(p, stream) : launch_ws<32, 4, false>(p, stream);
    if (p.C_out <= 64) return fits<64, 2, true>(p) ? launch_ws<64, 2, true>(p, stream) : launch_ws<64, 4, false>(p, stream);
    // C_out > 128: slices of 128 (or 64) output channels, each CTA keeps one slice's weights
    if (fits<128, 4, false, 2>(p)) return launch_ws<128, 4, false, 2>(p, stream);
    if (fits<128, 2, true>(p)) return launch_ws<128, 2, true>(p, stream);
    if (fits<128, 2, false>(p)) return launch_ws<128, 2, false>(p, stream);     // long K: fewer producer groups, smaller staging ring
    return fits<64, 2, true>(p) ? launch_ws<64, 2, true>(p, stream) : launch_ws<64, 4, false>(p, stream);
}

}  // namespace bcnn
