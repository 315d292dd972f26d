// Convolution module on pointwise layers (Section 4.2.1, Figure 4): P >= 1 binary branches on the tensor cores, then per
// branch batch norm, the branch sum, + identity, PReLU, fp16 map and the next module's signs, in one pass.  P = kh * kw
// shifted branches (the stand-in for a binary kh x kw convolution) run here too.
//
// Bound by the fp16 maps' traffic (2 bytes of identity read and 2 bytes written per output) as long as the epilogue
// spends less than about 20 instructions per output, so everything is built around the epilogue:
//   * identity tiles arrive and output tiles leave by tiled TMA copies of 128 rows x BN channels through a ring of NS tiles per
//     epilogue team in shared memory (swizzled: one 16-byte access per lane and row without bank conflicts); a loader warp and a
//     store warp issue them (an issue costs its warp some 500 cycles), the epilogue turns a tile in place;
//   * accumulators are loaded so that a lane holds a quarter of a part's channels of four rows (16x256b; the weights' rows are
//     permuted to make them consecutive channels): a channel's values - per branch {scale, shift}, then {slope, sign threshold}, pairs of
//     channels in 16 bytes - are fetched once for four rows, the four rows are independent chains, and sign bits end in whole
//     bytes.  With a row per lane a P = 2 part took 3800 cycles of a team, now 2640 (P = 1: 2150, 1780).  The constant K - 2 popc of a
//     dot product is not among them, an MMA against a constant tile puts it into the accumulator (tc_slot.cuh);
//   * the arithmetic runs on pairs (f32x2: the same IEEE operations, half the issue slots); PReLU is a compare and a predicated product; the
//     next sign is one fp16 compare per pair against the smallest fp16 value that passes;
//   * two epilogue teams take alternate PARTS (128 rows x BN channels).
// The binary products are cheap beside that: a CTA keeps RS slices of BN channels' expanded weights in shared memory, expands
// a row tile once (256-bit stages in a ring in tensor memory, as in conv_tc_ws.cu) and multiplies it against every resident
// slice; branch p of a part has BN accumulator columns of its own (its result is scaled before the sum).  A branch's K
// is padded to an even number of words: two words per MMA.
// Arithmetic (bit-exact against the oracle): t_p = dot_p * scale_p + shift_p, summed in branch order, + identity, PReLU,
// fp16, sign of (stored value + next bias): one fp32 operation per step, no contraction.
// "Part full" barriers form a ring of MAX_NBUF, not of the accumulator buffers in use: a parity wait for part n is right once
// part n - MAX_NBUF is done, and the team has seen part n - TEAMS done (with one buffer and two teams the second team's first
// wait would pass on the barrier's empty history).
// What a launch does once - weights, parameters, constants - is written as small rolled loops with its divisions prepared on the host: an
// instruction that runs for the first time costs some ten cycles, and unrolled eight times this set-up took 5 us.  In microseconds,
// before and after: P = 2, 256 channels, M = 50176: 23.6, 18.6; P = 3, 160 channels, M = 96228: 47.7, 31.8; P = 3, 96 channels, M = 10496: 10.1, 7.6;
// nine taps, 128 channels, M = 12544: 31.1, 19.9; P = 1, 128 channels: M = 1782 4.9, 3.9, M = 153064 18.8, 15.9 (12.3 of the maps' traffic).
// Every mbarrier wait is bounded and reports through the device error word.
#include "tc_slot.cuh"
#include "tensor_map.cuh"

namespace bcnn {

namespace {

using namespace tc;

constexpr int ERR_MOD_PRODUCER = 171, ERR_MOD_ISSUER = 172, ERR_MOD_EPILOGUE = 173, ERR_MOD_IDENTITY = 174, ERR_MOD_LOADER = 175, ERR_MOD_STORE = 176;

constexpr int G = 2;                      // producer groups of four warps
constexpr int PF = 3;                     // packed-word stages in flight per producer thread
constexpr int TEAMS = 2, NS = 3;          // epilogue teams of four warps; staging tiles per team
constexpr int ISSUER = 0, LOADER = 1, STORER = 2 /* + team */, FIRST_PRODUCER = STORER + TEAMS, FIRST_EPILOGUE = FIRST_PRODUCER + 4 * G;
constexpr int THREADS = 32 * (FIRST_EPILOGUE + 4 * TEAMS);
constexpr int PROD_THREADS = G * BM;
constexpr int HALF_BYTES = PROD_THREADS * 16, SLOT_BYTES = 2 * HALF_BYTES;
constexpr int MAX_STAGES = 11, MAX_NBUF = 4;
constexpr int MAX_SMEM = 226 * 1024;

struct ModPlan {
    ConvProblem q;            // the layer as its gather sees it: cw = words of an input pixel (all branches)
    const float *scale, *shift;       // [P][C_out]
    const int32_t *pad_dot;   // [P][C_out] or nullptr (0)
    int P, bcw, kwp;          // branches; words of a branch, padded to even
    int kst;                  // 256-bit stages of a row
    int stages;               // ring slots
    int nbuf;                 // accumulator buffers
    int rs, ng, slices;       // resident slices, CTA groups, slices of BN channels
    int m_tiles, step;        // row tiles; CTAs of a group
    uint32_t ng_mul, ng_shift, step_mul, step_shift;      // exact_div by ng and step
    uint32_t kwp_mul, kwp_shift, row_mul, row_shift;      // ... by kwp and by the gw-word pieces of a branch's weight row
    TileStep ts;              // from a row tile to the CTA's next
    int units, gw;            // gather units of a row
    uint32_t off_bits, off_stage, off_table, off_pad, off_tab, off_const, off_raw;      // shared-memory offsets from the 1024-byte aligned base (weights first)
    int early_tiles;          // staging tiles ahead of the packed weights, which lie over the others until they are expanded
};

// a pair of channels in the parameter table: P entries of 16 bytes {scale, shift} x 2, then 16 bytes {slope x 2, sign threshold x 2 (fp16), -}
__host__ __device__ inline uint32_t pair_bytes(int P) { return 16u * (uint32_t)P + 16u; }
// constant tiles: four 32-byte rows of (slice, branch) pairs side by side
__host__ __device__ inline int const_tiles(int rs, int P) { return (rs * P + 3) / 4; }

__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ unsigned long long bits2(uint32_t a, uint32_t b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ float2 floats2(unsigned long long v)
{
    float2 f;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
    return f;
}
// The two products one by one: ptxas contracts mul.rn.f32x2 (and a multiply-add with -0) with the addition behind it, one
// rounding instead of two; __fmul_rn is never contracted.
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b)
{
    const float2 x = floats2(a), y = floats2(b);
    return bits2(__float_as_uint(__fmul_rn(x.x, y.x)), __float_as_uint(__fmul_rn(x.y, y.y)));
}
// 8 accumulator columns of this warp's 32 rows, lane l = columns 2 (l % 4) and + 1 of rows l / 4 + 8 i in v[2 i], v[2 i + 1]: a
// lane meets two channels instead of all of them, so a channel's parameters are fetched once for four rows.
__device__ __forceinline__ void tc_ld8_quads_nowait(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr) : "memory");
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "r"(taddr + (16u << 16)) : "memory");
}
__device__ __forceinline__ void pin_regs8(uint32_t (&v)[8])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]) :: "memory");
}
__device__ __forceinline__ uint32_t ld_shared_b32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
// u >= 0 ? u : slope * u
__device__ __forceinline__ float prelu(float u, float slope)
{
    asm("{\n\t.reg .pred p;\n\tsetp.ge.f32 p, %0, 0f00000000;\n\t@!p mul.rn.f32 %0, %0, %1;\n\t}" : "+f"(u) : "f"(slope));
    return u;
}
// The smallest fp16 y for which y + nb >= 0 in fp32.  A sum of two numbers has the sign of the exact sum (nothing underflows to 0),
// so for finite nb that is -nb rounded up; a NaN, which no y reaches, where no y will do (y + nb is -infinity or NaN); and
// the most negative number for nb = +infinity, where only -infinity and NaN give no sum >= 0.
__device__ __forceinline__ uint16_t sign_threshold(float nb)
{
    if (!(nb > -INFINITY)) return 0x7E00u;
    if (nb == INFINITY) return 0xFBFFu;
    return __half_as_ushort(__float2half_ru(-nb));
}
// Accumulator column of channel c of a part.  Column 8 k + 2 q + o is held by lane 4 r + q of a load, which is to own the BN / 4
// consecutive channels from q * BN / 4: 16-byte pieces of the identity's and the output's rows, and whole bytes of sign bits.
template <int BN> __host__ __device__ constexpr int column_of_channel(int c)
{
    return ((c >> 1) & (BN / 8 - 1)) * 8 + c / (BN / 4) * 2 + (c & 1);
}
template <int BN> __host__ __device__ constexpr int channel_of_column(int n) { return ((n >> 1) & 3) * (BN / 4) + (n >> 3) * 2 + (n & 1); }
// bytes of a lane's share of the parameter table (16 more than its entries: the four shares lie in different banks)
template <int BN> __host__ __device__ constexpr uint32_t share_bytes(uint32_t pair) { return (uint32_t)(BN / 8) * pair + 16u; }

// BN: channels of a part (64, 32); PP: branches; SHIFTED: taps with a row mask
template <int BN, int PP, bool SHIFTED, bool HAS_ID>
__global__ void __launch_bounds__(THREADS, 1)
conv_tc_mod_kernel(const ModPlan L, const __grid_constant__ CUtensorMap idmap, const __grid_constant__ CUtensorMap ymap)
{
    constexpr int TILE_BYTES = BM * BN * 2, ROW_BYTES = BN * 2, W_STAGE = BN * ROWB;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[2 * MAX_STAGES + 2 * MAX_NBUF + 3 * TEAMS * NS + 1];
    __shared__ uint32_t tmem_base_smem;
    __shared__ int abort_flag_smem;

    const ConvProblem &p = L.q;
    constexpr int P = PP;
    constexpr bool ROLLED = SHIFTED || PP >= 11;              // (below: the channel pairs of a piece in a loop)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kst = L.kst, stages = L.stages;
    const int idx = (int)exact_div(blockIdx.x, L.ng_mul, L.ng_shift), cg = (int)blockIdx.x - idx * L.ng, step = L.step;
    const int rs = min(L.rs, L.slices - cg * L.rs);
    const int my_tiles = idx < L.m_tiles ? (int)exact_div((uint32_t)(L.m_tiles - 1 - idx), L.step_mul, L.step_shift) + 1 : 0;
    const int parts = my_tiles * rs;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;         // [rs][kst][BN rows][128 B] weights, then the rest
    const uint32_t bits_ring = base + L.off_bits, staging = base + L.off_stage, table = base + L.off_table;
    const uint32_t tab = base + L.off_tab, pads = base + L.off_pad, cexp = base + L.off_const;
    const uint32_t bar0 = smem_u32(bars);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (MAX_STAGES + s); };
    static_assert(MAX_NBUF >= TEAMS, "ring of part-full barriers");
    auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * MAX_STAGES + b); };
    auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * MAX_STAGES + MAX_NBUF + b); };
    auto id_full = [&](int t, int s) { return bar0 + 8u * (2 * MAX_STAGES + 2 * MAX_NBUF + t * NS + s); };
    auto slot_free = [&](int t, int s) { return bar0 + 8u * (2 * MAX_STAGES + 2 * MAX_NBUF + TEAMS * NS + t * NS + s); };
    auto out_full = [&](int t, int s) { return bar0 + 8u * (2 * MAX_STAGES + 2 * MAX_NBUF + 2 * TEAMS * NS + t * NS + s); };
    const uint32_t ready_bar = bar0 + 8u * (2 * MAX_STAGES + 2 * MAX_NBUF + 3 * TEAMS * NS);      // the resident weights are expanded
    volatile int *abort_flag = &abort_flag_smem;

    constexpr int NBARS = sizeof(bars) / 8;
    if (tid < NBARS) {
        // a full slot: its four producer warps; a free buffer: a team; an output tile: a team; the weights: all epilogue warps; else one
        constexpr int T0 = 2 * MAX_STAGES + MAX_NBUF, O0 = 2 * MAX_STAGES + 2 * MAX_NBUF + 2 * TEAMS * NS;
        const bool team = tid < MAX_STAGES || (tid >= T0 && tid < T0 + MAX_NBUF) || (tid >= O0 && tid < O0 + TEAMS * NS);
        mbar_init(bar0 + 8u * tid, tid == NBARS - 1 ? 4 * TEAMS : (team ? 4 : 1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 0) abort_flag_smem = 0;
    if (warp == ISSUER) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // gather table: unit u = K words u * gw ..; word w belongs to branch w / kwp (its tap when shifted)
#pragma unroll 1
    for (int u = tid; u < L.units; u += THREADS) {
        const int w = u * L.gw, br = (int)exact_div((uint32_t)w, L.kwp_mul, L.kwp_shift), j = w - br * L.kwp;
        uint32_t ent = (uint32_t)TAP_NONE << 27;
        if (br < P && j < L.bcw) {
            int off = br * L.bcw + j;
            if (SHIFTED) {
                const int r = br / p.kw, t = br - r * p.kw;
                off += (r * p.W + t) * p.cw;
            }
            ent = (uint32_t)off | ((uint32_t)(SHIFTED ? br : 0) << 27);
        }
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(tab + 4u * u), "r"(ent) : "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    // (each role that touches global memory waits for the previous kernel behind its own set-up: instructions that run for the first
    // time cost some ten cycles each, which hide in that kernel's tail)
    const uint32_t tmem_base = tmem_base_smem;

    // part n = (row tile n / rs, slice n % rs); team n % TEAMS, its m = n / TEAMS-th part, staging tile m % NS
    struct Part {
        int row, slice;
        __device__ __forceinline__ void skip(int n, int rs, int rows) { for (slice += n; slice >= rs; slice -= rs) row += rows; }
    };
    const int tile_rows = step * BM, ch_base = cg * L.rs * BN;
    auto stage_tile = [&](int t, int s) { return staging + (uint32_t)((s * TEAMS + t) * TILE_BYTES); };      // in the order of their first use

    if (warp == ISSUER) {
        // ------------------------------------------------------------------ MMA issuer
        constexpr uint32_t idesc = make_idesc_f4(BN);
        const uint64_t desc0 = make_desc(base);
        const uint32_t desc_hi = (uint32_t)(desc0 >> 32), b_lo0 = (uint32_t)desc0;
        const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem_base, 0);
        const uint32_t sf = tmem_u + (uint32_t)CB_COL, c_lo0 = (uint32_t)make_desc(cexp), a_col0 = tmem_u + (uint32_t)(L.nbuf * P * BN);
        const int per_branch = L.kwp >> 1, granules = P * per_branch;      // two-word MMAs of a branch, of a row
        // (the elected lane runs the whole loop: a vote and a reconvergence per instruction cost more than the instruction)
        if (elect_one()) {
            bool ok = mbar_wait(ready_bar, 0, abort_flag, p.err, ERR_MOD_ISSUER);
            int s = 0, buf = 0, slot0 = 0;                      // part = (row tile, slice s); its buffer; the tile's first item and ring slot
            uint32_t buf_phase = 1, ring_phase0 = 0;                       // first use of every accumulator buffer: free
            for (int n = 0; n < parts && ok; ++n) {
                ok = mbar_wait(tempty_bar(buf), buf_phase, abort_flag, p.err, ERR_MOD_ISSUER);
                if (!ok) break;
                const uint32_t d0 = tmem_u + (uint32_t)(buf * P * BN);
                int br = 0, j = 0, slot = slot0;                           // branch and MMA within it
                uint32_t ring_phase = ring_phase0;
                for (int k = 0; k < kst; ++k) {
                    if (s == 0) {
                        ok = mbar_wait(full_bar(slot), ring_phase, abort_flag, p.err, ERR_MOD_ISSUER);
                        if (!ok) break;
                    }
                    tc_fence_after();
                    const uint32_t a_t = a_col0 + (uint32_t)slot * 32u, b_lo = b_lo0 + (uint32_t)((s * kst + k) * (W_STAGE >> 4));
                    const int here = min(4, granules - 4 * k);
                    for (int g4 = 0; g4 < here; ++g4) {
                        const uint32_t d = d0 + (uint32_t)(br * BN);
                        if (j == 0) {                                      // the branch's constants
                            const int ct = s * P + br;
                            tc_mma_const(d, tmem_u, c_lo0 + (uint32_t)((ct >> 2) * (W_STAGE >> 4) + 2 * (ct & 3)), desc_hi, idesc);
                        }
                        tc_mma_f4_ts(d, a_t + 8u * g4, b_lo + 2u * g4, desc_hi, idesc, sf, 1u);
                        if (++j == per_branch) { j = 0; ++br; }
                    }
                    if (s == rs - 1) tc_commit(empty_bar(slot));           // the row tile's last part: the stage may be refilled
                    if (++slot == stages) { slot = 0; ring_phase ^= 1u; }
                }
                if (!ok) break;
                tc_commit(tfull_bar(n % MAX_NBUF));
                if (++buf == L.nbuf) { buf = 0; buf_phase ^= 1u; }
                if (++s == rs) { s = 0; slot0 = slot; ring_phase0 = ring_phase; }
            }
        }
        __syncwarp();
    } else if (warp == LOADER) {
        // ------------------------------------------------------------------ identity tiles
        if (HAS_ID) {
            int issued = 0, team = 0, s = 0;
            uint32_t phase = 1;                                             // first lap: tiles are free
            Part at = {idx * BM, 0};
            pdl_wait();
#pragma unroll 1
            for (int n = 0; n < parts; ++n, ++issued, at.skip(1, rs, tile_rows)) {
                // the epilogue's warps are done with the packed weights, which lay here
                if (n == L.early_tiles && !mbar_wait_warp(ready_bar, 0, abort_flag, p.err, ERR_MOD_LOADER)) break;
                if (!mbar_wait_warp(slot_free(team, s), phase, abort_flag, p.err, ERR_MOD_LOADER)) break;
                if (lane == 0) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(id_full(team, s)), "r"((uint32_t)TILE_BYTES) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(stage_tile(team, s)), "l"(reinterpret_cast<uint64_t>(&idmap)), "r"(ch_base + at.slice * BN), "r"(at.row),
                                   "r"(id_full(team, s)) : "memory");
                }
                __syncwarp();
                if (++team == TEAMS) {
                    team = 0;
                    if (++s == NS) { s = 0; phase ^= 1u; }
                }
            }
            // after a time-out elsewhere: copies still in flight must land before the CTA's shared memory goes away
            if (*abort_flag)
                for (int n = issued > TEAMS * NS ? issued - TEAMS * NS : 0; n < issued; ++n)
                    mbar_wait_warp(id_full(n % TEAMS, (n / TEAMS) % NS), (uint32_t)(n / TEAMS / NS) & 1u, abort_flag, nullptr, 0);
        }
    } else if (warp < FIRST_PRODUCER) {
        // ------------------------------------------------------------------ output tiles of team warp - STORER
        const int team = warp - STORER;
        int s = 0, before = -1;
        uint32_t phase = 0;
        Part at = {idx * BM, 0};
        at.skip(team, rs, tile_rows);
        pdl_wait();
#pragma unroll 1
        for (int n = team; n < parts; n += TEAMS, at.skip(TEAMS, rs, tile_rows)) {
            if (!mbar_wait_warp(out_full(team, s), phase, abort_flag, p.err, ERR_MOD_STORE)) break;
            if (lane == 0) {
                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                             ::"l"(reinterpret_cast<uint64_t>(&ymap)), "r"(ch_base + at.slice * BN), "r"(at.row), "r"(stage_tile(team, s)) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                if (before >= 0) {                                          // the store before this one has read its tile
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    mbar_arrive(slot_free(team, before));
                }
            }
            __syncwarp();
            before = s;
            if (++s == NS) { s = 0; phase ^= 1u; }
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    } else if (warp >= FIRST_EPILOGUE) {
        // ------------------------------------------------------------------ epilogue
        // ---- one-off, while the first rows and identity tiles arrive: the resident slices' packed weights and parameters come to shared
        // memory in one go, eight lanes expand a (branch, slice, channel) row and count its bits, then the constants (the issuer
        // waits for weights and constants).  Rolled loops on purpose: this code runs once, and its instructions come from memory.
        // (A thread per word with eight loads in flight, an atomic per word and a division per index took 5 us for two branches
        // of 256 channels, a quarter of the kernel at 50176 rows.)  What comes lies over the staging tiles behind the first ones, which hold nothing
        // until all of it is expanded: in an area of its own it left P = 2, 256 channels two resident slices instead of four, and P = 8, 1024
        // channels no room at all.  (Without an identity these same warps are the tiles' first users.)
        constexpr int ETHREADS = 128 * TEAMS;
        const int etid = tid - 32 * FIRST_EPILOGUE;
        const int rows1 = rs * BN, rows_w = P * rows1;                      // rows of a branch, of all
        const int chans = min(rows1, p.C_out - ch_base);                    // the channels that exist
        const uint32_t pair = pair_bytes(P), share = share_bytes<BN>(pair);
        const uint32_t raw = base + L.off_raw, raw_par = raw + (uint32_t)(rows_w * L.bcw) * 4u;      // weights; then scale, shift (, pad) by branch, slope, next bias
        constexpr int PA = SHIFTED ? 3 : 2;
        pdl_wait();
#pragma unroll 1
        for (int br = 0; br < P; ++br) {
            const long first = (long)br * p.C_out + ch_base;
            const uint32_t *src = p.w + first * L.bcw;
            const uint32_t dst = raw + (uint32_t)(br * rows1 * L.bcw) * 4u, dpar = raw_par + (uint32_t)(PA * br * rows1) * 4u;
#pragma unroll 1
            for (int i = 4 * etid; i < chans * L.bcw; i += 4 * ETHREADS) cp_async16(dst + 4u * i, src + i, true);
            if (4 * etid < chans) {
                cp_async16(dpar + 16u * etid, L.scale + first + 4 * etid, true);
                cp_async16(dpar + 4u * rows1 + 16u * etid, L.shift + first + 4 * etid, true);
                if (SHIFTED) cp_async16(dpar + 8u * rows1 + 16u * etid, L.pad_dot ? L.pad_dot + first + 4 * etid : reinterpret_cast<const int32_t *>(L.scale), L.pad_dot != nullptr);
            }
        }
        const uint32_t raw_slope = raw_par + (uint32_t)(PA * P * rows1) * 4u, raw_nb = raw_slope + 4u * rows1;
        if (4 * etid < chans) {
            cp_async16(raw_slope + 16u * etid, p.slope + ch_base + 4 * etid, true);
            cp_async16(raw_nb + 16u * etid, p.next_bias ? p.next_bias + ch_base + 4 * etid : p.slope, p.next_bias != nullptr);
        }
        cp_async_commit();
        cp_async_wait<0>();
        asm volatile("bar.sync 1, %0;" ::"n"(ETHREADS) : "memory");
        // A piece is four words of a row where a branch has a multiple of four, else two (the last one half empty if bcw is odd).  Rows
        // go by accumulator column: neighbouring lanes then write to different places of the swizzle.
        const int pw = L.gw == 4 ? 4 : 2, per_row = L.kwp / pw, pieces = rows_w * per_row;
#pragma unroll 1
        for (int i = etid; i < pieces; i += ETHREADS) {
            const int r = (int)exact_div((uint32_t)i, L.row_mul, L.row_shift), j = (i - r * per_row) * pw;
            const int col = r % BN, sb = r / BN, sl = sb / P, br = sb - sl * P;
            const uint32_t src = raw + (uint32_t)((br * rows1 + sl * BN + channel_of_column<BN>(col)) * L.bcw + j) * 4u;
            const int kw = br * L.kwp + j;
            const uint32_t dst = base + (uint32_t)((sl * kst + (kw >> 3)) * W_STAGE + col * ROWB), x = (uint32_t)((kw & 7) ^ (col & 7)) << 4;
            if (pw == 4) {
                const uint4 w = ld_shared_v4(src);
                const uint4 o0 = expand_w4(w.x), o1 = expand_w4(w.y), o2 = expand_w4(w.z), o3 = expand_w4(w.w);
                st_shared_v4(dst + x, o0.x, o0.y, o0.z, o0.w);
                st_shared_v4(dst + (x ^ 16u), o1.x, o1.y, o1.z, o1.w);
                st_shared_v4(dst + (x ^ 32u), o2.x, o2.y, o2.z, o2.w);
                st_shared_v4(dst + (x ^ 48u), o3.x, o3.y, o3.z, o3.w);
            } else {
                const bool two = j + 1 < L.bcw;
                const uint4 o0 = expand_w4(ld_shared_b32(src)), o1 = two ? expand_w4(ld_shared_b32(src + 4u)) : make_uint4(0u, 0u, 0u, 0u);
                st_shared_v4(dst + x, o0.x, o0.y, o0.z, o0.w);
                st_shared_v4(dst + (x ^ 16u), o1.x, o1.y, o1.z, o1.w);
            }
        }
#pragma unroll 1
        for (int r = etid; r < rows1; r += ETHREADS) {
            const int c = r % BN, sl = r / BN, col = column_of_channel<BN>(c);
            const uint32_t odd = (uint32_t)(c & 1);
            const int pi = (sl * 4 + c / (BN / 4)) * (BN / 8) + ((c >> 1) & (BN / 8 - 1));
            const uint32_t ent = table + (uint32_t)(sl * 4 + c / (BN / 4)) * share + (uint32_t)((c >> 1) & (BN / 8 - 1)) * pair + 4u * odd;
#pragma unroll 1
            for (int br = 0; br < P; ++br) {
                const int ct = sl * P + br;
                const uint32_t par = raw_par + (uint32_t)(PA * br * rows1 + r) * 4u, wrow = raw + (uint32_t)((br * rows1 + r) * L.bcw) * 4u;
                int pop = 0;
                if (pw == 4) {
#pragma unroll 2
                    for (int j = 0; j < L.bcw; j += 4) {
                        const uint4 w = ld_shared_v4(wrow + 4u * j);
                        pop += __popc(w.x) + __popc(w.y) + __popc(w.z) + __popc(w.w);
                    }
                } else {
#pragma unroll 4
                    for (int j = 0; j < L.bcw; ++j) pop += __popc(ld_shared_b32(wrow + 4u * j));
                }
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * br), "r"(ld_shared_b32(par)) : "memory");
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * br + 8u), "r"(ld_shared_b32(par + 4u * rows1)) : "memory");
                if (SHIFTED) {
                    const float pd = (float)(int)ld_shared_b32(par + 8u * rows1);
                    asm volatile("st.shared.b32 [%0], %1;" ::"r"(pads + (uint32_t)(pi * P + br) * 8u + 4u * odd), "r"(__float_as_uint(pd)) : "memory");
                }
                store_const_row<false>(32 * L.bcw - 2 * pop, cexp + (uint32_t)((ct >> 2) * W_STAGE + col * ROWB), (col & 7) ^ (2 * (ct & 3)));
            }
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * P), "r"(ld_shared_b32(raw_slope + 4u * r)) : "memory");
            const uint16_t th = sign_threshold(__uint_as_float(ld_shared_b32(raw_nb + 4u * r)));
            asm volatile("st.shared.b16 [%0], %1;" ::"r"(ent + 16u * P + 8u - 2u * odd), "h"(th) : "memory");
        }
        fence_async_proxy();
        __syncwarp();
        if (lane == 0) mbar_arrive(ready_bar);
        asm volatile("bar.sync 1, %0;" ::"n"(ETHREADS) : "memory");
        // Lane 4 r + q works on the BN / 4 consecutive channels q and on the four rows quad * 32 + r + 8 i.
        const int team = (warp - FIRST_EPILOGUE) >> 2, quad = warp & 3, lq = lane & 3, row = quad * 32 + (lane >> 2);
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const bool want_bits = p.out != nullptr;
        // rows 8 apart lie at the same place of the swizzle
        const uint32_t sw = BN == 64 ? (uint32_t)(row & 7) : (uint32_t)((row >> 1) & 3);
        int s = 0, buf = team % L.nbuf;                                     // staging tile, accumulator buffer
        uint32_t phase = 0;
        Part part = {idx * BM, 0};
        part.skip(team, rs, tile_rows);
        bool ok;
#pragma unroll 1
        for (int n = team; n < parts; n += TEAMS, part.skip(TEAMS, rs, tile_rows)) {
            const int em = part.row + row, ch0 = ch_base + part.slice * BN;
            if (HAS_ID) ok = mbar_wait_warp(id_full(team, s), phase, abort_flag, p.err, ERR_MOD_IDENTITY);
            else ok = mbar_wait_warp(slot_free(team, s), phase ^ 1u, abort_flag, p.err, ERR_MOD_IDENTITY);
            if (!ok) break;
            uint32_t inside[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu};      // taps of these rows inside the image
            if (SHIFTED) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    RowCursor rc;
                    rc.m = (uint32_t)(em + 8 * i);
                    row_locate(p, rc);
                    row_window(p, L.ts, rc);
                    inside[i] = rc.mask;
                }
            }
            if (!mbar_wait_warp(tfull_bar(n % MAX_NBUF), (uint32_t)(n / MAX_NBUF) & 1u, abort_flag, p.err, ERR_MOD_EPILOGUE)) break;
            tc_fence_after();
            const uint32_t acc = t_lane + (uint32_t)(buf * P * BN);
            const uint32_t tile = stage_tile(team, s) + (uint32_t)(row * ROW_BYTES);
            const int sl = part.slice;
            const uint32_t tb = table + (uint32_t)(sl * 4 + lq) * share, pb = pads + (uint32_t)((sl * 4 + lq) * (BN / 8) * P) * 8u;
            // The branches are unrolled (P = 8, 64 channels at M = 50176 25.7 in a loop, 16.8 us), the four pairs of channels of a piece too where that is
            // little code: with them in a loop nine taps of 128 channels take 45.9 us instead of 54.7, thirteen branches of 64 30.5 instead of
            // 32.4, but eight of 64 17.6 instead of 16.8.
            // (two channels, branch) of four rows at a time; the next piece's accumulators and parameters are on their way while one is
            // worked on (a load and its wait in turn were a third of a part's time)
            uint32_t nv[8], sg[4] = {0u, 0u, 0u, 0u};                       // sg: even channels' bits in the low halves, odd ones' in the high
            tc_ld8_quads_nowait(acc, nv);
            uint4 nss = ld_shared_v4(tb);
#pragma unroll 1
            for (int k4 = 0; k4 < BN / 8; k4 += 4) {
                // a 16-byte piece of each row: eight channels
                const uint32_t at = tile + (((uint32_t)(BN / 32 * lq + k4 / 4) ^ sw) << 4);
                uint32_t io[4][4], sg4[4] = {0u, 0u, 0u, 0u};
                if (HAS_ID) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 q = ld_shared_v4(at + (uint32_t)(8 * i * ROW_BYTES));
                        io[i][0] = q.x; io[i][1] = q.y; io[i][2] = q.z; io[i][3] = q.w;
                    }
                }
#pragma unroll(ROLLED ? 1 : 4)
                for (int kk = 0; kk < 4; ++kk) {
                    const int k = k4 + kk;
                    unsigned long long t[4];
                    uint4 sn;
#pragma unroll
                    for (int b = 0; b < P; ++b) {
                        const bool last_branch = b == P - 1;
                        const uint4 ss = nss;                           // two channels' scales and shifts
                        tc_wait_ld();
                        pin_regs8(nv);
                        unsigned long long dot[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) dot[i] = bits2(nv[2 * i], nv[2 * i + 1]);
                        if (last_branch) sn = ld_shared_v4(tb + (uint32_t)k * pair + 16u * P);     // slopes, sign thresholds
                        if (k < BN / 8 - 1 || !last_branch) {
                            tc_ld8_quads_nowait(acc + (uint32_t)(last_branch ? (k + 1) * 8 : (b + 1) * BN + k * 8), nv);
                            nss = ld_shared_v4(tb + (last_branch ? (uint32_t)(k + 1) * pair : (uint32_t)k * pair + 16u * (b + 1)));
                        } else {                                        // the accumulators are in registers
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(tempty_bar(buf));
                        }
                        if (SHIFTED) {
                            unsigned long long pd;
                            asm volatile("ld.shared.b64 %0, [%1];" : "=l"(pd) : "r"(pb + (uint32_t)(k * P + b) * 8u) : "memory");
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (!((inside[i] >> b) & 1u)) dot[i] = pd;
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const unsigned long long tp = add2(mul2(dot[i], bits2(ss.x, ss.y)), bits2(ss.z, ss.w));
                            t[i] = b == 0 ? tp : add2(t[i], tp);
                        }
                    }
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        unsigned long long u = t[i];
                        if (HAS_ID) {
                            const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&io[i][ROLLED ? 0 : kk]));
                            u = add2(u, bits2(__float_as_uint(f.x), __float_as_uint(f.y)));
                        }
                        const float2 uf = floats2(u);
                        const __half2 y2 = __floats2half2_rn(prelu(uf.x, __uint_as_float(sn.x)), prelu(uf.y, __uint_as_float(sn.y)));
                        if (ROLLED) {
                            io[i][0] = io[i][1];
                            io[i][1] = io[i][2];
                            io[i][2] = io[i][3];
                        }
                        io[i][ROLLED ? 3 : kk] = *reinterpret_cast<const uint32_t *>(&y2);
                        if (want_bits) sg4[i] |= __hge2_mask(y2, *reinterpret_cast<const __half2 *>(&sn.z)) & (0x00020001u << (2 * kk));
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    st_shared_v4(at + (uint32_t)(8 * i * ROW_BYTES), io[i][0], io[i][1], io[i][2], io[i][3]);
                    sg[i] |= sg4[i] << (2 * k4);
                }
            }
            fence_async_proxy();                                            // the tile's generic stores -> the copy engine
            __syncwarp();
            if (lane == 0) mbar_arrive(out_full(team, s));
            if (want_bits && ch0 + lq * (BN / 4) < p.C_out) {
                const long pitch = p.C_out >> 3;
                uint8_t *dst = static_cast<uint8_t *>(p.out) + (long)em * pitch + ((ch0 + lq * (BN / 4)) >> 3);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t bits = sg[i] | (sg[i] >> 16);
                    if (em + 8 * i < p.M) {
                        if (BN == 64) *reinterpret_cast<uint16_t *>(dst + 8 * i * pitch) = (uint16_t)bits;
                        else dst[8 * i * pitch] = (uint8_t)bits;
                    }
                }
            }
            if (++s == NS) { s = 0; phase ^= 1u; }
            buf += TEAMS;
            while (buf >= L.nbuf) buf -= L.nbuf;
        }
    } else if (warp >= FIRST_PRODUCER) {
        // ------------------------------------------------------------------ producers: items grp, grp + G, ... of the (tile, stage) list
        const int ptid = tid - 32 * FIRST_PRODUCER, grp = ptid >> 7, quad = warp & 3, row = quad * 32 + lane;
        const uint32_t bits0 = bits_ring + (uint32_t)ptid * 16u, bits_end = bits0 + PF * SLOT_BYTES;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t st0 = lane_base + (uint32_t)(L.nbuf * P * BN);
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        const int total = my_tiles * kst;
        const TileStep &ts = L.ts;
        if (grp == 0) write_const_block(lane_base);
        RowCursor rc;
        rc.m = (uint32_t)idx * BM + (uint32_t)row;
        row_locate(p, rc);
        int l_k = grp, l_left = total > grp ? (total - grp + G - 1) / G : 0;
        while (l_k >= kst) { l_k -= kst; row_step(p, ts, rc); }
        row_window(p, ts, rc);
        uint32_t l_dst = bits0;
        auto issue = [&]() {
            const uint32_t at = tab + (uint32_t)l_k * (32u / (uint32_t)L.gw);
            if (L.gw == 4) gather_stage8<4>(p.x, rc, at, l_dst, HALF_BYTES);
            else if (L.gw == 2) gather_stage8<2>(p.x, rc, at, l_dst, HALF_BYTES);
            else gather_stage8<1>(p.x, rc, at, l_dst, HALF_BYTES);
            l_dst += SLOT_BYTES;
            if (l_dst == bits_end) l_dst = bits0;
            --l_left;
            l_k += G;
            if (l_k >= kst) {
                do { l_k -= kst; row_step(p, ts, rc); } while (l_k >= kst);
                row_window(p, ts, rc);
            }
        };
        pdl_wait();
#pragma unroll 1
        for (int i = 0; i < PF - 1; ++i) {
            if (l_left > 0) issue();
            cp_async_commit();
        }
        uint32_t c_src = bits0, phase = 1;            // first pass through the ring: slots are free
        int s = grp;
        while (s >= stages) { s -= stages; phase ^= 1u; }
#pragma unroll 1
        for (int it = grp; it < total; it += G) {
            if (l_left > 0) issue();
            cp_async_commit();
            cp_async_wait<PF - 1>();
            uint32_t v[32];
            expand_stage8(ld_shared_v4(c_src), ld_shared_v4(c_src + HALF_BYTES), v);
            c_src += SLOT_BYTES;
            if (c_src == bits_end) c_src = bits0;
            if (!mbar_wait_warp(empty_bar(s), phase, abort_flag, p.err, ERR_MOD_PRODUCER)) break;
            tc_fence_after();
            tc_st32(st0 + (uint32_t)s * 32u, v);
            tc_fence_before();
            __syncwarp();
            mbar_arrive_pred(full_bar(s), lane0);
            s += G;
            if (s >= stages) { s -= stages; phase ^= 1u; }
        }
        cp_async_wait<0>();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == ISSUER)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

// The plan for BN-channel slices, or false where the layer does not fit.
template <int BN>
bool make_plan(ModPlan &L, bool shifted, int &smem)
{
    const ConvProblem &q = L.q;
    L.kst = (L.P * L.kwp + 7) / 8;
    // as many accumulator buffers as leave ring slots for a row tile and the next one's start (at least one per producer group)
    const int want = L.kst + 1 < 3 ? 3 : (L.kst + 1 > 8 ? 8 : L.kst + 1);
    L.nbuf = MAX_NBUF;
    while (L.nbuf > 1 && (CB_COL - L.nbuf * L.P * BN) / 32 < (L.nbuf > 2 ? want : G)) --L.nbuf;
    const int stages = (CB_COL - L.nbuf * L.P * BN) / 32;
    if (stages < G) return false;
    L.stages = stages < MAX_STAGES ? stages : MAX_STAGES;
    L.slices = (q.C_out + BN - 1) / BN;
    L.units = L.kst * (8 / L.gw);
    exact_div_params((uint32_t)L.kwp, L.kwp_mul, L.kwp_shift);
    exact_div_params((uint32_t)(L.kwp / (L.gw == 4 ? 4 : 2)), L.row_mul, L.row_shift);
    const long slice_bytes = (long)L.kst * BN * ROWB, staging = (long)TEAMS * NS * BM * BN * 2;
    const int sms = sm_count();
    long best = -1;
    for (int rs = 1; rs <= L.slices && rs <= 16; ++rs) {
        if (rs > 1 && L.kst > L.stages) break;               // the row tile's stages stay in the ring for all its parts
        const long table = (long)rs * 4 * share_bytes<BN>(pair_bytes(L.P));
        const long pad = shifted ? (long)rs * (BN / 2) * L.P * 8 : 0, consts = (long)const_tiles(rs, L.P) * BN * ROWB;
        const long raw = (long)rs * BN * 4 * (L.P * (L.bcw + (shifted ? 3 : 2)) + 2);
        // the packed weights over the staging tiles but a team's first, or, where that is too much, over all of them: the first identity
        // tiles then wait too
        int early = TEAMS;
        auto bytes_of = [&]() {
            const long over = (long)early * BM * BN * 2 + raw, area = over > staging ? over : staging;
            return 1024 + rs * slice_bytes + consts + pad + area + (long)PF * SLOT_BYTES + table + 4L * L.units + 64;
        };
        if (bytes_of() > MAX_SMEM) early = 0;
        const long bytes = bytes_of();
        if (bytes > MAX_SMEM) break;
        const int ng = (L.slices + rs - 1) / rs, per = sms / ng;
        if (per < 1) continue;
        // parts on the longest CTA, and a little for a row tile's expansion
        const long tiles = (L.m_tiles + per - 1) / per, cost = tiles * (8L * rs + L.kst);
        if (best >= 0 && cost > best) continue;
        best = cost;
        L.rs = rs;
        L.ng = ng;
        L.off_const = (uint32_t)(rs * slice_bytes);
        L.off_stage = L.off_const + (uint32_t)consts;
        L.early_tiles = early;
        L.off_raw = L.off_stage + (uint32_t)(early * BM * BN * 2);
        L.off_bits = L.off_raw + (uint32_t)raw;
        if (L.off_bits < L.off_stage + (uint32_t)staging) L.off_bits = L.off_stage + (uint32_t)staging;
        L.off_table = L.off_bits + (uint32_t)PF * SLOT_BYTES;
        L.off_pad = L.off_table + (uint32_t)table;
        L.off_tab = (L.off_pad + (uint32_t)pad + 15u) & ~15u;
        smem = (int)bytes;
    }
    return best >= 0;
}

template <int BN, int PP, bool SHIFTED>
int launch_plan(ModPlan &L, int smem, cudaStream_t stream)
{
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return BCNN_ERR_CUDA;
    const ConvProblem &q = L.q;
    const cuuint64_t dims[2] = {(cuuint64_t)q.C_out, (cuuint64_t)q.M}, strides[1] = {(cuuint64_t)q.C_out * 2};
    const cuuint32_t box[2] = {BN, BM}, estr[2] = {1, 1};
    CUtensorMap map[2];
    for (int i = 0; i < 2; ++i) {
        void *ptr = i || !q.identity ? static_cast<void *>(q.y_real) : const_cast<uint16_t *>(q.identity);
        if (encode(&map[i], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, ptr, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   BN == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return BCNN_ERR_CUDA;
    }
    auto k = q.identity ? conv_tc_mod_kernel<BN, PP, SHIFTED, true> : conv_tc_mod_kernel<BN, PP, SHIFTED, false>;
    if (!allow_smem((const void *)k, MAX_SMEM)) return BCNN_ERR_CUDA;
    int per = sm_count() / L.ng;
    if (per > L.m_tiles) per = L.m_tiles;
    L.step = per;
    exact_div_params((uint32_t)L.ng, L.ng_mul, L.ng_shift);
    exact_div_params((uint32_t)per, L.step_mul, L.step_shift);
    L.ts = make_tile_step(q, (uint32_t)(BM * per));
    if (smem < 120 * 1024) smem = 120 * 1024;                // one CTA per multiprocessor (it takes all of tensor memory)
    return launch(k, (unsigned)(per * L.ng), THREADS, smem, stream, L, map[0], map[1]);
}

// Channels of a part (64, 32) with the plan for them, or 0 where the layer is not this engine's.
int plan_mod(ModPlan &L, bool shifted, int &smem)
{
    const ConvProblem &q = L.q;
    L.kwp = (L.bcw + 1) & ~1;
    L.gw = L.bcw % 4 == 0 ? 4 : (L.bcw % 2 == 0 ? 2 : 1);
    if (L.P > 13 || (shifted && L.P != 9) || q.C_out % 32 != 0 || q.M < 1) return 0;          // (odd squares up to 13: 9)
    if ((long)q.B * q.H * q.W * q.cw >= (1L << 31) || (long)q.kh * q.W * q.cw >= (1L << 27) || 32L * L.bcw > CONST_MAX) return 0;
    L.m_tiles = (q.M - 1) / BM + 1;
    // 64-channel parts; 32 where that leaves a multiprocessor less than two parts (a part is 2 us of latency per 64 channels)
    if (L.P <= 3 && !shifted && q.C_out > 32 && (long)L.m_tiles * ((q.C_out + 63) / 64) > sm_count() && make_plan<64>(L, shifted, smem)) return 64;
    return make_plan<32>(L, shifted, smem) ? 32 : 0;
}

int launch_mod(ModPlan &L, bool shifted, cudaStream_t stream)
{
    int smem = 0;
    const int width = plan_mod(L, shifted, smem);
    if (width == 0) return BCNN_ERR_UNSUPPORTED;
    L.q.err = device_error_word();
    if (width == 64) {
        if (L.P == 1) return launch_plan<64, 1, false>(L, smem, stream);
        if (L.P == 2) return launch_plan<64, 2, false>(L, smem, stream);
        return launch_plan<64, 3, false>(L, smem, stream);
    }
    if (shifted) return launch_plan<32, 9, true>(L, smem, stream);
    switch (L.P) {
    case 1: return launch_plan<32, 1, false>(L, smem, stream);
    case 2: return launch_plan<32, 2, false>(L, smem, stream);
    case 3: return launch_plan<32, 3, false>(L, smem, stream);
    case 4: return launch_plan<32, 4, false>(L, smem, stream);
    case 5: return launch_plan<32, 5, false>(L, smem, stream);
    case 6: return launch_plan<32, 6, false>(L, smem, stream);
    case 7: return launch_plan<32, 7, false>(L, smem, stream);
    case 8: return launch_plan<32, 8, false>(L, smem, stream);
    case 9: return launch_plan<32, 9, false>(L, smem, stream);
    case 10: return launch_plan<32, 10, false>(L, smem, stream);
    case 11: return launch_plan<32, 11, false>(L, smem, stream);
    case 12: return launch_plan<32, 12, false>(L, smem, stream);
    default: return launch_plan<32, 13, false>(L, smem, stream);
    }
}

}  // namespace

// One branch: a pointwise layer's module (mode 2 problem).
int launch_conv_tc_mod(const ConvProblem &p, cudaStream_t stream)
{
    if (p.mode != 2 || p.kh != 1 || p.kw != 1 || p.stride != 1 || p.pad != 0) return BCNN_ERR_UNSUPPORTED;
    ModPlan L = {};
    L.q = p;
    L.scale = p.bn_scale;
    L.shift = p.bn_shift;
    L.P = 1;
    L.bcw = p.cw;
    return launch_mod(L, false, stream);
}

// The module engine's view of a branch module; false for a window it does not take.
static bool branch_plan(const BranchProblem &b, ModPlan &L, bool &shifted)
{
    shifted = b.kh * b.kw > 1;
    if ((shifted && b.kh != b.kw) || b.M >= (1L << 31) || b.H >= (1 << 30) || b.P * (long)b.cw >= (1L << 20)) return false;
    L = {};
    ConvProblem &q = L.q;
    q.x = b.x; q.w = b.w; q.out = b.y_bits;
    q.B = b.B; q.H = b.H; q.W = b.W; q.C_in = b.C_in; q.C_out = b.C_out;
    q.kh = b.kh; q.kw = b.kw; q.stride = 1; q.pad = (b.kh - 1) / 2; q.OH = b.H; q.OW = b.W;
    q.cw = b.P * b.cw;
    q.M = (int)b.M;
    q.slope = b.slope; q.next_bias = b.next_bias; q.identity = b.identity; q.y_real = b.y_real;
    exact_div_params((uint32_t)b.W, q.ow_mul, q.ow_shift);
    exact_div_params((uint32_t)((long)b.H * b.W), q.ohw_mul, q.ohw_shift);
    L.scale = b.bn_scale; L.shift = b.bn_shift; L.pad_dot = b.pad_dot;
    L.P = b.P;
    L.bcw = b.cw;
    return true;
}

int launch_branches_tc_mod(const BranchProblem &b, cudaStream_t stream)
{
    ModPlan L;
    bool shifted;
    return branch_plan(b, L, shifted) ? launch_mod(L, shifted, stream) : BCNN_ERR_UNSUPPORTED;
}

// Channels of a part (0: not this engine's), resident slices, stages of a row, ring slots, staging tiles ahead of the packed weights.
void branches_tc_mod_plan(const BranchProblem &b, int (&plan)[5])
{
    ModPlan L;
    bool shifted;
    int smem = 0;
    plan[0] = branch_plan(b, L, shifted) ? plan_mod(L, shifted, smem) : 0;
    plan[1] = plan[0] ? L.rs : 0;
    plan[2] = plan[0] ? L.kst : 0;
    plan[3] = plan[0] ? L.stages : 0;
    plan[4] = plan[0] ? L.early_tiles : 0;
}

}  // namespace bcnn
