// Convolution module on pointwise layers (Section 4.2.1, Figure 4): P >= 1 binary branches on the tensor cores, then per
// branch batch norm, the branch sum, + identity, PReLU, fp16 map and the next module's signs, in one pass.  P = kh * kw
// shifted branches (the stand-in for a binary kh x kw convolution) run here too.
//
// Bound by the fp16 maps' traffic (2 bytes of identity read and 2 bytes written per output) as long as the epilogue
// spends less than about 20 instructions per output, so everything is built around the epilogue:
//   * identity tiles arrive and output tiles leave by tiled TMA copies of 128 rows x BN channels through a ring of NS tiles per
//     epilogue team in shared memory (swizzled: one 16-byte access per lane and row without bank conflicts); a loader warp and a
//     store warp issue them (an issue costs its warp some 500 cycles), the epilogue turns a tile in place;
//   * per-channel values lie in shared memory as pairs of channels, read as 16-byte broadcasts - four cycles of the shared-memory
//     pipe each, the epilogue's scarcest resource: one per branch {scale, shift} and one {slope, next bias}.  The constant
//     K - 2 popc of a dot product is not among them, an MMA against a constant tile puts it into the accumulator
//     (tc_slot.cuh);
//   * the arithmetic runs on pairs (f32x2: the same IEEE operations, half the issue slots);
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
    int m_tiles;
    int units, gw;            // gather units of a row
    uint32_t off_bits, off_stage, off_table, off_pad, off_pop, off_tab, off_const;      // shared-memory offsets from the 1024-byte aligned base (weights first)
};

// per-channel-pair table of a slice: P entries of 16 bytes {scale, shift} x 2, then 16 bytes {slope, next bias} x 2
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
__device__ __forceinline__ void tc_ld8_nowait(uint32_t taddr, uint32_t (&v)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void pin_regs8(uint32_t (&v)[8])
{
    asm volatile("" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]) :: "memory");
}

// BN: channels of a part (64, 32); PP: branches where known to the compiler (1, 2), else 0; SHIFTED: taps with a row mask
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
    const int P = PP ? PP : L.P;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int kst = L.kst, stages = L.stages;
    const int cg = (int)blockIdx.x % L.ng, idx = (int)blockIdx.x / L.ng, step = (int)gridDim.x / L.ng;
    const int rs = min(L.rs, L.slices - cg * L.rs);
    const int my_tiles = idx < L.m_tiles ? (L.m_tiles - 1 - idx) / step + 1 : 0;
    const int parts = my_tiles * rs;
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;         // [rs][kst][BN rows][128 B] weights, then the rest
    const uint32_t bits_ring = base + L.off_bits, staging = base + L.off_stage, table = base + L.off_table, pops = base + L.off_pop;
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

    if (tid == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(full_bar(s), 4);
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < MAX_NBUF; ++b) {
            mbar_init(tfull_bar(b), 1);
            mbar_init(tempty_bar(b), 4);
        }
        for (int t = 0; t < TEAMS; ++t) {
            for (int s = 0; s < NS; ++s) {
                mbar_init(id_full(t, s), 1);
                mbar_init(slot_free(t, s), 1);
                mbar_init(out_full(t, s), 4);
            }
        }
        mbar_init(ready_bar, 4 * TEAMS);
        abort_flag_smem = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == ISSUER) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // gather table: unit u = K words u * gw ..; word w belongs to branch w / kwp (its tap when shifted)
    for (int u = tid; u < L.units; u += THREADS) {
        const int w = u * L.gw, br = w / L.kwp, j = w - br * L.kwp;
        uint32_t ent = (uint32_t)TAP_NONE << 27;
        if (br < P && j < L.bcw) {
            const int r = br / p.kw, t = br - r * p.kw;
            ent = (uint32_t)((SHIFTED ? (r * p.W + t) * p.cw : 0) + br * L.bcw + j) | ((uint32_t)(SHIFTED ? br : 0) << 27);
        }
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(tab + 4u * u), "r"(ent) : "memory");
    }
    const int npop = rs * P * BN;
    for (int i = tid; i < npop; i += THREADS) asm volatile("st.shared.b32 [%0], %1;" ::"r"(pops + 4u * i), "r"(0) : "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    pdl_trigger();
    pdl_wait();
    const uint32_t tmem_base = tmem_base_smem;

    // part n = (row tile n / rs, slice n % rs); team n % TEAMS, its m = n / TEAMS-th part, staging tile m % NS
    auto part_row = [&](int n) { return (idx + (n / rs) * step) * BM; };
    auto part_ch = [&](int n) { return (cg * L.rs + n % rs) * BN; };

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
            int issued = 0;
            for (int n = 0; n < parts; ++n, ++issued) {
                const int team = n % TEAMS, m = n / TEAMS, s = m % NS, lap = m / NS;
                if (lap > 0 && !mbar_wait_warp(slot_free(team, s), (uint32_t)(lap - 1) & 1u, abort_flag, p.err, ERR_MOD_LOADER)) break;
                if (lane == 0) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(id_full(team, s)), "r"((uint32_t)TILE_BYTES) : "memory");
                    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                                 ::"r"(staging + (uint32_t)((team * NS + s) * TILE_BYTES)), "l"(reinterpret_cast<uint64_t>(&idmap)), "r"(part_ch(n)), "r"(part_row(n)),
                                   "r"(id_full(team, s)) : "memory");
                }
                __syncwarp();
            }
            // after a time-out elsewhere: copies still in flight must land before the CTA's shared memory goes away
            if (*abort_flag)
                for (int n = issued > TEAMS * NS ? issued - TEAMS * NS : 0; n < issued; ++n)
                    mbar_wait_warp(id_full(n % TEAMS, (n / TEAMS) % NS), (uint32_t)(n / TEAMS / NS) & 1u, abort_flag, nullptr, 0);
        }
    } else if (warp < FIRST_PRODUCER) {
        // ------------------------------------------------------------------ output tiles of team warp - STORER
        const int team = warp - STORER;
        for (int n = team; n < parts; n += TEAMS) {
            const int m = n / TEAMS, s = m % NS;
            if (!mbar_wait_warp(out_full(team, s), (uint32_t)(m / NS) & 1u, abort_flag, p.err, ERR_MOD_STORE)) break;
            if (lane == 0) {
                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                             ::"l"(reinterpret_cast<uint64_t>(&ymap)), "r"(part_ch(n)), "r"(part_row(n)), "r"(staging + (uint32_t)((team * NS + s) * TILE_BYTES)) : "memory");
                asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                if (m > 0) {                                                // the store before this one has read its tile
                    asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                    mbar_arrive(slot_free(team, (m - 1) % NS));
                }
            }
            __syncwarp();
        }
        if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
    } else if (warp >= FIRST_EPILOGUE) {
        // ------------------------------------------------------------------ epilogue
        // ---- one-off, while the first rows and identity tiles arrive: the resident slices' weights (the issuer waits for them)
        // with their bit counts, then the table.  Eight words are in flight per thread, and a channel's parameters before them.
        constexpr int ETHREADS = 128 * TEAMS;
        const int etid = tid - 32 * FIRST_EPILOGUE;
        // parameters of a (slice, branch, channel) triple
        struct Params { float sc, sh, pd, slope, nb; };
        auto load_params = [&](int i) {
            const int c = i % BN, sb = i / BN, br = sb % P, ch = (cg * L.rs + sb / P) * BN + c;
            const bool have = i < rs * P * BN && ch < p.C_out;
            const long at = (long)br * p.C_out + ch;
            Params q;
            q.sc = have ? __ldg(L.scale + at) : 0.f;
            q.sh = have ? __ldg(L.shift + at) : 0.f;
            q.pd = SHIFTED && have && L.pad_dot ? (float)__ldg(L.pad_dot + at) : 0.f;
            q.slope = br == 0 && have ? __ldg(p.slope + ch) : 0.f;
            q.nb = br == 0 && have && p.next_bias ? __ldg(p.next_bias + ch) : 0.f;
            return q;
        };
        Params q = load_params(etid);
        {
            constexpr int WU = 8;
            const int total = rs * kst * BN * 8;
            for (int i0 = etid; i0 < total; i0 += WU * ETHREADS) {
                uint32_t w[WU];
                bool live[WU];
                int pop_at[WU];
                uint32_t dst[WU];
#pragma unroll
                for (int u = 0; u < WU; ++u) {
                    const int i = i0 + u * ETHREADS, e = i & 7, rk = i >> 3, row_s = rk / kst, kt = rk - row_s * kst;     // row_s = slice * BN + row
                    const int sl = row_s / BN, row = row_s % BN, ch = (cg * L.rs + sl) * BN + row;
                    const int kw = kt * 8 + e, br = kw / L.kwp, j = kw - br * L.kwp;
                    live[u] = i < total && br < P && j < L.bcw && ch < p.C_out;
                    w[u] = live[u] ? __ldg(p.w + ((long)br * p.C_out + ch) * L.bcw + j) : 0u;
                    pop_at[u] = (sl * P + br) * BN + row;
                    dst[u] = base + (uint32_t)((sl * kst + kt) * W_STAGE + row * ROWB + ((e ^ (row & 7)) << 4));
                }
#pragma unroll
                for (int u = 0; u < WU; ++u) {
                    if (i0 + u * ETHREADS >= total) break;
                    const uint4 o = live[u] ? expand_w4(w[u]) : make_uint4(0u, 0u, 0u, 0u);
                    st_shared_v4(dst[u], o.x, o.y, o.z, o.w);
                    if (live[u]) asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(pops + 4u * pop_at[u]), "r"(__popc(w[u])) : "memory");
                }
            }
        }
        asm volatile("bar.sync 1, %0;" ::"n"(ETHREADS) : "memory");
        for (int i = etid; i < rs * P * BN; i += ETHREADS) {                // (slice, branch, channel)
            const int c = i % BN, sb = i / BN, br = sb % P, sl = sb / P;
            if (i != etid) q = load_params(i);
            int pop;
            asm volatile("ld.shared.b32 %0, [%1];" : "=r"(pop) : "r"(pops + 4u * i) : "memory");
            const uint32_t pair = (uint32_t)((sl * BN + c) >> 1), odd = 4u * (c & 1), ent = table + pair * pair_bytes(P) + odd;
            const int ct = sl * P + br;
            store_const_row<false>(32 * L.bcw - 2 * pop, cexp + (uint32_t)((ct >> 2) * W_STAGE + c * ROWB), (c & 7) ^ (2 * (ct & 3)));
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * br), "r"(__float_as_uint(q.sc)) : "memory");
            asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * br + 8u), "r"(__float_as_uint(q.sh)) : "memory");
            if (SHIFTED) asm volatile("st.shared.b32 [%0], %1;" ::"r"(pads + (pair * P + br) * 8u + odd), "r"(__float_as_uint(q.pd)) : "memory");
            if (br == 0) {
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * P), "r"(__float_as_uint(q.slope)) : "memory");
                asm volatile("st.shared.b32 [%0], %1;" ::"r"(ent + 16u * P + 8u), "r"(__float_as_uint(q.nb)) : "memory");
            }
        }
        fence_async_proxy();
        __syncwarp();
        if (lane == 0) mbar_arrive(ready_bar);
        asm volatile("bar.sync 1, %0;" ::"n"(ETHREADS) : "memory");
        const int team = (warp - FIRST_EPILOGUE) >> 2, quad = warp & 3, row = quad * 32 + lane;
        const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
        const int owords = p.C_out >> 5;
        const bool want_bits = p.out != nullptr;
        const TileStep ts = make_tile_step(p, 0);
        bool ok = true;
        for (int n = team; n < parts; n += TEAMS) {
            const int m = n / TEAMS, s = m % NS, lap = m / NS;
            const int em = part_row(n) + row, ch0 = part_ch(n);
            if (HAS_ID) ok = mbar_wait_warp(id_full(team, s), (uint32_t)lap & 1u, abort_flag, p.err, ERR_MOD_IDENTITY);
            else if (lap > 0) ok = mbar_wait_warp(slot_free(team, s), (uint32_t)(lap - 1) & 1u, abort_flag, p.err, ERR_MOD_IDENTITY);
            if (!ok) break;
            uint32_t inside = 0xffffffffu;                                  // taps of this row inside the image
            if (SHIFTED) {
                RowCursor rc;
                rc.m = (uint32_t)em;
                row_locate(p, rc);
                row_window(p, ts, rc);
                inside = rc.mask;
            }
            if (!mbar_wait_warp(tfull_bar(n % MAX_NBUF), (uint32_t)(n / MAX_NBUF) & 1u, abort_flag, p.err, ERR_MOD_EPILOGUE)) break;
            tc_fence_after();
            const uint32_t acc = t_lane + (uint32_t)((n % L.nbuf) * P * BN);
            const uint32_t tile = staging + (uint32_t)((team * NS + s) * TILE_BYTES) + (uint32_t)(row * ROW_BYTES);
            const uint32_t sw = BN == 64 ? (uint32_t)(row & 7) : (uint32_t)((row >> 1) & 3);
            const uint32_t tb = table + (uint32_t)((n % rs) * (BN / 2)) * pair_bytes(P), pb = pads + (uint32_t)((n % rs) * (BN / 2) * P) * 8u;
            uint32_t words[BN / 32];
            // (8 channels, branch) at a time; the next piece's accumulators are on their way while one is worked on (a load and
            // its wait in turn were a third of a part's time)
            uint32_t nv[8];
            tc_ld8_nowait(acc, nv);
#pragma unroll
            for (int c8 = 0; c8 < BN / 8; ++c8) {
                unsigned long long t[4];
#pragma unroll
                for (int br = 0; br < (PP ? PP : 1); ++br) {
                    int b = br;
                    do {
                        tc_wait_ld();
                        pin_regs8(nv);
                        unsigned long long dot[4];
#pragma unroll
                        for (int j = 0; j < 4; ++j) dot[j] = bits2(nv[2 * j], nv[2 * j + 1]);
                        const bool last_branch = b == P - 1;
                        if (c8 < BN / 8 - 1 || !last_branch) {
                            tc_ld8_nowait(acc + (uint32_t)(last_branch ? (c8 + 1) * 8 : (b + 1) * BN + c8 * 8), nv);
                        } else {                                            // the accumulators are in registers
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(tempty_bar(n % L.nbuf));
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const uint4 ss = ld_shared_v4(tb + (uint32_t)(c8 * 4 + j) * pair_bytes(P) + 16u * b);
                            if (SHIFTED && !((inside >> b) & 1u))
                                asm volatile("ld.shared.b64 %0, [%1];" : "=l"(dot[j]) : "r"(pb + (uint32_t)((c8 * 4 + j) * P + b) * 8u) : "memory");
                            const unsigned long long tp = add2(mul2(dot[j], bits2(ss.x, ss.y)), bits2(ss.z, ss.w));
                            t[j] = b == 0 ? tp : add2(t[j], tp);
                        }
                    } while (!PP && ++b < P);
                }
                const uint32_t at = tile + (((uint32_t)c8 ^ sw) << 4);
                uint32_t idw[4] = {0u, 0u, 0u, 0u}, ow[4], bits = 0;
                if (HAS_ID) {
                    const uint4 q = ld_shared_v4(at);
                    idw[0] = q.x; idw[1] = q.y; idw[2] = q.z; idw[3] = q.w;
                }
                float2 yf[4];
                uint4 sn[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    sn[j] = ld_shared_v4(tb + (uint32_t)(c8 * 4 + j) * pair_bytes(P) + 16u * P);               // slope, next bias
                    unsigned long long u = t[j];
                    if (HAS_ID) {
                        const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&idw[j]));
                        u = add2(u, bits2(__float_as_uint(f.x), __float_as_uint(f.y)));
                    }
                    const float2 uf = floats2(u), wf = floats2(mul2(bits2(sn[j].x, sn[j].y), u));
                    const __half2 y2 = __floats2half2_rn(uf.x >= 0.f ? uf.x : wf.x, uf.y >= 0.f ? uf.y : wf.y);
                    ow[j] = *reinterpret_cast<const uint32_t *>(&y2);
                    yf[j] = __half22float2(y2);
                }
                st_shared_v4(at, ow[0], ow[1], ow[2], ow[3]);
                if (want_bits) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float2 v = floats2(add2(bits2(__float_as_uint(yf[j].x), __float_as_uint(yf[j].y)), bits2(sn[j].z, sn[j].w)));
                        bits |= (v.x >= 0.f ? 1u : 0u) << (2 * j);
                        bits |= (v.y >= 0.f ? 1u : 0u) << (2 * j + 1);
                    }
                }
                if (c8 & 3) words[c8 >> 2] |= bits << (8 * (c8 & 3));
                else words[c8 >> 2] = bits;
            }
            fence_async_proxy();                                            // the tile's generic stores -> the copy engine
            __syncwarp();
            if (lane == 0) mbar_arrive(out_full(team, s));
            if (p.out && em < p.M) {
                uint32_t *dst = static_cast<uint32_t *>(p.out) + (long)em * owords + (ch0 >> 5);
                if (BN == 64 && (owords & 1) == 0) {
                    *reinterpret_cast<uint2 *>(dst) = make_uint2(words[0], words[BN / 32 - 1]);
                } else {
#pragma unroll
                    for (int k = 0; k < BN / 32; ++k)
                        if ((ch0 >> 5) + k < owords) dst[k] = words[k];
                }
            }
        }
    } else if (warp >= FIRST_PRODUCER) {
        // ------------------------------------------------------------------ producers: items grp, grp + G, ... of the (tile, stage) list
        const int ptid = tid - 32 * FIRST_PRODUCER, grp = ptid >> 7, quad = warp & 3, row = quad * 32 + lane;
        const uint32_t bits0 = bits_ring + (uint32_t)ptid * 16u, bits_end = bits0 + PF * SLOT_BYTES;
        const uint32_t lane_base = tmem_base + ((uint32_t)(quad * 32) << 16);
        const uint32_t st0 = lane_base + (uint32_t)(L.nbuf * P * BN);
        const uint32_t lane0 = lane == 0 ? 1u : 0u;
        const int total = my_tiles * kst;
        const TileStep ts = make_tile_step(p, (uint32_t)(BM * step));
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
    const long slice_bytes = (long)L.kst * BN * ROWB, staging = (long)TEAMS * NS * BM * BN * 2;
    const int sms = sm_count();
    long best = -1;
    for (int rs = 1; rs <= L.slices && rs <= 16; ++rs) {
        if (rs > 1 && L.kst > L.stages) break;               // the row tile's stages stay in the ring for all its parts
        const long pops = (long)rs * L.P * BN * 4, table = (long)rs * (BN / 2) * pair_bytes(L.P);
        const long pad = shifted ? (long)rs * (BN / 2) * L.P * 8 : 0, consts = (long)const_tiles(rs, L.P) * BN * ROWB;
        const long bytes = 1024 + rs * slice_bytes + consts + pad + staging + pops + (long)PF * SLOT_BYTES + table + 4L * L.units + 64;
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
        L.off_pop = L.off_stage + (uint32_t)staging;
        L.off_bits = L.off_pop + (uint32_t)pops;
        L.off_table = L.off_bits + (uint32_t)PF * SLOT_BYTES;
        L.off_pad = L.off_table + (uint32_t)table;
        L.off_tab = (L.off_pad + (uint32_t)pad + 15u) & ~15u;
        smem = (int)bytes;
    }
    return best >= 0;
}

template <int BN, int PP, bool SHIFTED>
int launch_plan(const ModPlan &L, int smem, cudaStream_t stream)
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
    if (smem < 120 * 1024) smem = 120 * 1024;                // one CTA per multiprocessor (it takes all of tensor memory)
    return launch(k, (unsigned)(per * L.ng), THREADS, smem, stream, L, map[0], map[1]);
}

int launch_mod(ModPlan &L, bool shifted, cudaStream_t stream)
{
    ConvProblem &q = L.q;
    L.kwp = (L.bcw + 1) & ~1;
    L.gw = L.bcw % 4 == 0 ? 4 : (L.bcw % 2 == 0 ? 2 : 1);
    q.err = device_error_word();
    if (L.P > 13 || q.C_out % 32 != 0 || q.M < 1) return BCNN_ERR_UNSUPPORTED;
    if ((long)q.B * q.H * q.W * q.cw >= (1L << 31) || (long)q.kh * q.W * q.cw >= (1L << 27) || 32L * L.bcw > CONST_MAX) return BCNN_ERR_UNSUPPORTED;
    L.m_tiles = (q.M - 1) / BM + 1;
    int smem = 0;
    // 64-channel parts; 32 where that leaves a multiprocessor less than two parts (a part is 2 us of latency per 64 channels)
    if (L.P <= 3 && q.C_out > 32 && (long)L.m_tiles * ((q.C_out + 63) / 64) > sm_count() && make_plan<64>(L, shifted, smem)) {
        if (shifted) return launch_plan<64, 0, true>(L, smem, stream);
        if (L.P == 1) return launch_plan<64, 1, false>(L, smem, stream);
        if (L.P == 2) return launch_plan<64, 2, false>(L, smem, stream);
        return launch_plan<64, 0, false>(L, smem, stream);
    }
    if (make_plan<32>(L, shifted, smem)) {
        if (shifted) return launch_plan<32, 0, true>(L, smem, stream);
        if (L.P == 1) return launch_plan<32, 1, false>(L, smem, stream);
        if (L.P == 2) return launch_plan<32, 2, false>(L, smem, stream);
        return launch_plan<32, 0, false>(L, smem, stream);
    }
    return BCNN_ERR_UNSUPPORTED;
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

int launch_branches_tc_mod(const BranchProblem &b, cudaStream_t stream)
{
    const bool shifted = b.kh * b.kw > 1;
    if ((shifted && b.kh != b.kw) || b.M >= (1L << 31) || b.H >= (1 << 30) || b.P * (long)b.cw >= (1L << 20)) return BCNN_ERR_UNSUPPORTED;
    ModPlan L = {};
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
    return launch_mod(L, shifted, stream);
}

}  // namespace bcnn
