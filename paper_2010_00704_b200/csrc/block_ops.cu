// The real-valued vector operations of the paper's building block and head: the 3x3 convolution module (real depth-
// wise 3x3 convolution, batch norm, PReLU; Section 4.2.1), S x S / S average pooling on the identity path of a down-
// sampling block (Section 4.2.3), channel replication as indexing (Section 4.2.2: channel c reads channel c mod C_in,
// no copy), global average pooling and the fully connected layer (Section 4.1).  All of them are bound by the memory
// traffic of the fp16 NHWC maps: a thread handles 8 consecutive channels (16 bytes) of one output pixel, arithmetic in
// fp32.  The depth-wise module can also emit the next binary module's sign bits (bias + sign of the stored value), so
// that the map is not read again by a pack pass.
#include "tc_common.cuh"
#include "tensor_map.cuh"
#include <cuda_fp16.h>
#include <climits>

namespace bcnn {

namespace {

__device__ __forceinline__ void unpack8(const uint4 &v, float (&f)[8])
{
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&w[q]));
        f[2 * q] = a.x;
        f[2 * q + 1] = a.y;
    }
}

// ---- depth-wise 3x3, stride 1 or 2 --------------------------------------------------------------------------------
// Bound by the fp16 maps' traffic once everything else is out of the way.  A CTA owns CB channels (32 or 64) and walks
// tiles of 8 x TW output pixels; a tile's input halo arrives by one tiled TMA copy (4D box, out-of-image = zero fill = the
// padding) into one of two buffers, the next tile's while this one is computed.  A thread owns four channels - weights and
// per-channel values in registers for the CTA's life - and slides along a strip of L = TW / 2 pixels of two output rows:
// every input column is read and converted once for both rows (4 or 5 8-byte shared loads at immediate offsets).  Per output
// value: nine multiply-adds in the fixed order (r, t), two at a time (f32x2: the same two IEEE operations, half the issue
// slots).  The kernel before this one kept one output pixel per thread and read 13 per-channel vectors from shared memory
// for each - 26 16-byte shared loads per 16 bytes of output, 0.7 TB/s at stride 1 (maps read + written once).
struct F4 { unsigned long long lo, hi; };                  // four fp32 values as two f32x2 pairs

__device__ __forceinline__ unsigned long long pack2(float a, float b)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c)
{
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ F4 to_f4(const uint2 &v)
{
    const float2 a = __half22float2(*reinterpret_cast<const __half2 *>(&v.x)), b = __half22float2(*reinterpret_cast<const __half2 *>(&v.y));
    return {pack2(a.x, a.y), pack2(b.x, b.y)};
}

constexpr int DW_TH = 8, DW_NR = 2, DW_STRIPS = DW_TH;        // strips of a tile: TH / NR row pairs x two segments
constexpr int ERR_DW_TIMEOUT = 161;

// S: stride; TW: output columns of a tile; CB: channels of a CTA
template <int S, int TW, int CB> struct DwCfg {
    static constexpr int L = TW / 2;
    static constexpr int HB = (DW_TH - 1) * S + 3, WB = (TW - 1) * S + 3;      // halo: rows, pixels
    static constexpr int G = CB / 4, THREADS = DW_STRIPS * G;
    static constexpr int BYTES = HB * WB * CB * 2, BUF = (BYTES + 127) / 128 * 128;     // a copy's bytes; buffers on 128-byte boundaries
    static constexpr int SMEM = 2 * BUF + 128;
};

template <int S, int TW, int CB, bool BITS>
__global__ void __launch_bounds__(DwCfg<S, TW, CB>::THREADS, 512 / DwCfg<S, TW, CB>::THREADS)
dw_tile_kernel(const __grid_constant__ CUtensorMap xmap, const float *w, const float *scale, const float *shift, const float *slope,
               const float *next_bias, uint16_t *y, uint8_t *y_bits, int C_in, int C, int OH, int OW,
               unsigned tiles_x, unsigned tiles_y, unsigned tiles, unsigned cblocks, int *err)
{
    using D = DwCfg<S, TW, CB>;
    constexpr int ROWS = (DW_NR - 1) * S + 3;                  // input rows of a strip: 4 or 5
    extern __shared__ unsigned char dw_raw[];
    __shared__ __align__(8) unsigned long long full[2];
    __shared__ int abort_flag;
    const unsigned tid = threadIdx.x, cb = blockIdx.x % cblocks, step = gridDim.x / cblocks;
    const uint32_t buf0 = (tc::smem_u32(dw_raw) + 127u) & ~127u, bar0 = tc::smem_u32(full);
    if (tid == 0) {
        tc::mbar_init(bar0, 1);
        tc::mbar_init(bar0 + 8, 1);
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const unsigned g = tid % D::G, st = tid / D::G;
    const int c0 = (int)cb * CB + 4 * (int)g;                  // first output channel; it reads channel c mod C_in
    const bool have = c0 < C;
    const int rp = (int)(st >> 1), sg = (int)(st & 1);
    pdl_wait();
    auto tile_at = [&](unsigned t, unsigned &b, int &oh0, int &ow0) {
        const unsigned per = tiles_x * tiles_y;
        b = t / per;
        const unsigned rem = t - b * per, ty = rem / tiles_x;
        oh0 = (int)ty * DW_TH;
        ow0 = (int)(rem - ty * tiles_x) * TW;
    };
    auto issue = [&](unsigned t, unsigned which) {              // one thread
        unsigned b;
        int oh0, ow0;
        tile_at(t, b, oh0, ow0);
        const uint32_t bar = bar0 + 8u * which;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)D::BYTES) : "memory");
        asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                     ::"r"(buf0 + which * (uint32_t)D::BUF), "l"(reinterpret_cast<uint64_t>(&xmap)), "r"((int)(cb * CB) % C_in), "r"(ow0 * S - 1),
                       "r"(oh0 * S - 1), "r"((int)b), "r"(bar) : "memory");
    };
    const unsigned first = blockIdx.x / cblocks;
    if (tid == 0) {
        if (first < tiles) issue(first, 0);
        if (first + step < tiles) issue(first + step, 1);
    }
    // weights of the four channels: 36 consecutive floats [c][9]
    F4 wt[9], sc, sh;
    float sl[4], nb[4];
    {
        float f[36];
        const int cw = have ? c0 : 0;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(w + (long)cw * 9) + i);
            f[4 * i] = v.x; f[4 * i + 1] = v.y; f[4 * i + 2] = v.z; f[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) wt[i] = {pack2(f[i], f[9 + i]), pack2(f[18 + i], f[27 + i])};
        const float4 a = __ldg(reinterpret_cast<const float4 *>(scale + cw)), d = __ldg(reinterpret_cast<const float4 *>(shift + cw));
        const float4 e = __ldg(reinterpret_cast<const float4 *>(slope + cw));
        const float4 n = BITS && next_bias ? __ldg(reinterpret_cast<const float4 *>(next_bias + cw)) : make_float4(0.f, 0.f, 0.f, 0.f);
        sc = {pack2(a.x, a.y), pack2(a.z, a.w)};
        sh = {pack2(d.x, d.y), pack2(d.z, d.w)};
        sl[0] = e.x; sl[1] = e.y; sl[2] = e.z; sl[3] = e.w;
        nb[0] = n.x; nb[1] = n.y; nb[2] = n.z; nb[3] = n.w;
    }
    const uint32_t my_off = (uint32_t)((2 * rp * S * D::WB + sg * D::L * S) * CB * 2) + 8u * g;
    unsigned n = 0;
    bool ok = true;
    for (unsigned t = first; t < tiles; t += step, ++n) {
        ok = tc::mbar_wait(bar0 + 8u * (n & 1u), (n >> 1) & 1u, &abort_flag, err, ERR_DW_TIMEOUT);
        if (__syncthreads_or(!ok)) break;
        unsigned b;
        int oh0, ow0;
        tile_at(t, b, oh0, ow0);
        const int oh = oh0 + DW_NR * rp, ow1 = ow0 + sg * D::L;
        const uint32_t src = buf0 + (n & 1u) * (uint32_t)D::BUF + my_off;
        uint16_t *yp = y + (((long)b * OH + oh) * OW + ow1) * C + c0;
        const bool row_ok[DW_NR] = {have && oh < OH, have && oh + 1 < OH};
        auto column = [&](int col, F4 (&c)[ROWS]) {             // column `col` of the strip's window
#pragma unroll
            for (int r = 0; r < ROWS; ++r) {
                uint2 v;
                asm volatile("ld.shared.v2.b32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(src + (uint32_t)((r * D::WB + col) * CB * 2)));
                c[r] = to_f4(v);
            }
        };
        F4 win[3][ROWS];
        column(0, win[0]);
        if (S == 1) column(1, win[1]);
#pragma unroll
        for (int i = 0; i < D::L; ++i) {
            const int ia = S == 1 ? i % 3 : (2 * i) % 3, im = S == 1 ? (i + 1) % 3 : (2 * i + 1) % 3, iz = S == 1 ? (i + 2) % 3 : (2 * i + 2) % 3;
            if (S == 2) column(2 * i + 1, win[im]);
            column(S * i + 2, win[iz]);
#pragma unroll
            for (int q = 0; q < DW_NR; ++q) {
                F4 acc = {0ull, 0ull};
#pragma unroll
                for (int r = 0; r < 3; ++r) {
                    acc.lo = fma2(win[ia][q * S + r].lo, wt[3 * r].lo, acc.lo); acc.hi = fma2(win[ia][q * S + r].hi, wt[3 * r].hi, acc.hi);
                    acc.lo = fma2(win[im][q * S + r].lo, wt[3 * r + 1].lo, acc.lo); acc.hi = fma2(win[im][q * S + r].hi, wt[3 * r + 1].hi, acc.hi);
                    acc.lo = fma2(win[iz][q * S + r].lo, wt[3 * r + 2].lo, acc.lo); acc.hi = fma2(win[iz][q * S + r].hi, wt[3 * r + 2].hi, acc.hi);
                }
                acc.lo = fma2(acc.lo, sc.lo, sh.lo);
                acc.hi = fma2(acc.hi, sc.hi, sh.hi);
                float v[4];
                unpack2(acc.lo, v[0], v[1]);
                unpack2(acc.hi, v[2], v[3]);
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = v[k] >= 0.f ? v[k] : sl[k] * v[k];
                const __half2 h0 = __floats2half2_rn(v[0], v[1]), h1 = __floats2half2_rn(v[2], v[3]);
                const bool live = row_ok[q] && ow1 + i < OW;
                uint16_t *dst = yp + (long)q * OW * C;
                if (live) *reinterpret_cast<uint2 *>(dst) = make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
                if (BITS) {
                    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
                    uint32_t bits = (__fadd_rn(f0.x, nb[0]) >= 0.f ? 1u : 0u) | (__fadd_rn(f0.y, nb[1]) >= 0.f ? 2u : 0u) |
                                    (__fadd_rn(f1.x, nb[2]) >= 0.f ? 4u : 0u) | (__fadd_rn(f1.y, nb[3]) >= 0.f ? 8u : 0u);
                    bits |= __shfl_down_sync(0xffffffffu, bits, 1) << 4;      // an even lane and its neighbour are one byte
                    if (live && (g & 1u) == 0) y_bits[(dst - y) >> 3] = (uint8_t)bits;
                }
            }
            yp += C;
        }
        __syncthreads();                                        // the buffer has been read
        if (tid == 0 && t + 2 * step < tiles) issue(t + 2 * step, n & 1u);
    }
    // after a time-out: copies still in flight must land before the CTA's shared memory goes away
    if (!ok || abort_flag) {
        for (unsigned k = 0; k < 2; ++k)
            if (first + (n + k) * step < tiles) tc::mbar_wait(bar0 + 8u * ((n + k) & 1u), ((n + k) >> 1) & 1u, &abort_flag, nullptr, 0);
    }
    pdl_trigger();
}

template <int S, int TW, int CB>
int launch_dw_tile(const uint16_t *x, const float *w, const float *scale, const float *shift, const float *slope, const float *next_bias,
                   uint16_t *y, uint8_t *y_bits, int B, int H, int W, int C_in, int C, int OH, int OW, cudaStream_t stream)
{
    using D = DwCfg<S, TW, CB>;
    EncodeTiledFn encode = encode_tiled_fn();
    if (!encode) return BCNN_ERR_CUDA;
    CUtensorMap xmap;
    const cuuint64_t dims[4] = {(cuuint64_t)C_in, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
    const cuuint64_t strides[3] = {(cuuint64_t)C_in * 2, (cuuint64_t)W * C_in * 2, (cuuint64_t)H * W * C_in * 2};
    const cuuint32_t box[4] = {CB, D::WB, D::HB, 1}, estr[4] = {1, 1, 1, 1};
    if (encode(&xmap, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<uint16_t *>(x), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return BCNN_ERR_CUDA;
    auto k = y_bits ? dw_tile_kernel<S, TW, CB, true> : dw_tile_kernel<S, TW, CB, false>;
    if (!allow_smem((const void *)k, D::SMEM)) return BCNN_ERR_CUDA;
    const unsigned tx = (unsigned)(OW + TW - 1) / TW, ty = (unsigned)(OH + DW_TH - 1) / DW_TH, tiles = tx * ty * (unsigned)B;
    const unsigned cblocks = (unsigned)(C + CB - 1) / CB;
    // resident blocks, the same number for every channel block and the same number of tiles (+-1) for each
    unsigned per = (unsigned)sm_count() * (unsigned)blocks_per_sm((const void *)k, D::THREADS, D::SMEM) / cblocks;
    if (per < 1) per = 1;
    if (per > tiles) per = tiles;
    return launch(k, per * cblocks, D::THREADS, D::SMEM, stream, xmap, w, scale, shift, slope, next_bias, y, y_bits, C_in, C, OH, OW, tx, ty, tiles, cblocks, device_error_word());
}

// Any stride and channel count (the tiles above take strides 1 and 2 and channel blocks that replication does not split): one output pixel x 8 channels per thread.
// x fp16 [B][H][W][C_in] -> y fp16 [B][OH][OW][C], C = R * C_in; w fp32 [C][3][3].
// The block's thread count is a multiple of the 8-channel groups, so a thread keeps its group; weights (tap-major, so
// that a warp's groups read consecutive 32-byte pieces) and per-channel values sit in shared memory.  A block walks a
// CONTIGUOUS range of output pixels, row after row, so that the input rows shared by vertically adjacent outputs are
// still in L1 when they are needed again (with a grid-stride walk every tap came from L2: nine times the input's
// bytes); a thread's pixel coordinates advance by the block's pass size, by carries.
__global__ void __launch_bounds__(256)
dwconv3x3_module_kernel(const uint16_t *x, const float *w, const float *scale, const float *shift, const float *slope,
                        const float *next_bias, uint16_t *y, uint8_t *y_bits,
                        int B, int H, int W, int C_in, int C, int S, int OH, int OW)
{
    // 13 per-channel vectors (nine taps, scale, shift, slope, next bias), each stored as two float4 arrays over the
    // 8-channel groups - channels 8g..8g+3 at [2q][g], 8g+4..8g+7 at [2q+1][g] - so that a warp's groups read
    // consecutive 16-byte pieces (one float per lane, or 32-byte pieces per lane, would conflict 8- and 2-way)
    extern __shared__ __align__(16) float dw_smem[];
    pdl_trigger();
    pdl_wait();
    const int groups = C / 8;
    const float4 *vec = reinterpret_cast<const float4 *>(dw_smem);
    for (int i = threadIdx.x; i < 13 * C; i += blockDim.x) {
        const int q = i / C, c = i % C;
        float val;
        if (q < 9) val = __ldg(w + c * 9 + q);
        else if (q == 9) val = __ldg(scale + c);
        else if (q == 10) val = __ldg(shift + c);
        else if (q == 11) val = __ldg(slope + c);
        else val = next_bias ? __ldg(next_bias + c) : 0.f;
        dw_smem[((2 * q + ((c & 7) >> 2)) * groups + (c >> 3)) * 4 + (c & 3)] = val;
    }
    __syncthreads();
    const int g = threadIdx.x % groups, ppb = blockDim.x / groups;      // pixels per block and pass
    const int c0 = 8 * g, ci0 = c0 % C_in;                     // replication: channel c reads channel c mod C_in
    const unsigned npix = (unsigned)B * OH * OW;
    const unsigned per_block = ((npix + gridDim.x - 1) / gridDim.x + ppb - 1) / ppb * ppb;     // a multiple of the pass size
    const unsigned stride = (unsigned)ppb;
    unsigned pix = blockIdx.x * per_block + threadIdx.x / groups;
    const unsigned pix_end = min(npix, (blockIdx.x + 1) * per_block);
    int b = (int)(pix / ((unsigned)OH * OW)), oh = (int)((pix / OW) % OH), ow = (int)(pix % OW);
    const int db = (int)(stride / ((unsigned)OH * OW)), doh = (int)((stride / OW) % OH), dow = (int)(stride % OW);
    for (; pix < pix_end; pix += stride) {
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        // all nine taps are requested before the first is used (predicated loads, zero outside the image)
        uint4 v[9];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            const int ih = oh * S - 1 + r;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const int iw = ow * S - 1 + t;
                const bool ok = ih >= 0 && ih < H && iw >= 0 && iw < W;
                v[r * 3 + t] = ok ? __ldg(reinterpret_cast<const uint4 *>(x + (((long)b * H + ih) * W + iw) * C_in + ci0)) : make_uint4(0u, 0u, 0u, 0u);
            }
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) {
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                float xv[8];
                unpack8(v[r * 3 + t], xv);
                const float4 w0 = vec[(2 * (r * 3 + t)) * groups + g], w1 = vec[(2 * (r * 3 + t) + 1) * groups + g];
                acc[0] = fmaf(xv[0], w0.x, acc[0]); acc[1] = fmaf(xv[1], w0.y, acc[1]);
                acc[2] = fmaf(xv[2], w0.z, acc[2]); acc[3] = fmaf(xv[3], w0.w, acc[3]);
                acc[4] = fmaf(xv[4], w1.x, acc[4]); acc[5] = fmaf(xv[5], w1.y, acc[5]);
                acc[6] = fmaf(xv[6], w1.z, acc[6]); acc[7] = fmaf(xv[7], w1.w, acc[7]);
            }
        }
        uint32_t ow4[4];
        uint32_t bits = 0;
        float sc8[8], sh8[8], sl8[8], nb8[8];
        {
            const float4 a0 = vec[18 * groups + g], a1 = vec[19 * groups + g], b0 = vec[20 * groups + g], b1 = vec[21 * groups + g];
            const float4 d0 = vec[22 * groups + g], d1 = vec[23 * groups + g], e0 = vec[24 * groups + g], e1 = vec[25 * groups + g];
            sc8[0] = a0.x; sc8[1] = a0.y; sc8[2] = a0.z; sc8[3] = a0.w; sc8[4] = a1.x; sc8[5] = a1.y; sc8[6] = a1.z; sc8[7] = a1.w;
            sh8[0] = b0.x; sh8[1] = b0.y; sh8[2] = b0.z; sh8[3] = b0.w; sh8[4] = b1.x; sh8[5] = b1.y; sh8[6] = b1.z; sh8[7] = b1.w;
            sl8[0] = d0.x; sl8[1] = d0.y; sl8[2] = d0.z; sl8[3] = d0.w; sl8[4] = d1.x; sl8[5] = d1.y; sl8[6] = d1.z; sl8[7] = d1.w;
            nb8[0] = e0.x; nb8[1] = e0.y; nb8[2] = e0.z; nb8[3] = e0.w; nb8[4] = e1.x; nb8[5] = e1.y; nb8[6] = e1.z; nb8[7] = e1.w;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float r2[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float tt = fmaf(acc[2 * q + e], sc8[2 * q + e], sh8[2 * q + e]);
                r2[e] = tt >= 0.f ? tt : sl8[2 * q + e] * tt;
            }
            const __half2 y2 = __floats2half2_rn(r2[0], r2[1]);
            ow4[q] = *reinterpret_cast<const uint32_t *>(&y2);
            if (y_bits) {
                const float2 yf = __half22float2(y2);
                bits |= (__fadd_rn(yf.x, nb8[2 * q]) >= 0.f ? 1u : 0u) << (2 * q);
                bits |= (__fadd_rn(yf.y, nb8[2 * q + 1]) >= 0.f ? 1u : 0u) << (2 * q + 1);
            }
        }
        *reinterpret_cast<uint4 *>(y + (long)pix * C + c0) = make_uint4(ow4[0], ow4[1], ow4[2], ow4[3]);
        if (y_bits) y_bits[((long)pix * C + c0) >> 3] = (uint8_t)bits;
        // next pixel of this thread: + stride, by carries
        ow += dow;
        if (ow >= OW) { ow -= OW; ++oh; }
        oh += doh;
        if (oh >= OH) { oh -= OH; ++b; }
        b += db;
    }
}

// S x S / S average pooling with replication, bound by the maps' traffic.  A thread takes 8 channels of AP output pixels
// (AP * S * S 16-byte loads in flight), reads every input value once and writes its R copies (channel c reads c mod C_in).
// SS: the stride where it is known to the compiler (1, 2), else 0.
constexpr int AP = 4;
template <int SS>
__global__ void __launch_bounds__(256)
avgpool_kernel(const uint16_t *x, uint16_t *y, unsigned items, int H, int W, int C_in, int R, int S_any)
{
    pdl_trigger();
    const int S = SS ? SS : S_any;
    const unsigned OW = (unsigned)(W / S), OH = (unsigned)(H / S), groups = (unsigned)C_in / 8;
    const long C = (long)C_in * R;
    const float inv = 1.0f / (float)(S * S);
    pdl_wait();
    const unsigned stride = gridDim.x * 256u, first = blockIdx.x * 256u + threadIdx.x;
    // AP items, `stride` apart, at a time: item = (output pixel, group of 8 channels)
    for (unsigned i0 = first; i0 < items; i0 += AP * stride) {
        float acc[AP][8];
        long src[AP], dst[AP];
        bool ok[AP];
#pragma unroll
        for (int u = 0; u < AP; ++u) {
            const unsigned i = i0 + u * stride;
            ok[u] = i < items && i >= i0;
            const unsigned pix = i / groups, g = i - pix * groups;
            const unsigned row = pix / OW, ow = pix - row * OW, b = row / OH, oh = row - b * OH;
            src[u] = (((long)b * H + (long)oh * S) * W + (long)ow * S) * C_in + 8 * g;
            dst[u] = (long)pix * C + 8 * g;
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[u][c] = 0.f;
        }
        if (SS) {
            uint4 v[AP][SS ? SS * SS : 1];
#pragma unroll
            for (int u = 0; u < AP; ++u)
#pragma unroll
                for (int q = 0; q < SS * SS; ++q)
                    v[u][q] = ok[u] ? __ldg(reinterpret_cast<const uint4 *>(x + src[u] + ((long)(q / (SS ? SS : 1)) * W + q % (SS ? SS : 1)) * C_in)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < AP; ++u)
#pragma unroll
                for (int q = 0; q < SS * SS; ++q) {
                    float xv[8];
                    unpack8(v[u][q], xv);
#pragma unroll
                    for (int c = 0; c < 8; ++c) acc[u][c] += xv[c];
                }
        } else {
            for (int r = 0; r < S; ++r)
                for (int t = 0; t < S; ++t)
#pragma unroll
                    for (int u = 0; u < AP; ++u)
                        if (ok[u]) {
                            float xv[8];
                            unpack8(__ldg(reinterpret_cast<const uint4 *>(x + src[u] + ((long)r * W + t) * C_in)), xv);
#pragma unroll
                            for (int c = 0; c < 8; ++c) acc[u][c] += xv[c];
                        }
        }
#pragma unroll
        for (int u = 0; u < AP; ++u) {
            uint32_t o[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const __half2 y2 = __floats2half2_rn(acc[u][2 * q] * inv, acc[u][2 * q + 1] * inv);
                o[q] = *reinterpret_cast<const uint32_t *>(&y2);
            }
            if (ok[u])
                for (int k = 0; k < R; ++k) *reinterpret_cast<uint4 *>(y + dst[u] + (long)k * C_in) = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

// pooled[b][c] = mean over the HW pixels.  A block takes GX groups of 8 channels of one image and cuts its pixels into
// 256 / GX slices (a thread per group and slice, eight 16-byte loads in flight), then adds the slices in shared memory: one thread per
// group alone leaves the chip with a few loads in flight per multiprocessor (7x7x1024 at batch 256: 22 us; floor 4).
__global__ void __launch_bounds__(256)
gap_kernel(const uint16_t *x, float *pooled, int HW, int C, int GX)
{
    __shared__ float part[256 * 9];                             // 8 sums per thread, rows of 9: no bank conflicts
    const int groups = C / 8, tiles = (groups + GX - 1) / GX;
    const int b = (int)(blockIdx.x / tiles), g0 = (int)(blockIdx.x - b * tiles) * GX;
    const int gi = (int)threadIdx.x % GX, slice = (int)threadIdx.x / GX, slices = 256 / GX;
    const bool have = g0 + gi < groups;
    pdl_wait();
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const uint16_t *src = x + (long)b * HW * C + 8 * (g0 + gi);
    constexpr int U = 8;
    if (have)
        for (int q0 = slice; q0 < HW; q0 += U * slices) {
            uint4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                v[u] = q0 + u * slices < HW ? __ldg(reinterpret_cast<const uint4 *>(src + (long)(q0 + u * slices) * C)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                float xv[8];
                unpack8(v[u], xv);
#pragma unroll
                for (int c = 0; c < 8; ++c) acc[c] += xv[c];
            }
        }
    pdl_trigger();
#pragma unroll
    for (int c = 0; c < 8; ++c) part[threadIdx.x * 9 + c] = acc[c];
    __syncthreads();
    const float inv = 1.0f / (float)HW;
    for (int i = threadIdx.x; i < 8 * GX; i += 256) {           // channel i of the block
        float t = 0.f;
        for (int sl = 0; sl < slices; ++sl) t += part[(sl * GX + (i >> 3)) * 9 + (i & 7)];
        if (8 * g0 + i < C) pooled[(long)b * C + 8 * g0 + i] = t * inv;
    }
}

// logits = pooled * w^T + bias as a tiled fp32 product: FT_M images x FT_N outputs per CTA, K in chunks of FT_K through a ring of
// cp.async stages.  The eight warps take four of a chunk's K values each and every warp owns all of the tile, 8 x 8 outputs
// per thread; the warps' sums are added through shared memory.  SPLIT CTAs (a cluster) share a tile's K where there are too few
// tiles for the chip, and add their sums through each other's shared memory (64 x 100 x 2048: 12.0 -> 5.4 us, 256 x 10 x 2048 10.5 ->
// 5.2).  32 outputs where tiles are few; with 64 a weight goes twice as far (256 x 1000 x 256: 7.4 and 6.7 us).  Up to a wave the CTAs ask
// for so much shared memory that each has its multiprocessor to itself: left to itself the scheduler pairs some of 130 to 148 while others idle
// (215 images x 656 outputs x 916: 16.0 -> 11.9 us).  In several waves of 32 outputs two share a multiprocessor,
// six stages or 59 KB each; with eight stages the times are those of one (498 x 708 x 1512: 55.8 and 45.4).  What is left at 256 x 1000 x 1024 (20.7 -> 19.6 us, 7.1 of the fp32 pipe) did not move with 16 x 8
// outputs per thread, pairs of multiply-adds, chunks of 64, 16-byte reads or a rolled loop.
constexpr int FT_M = 32, FT_K = 32, FT_THREADS = 256, FT_PITCH = FT_K + 4;
constexpr int FT_PIECES = FT_K / 4, FT_ROWS = FT_THREADS / FT_PIECES, FT_KW = FT_K / 8;      // 16-byte pieces of a row, rows loaded at a time, a warp's K values

__host__ __device__ constexpr int ft_stages(int n) { return n == 32 ? 6 : 8; }
constexpr int ft_smem(int n) { return (ft_stages(n) * (FT_M + n) * FT_PITCH + FT_M * n) * 4; }
constexpr int FT_ALONE = 116 * 1024;
template <int SPLIT, int FT_N>
__global__ void __launch_bounds__(FT_THREADS, FT_N == 32 ? 2 : 1)
fc_tile_kernel(const float *pooled, const float *w, const float *bias, float *logits, int B, int C, int N, int per)
{
    constexpr int FT_STAGES = ft_stages(FT_N), FT_STAGE_FLOATS = (FT_M + FT_N) * FT_PITCH, NJ = FT_N / 8;
    static_assert(8 * FT_M * FT_N <= FT_STAGES * FT_STAGE_FLOATS, "the warps' sums fit the stages");
    extern __shared__ __align__(16) float sm[];                 // [FT_STAGES][FT_STAGE_FLOATS], [FT_M][FT_N] sums of this CTA
    const int tid = threadIdx.x, warp = tid >> 5, tm = (tid & 31) >> 3, tn = tid & 7;
    const int rank = (int)blockIdx.x % SPLIT;
    const int b0 = blockIdx.y * FT_M, n0 = (int)blockIdx.x / SPLIT * FT_N;
    // `per` chunks of K are this CTA's
    const int k_end = min(C, (rank + 1) * per * FT_K), k_first = rank * per * FT_K;
    const int chunks = max(0, (k_end - k_first + FT_K - 1) / FT_K);
    const uint32_t base = tc::smem_u32(sm);
    const int lrow = tid / FT_PIECES, lk = 4 * (tid % FT_PIECES);
    pdl_wait();
    auto load = [&](int ch) {
        if (ch < chunks) {
            const int k = k_first + ch * FT_K + lk;
            const uint32_t dst = base + (uint32_t)(((ch % FT_STAGES) * FT_STAGE_FLOATS + lrow * FT_PITCH + lk) * 4);
#pragma unroll
            for (int i = 0; i < (FT_M + FT_N) / FT_ROWS; ++i) {
                const int row = lrow + FT_ROWS * i, gr = FT_ROWS * i < FT_M ? b0 + row : n0 + row - FT_M;
                const bool ok = k < k_end && gr < (FT_ROWS * i < FT_M ? B : N);
                tc::cp_async16(dst + (uint32_t)(FT_ROWS * i * FT_PITCH * 4), (FT_ROWS * i < FT_M ? pooled : w) + (ok ? (long)gr * C + k : 0), ok);
            }
        }
        tc::cp_async_commit();
    };
    float acc[8][NJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = 0.f;
#pragma unroll 1
    for (int ch = 0; ch < FT_STAGES - 1; ++ch) load(ch);
#pragma unroll 1
    for (int ch = 0; ch < chunks; ++ch) {
        tc::cp_async_wait<FT_STAGES - 2>();
        __syncthreads();                                        // chunk ch has landed; everybody is done reading chunk ch - 1
        load(ch + FT_STAGES - 1);
        const float *pa = sm + (ch % FT_STAGES) * FT_STAGE_FLOATS + tm * FT_PITCH + FT_KW * warp;
        const float *pb = sm + (ch % FT_STAGES) * FT_STAGE_FLOATS + (FT_M + tn) * FT_PITCH + FT_KW * warp;
#pragma unroll
        for (int h = 0; h < FT_KW / 2; ++h) {
            float2 fa[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) fa[i] = *reinterpret_cast<const float2 *>(pa + 4 * i * FT_PITCH + 2 * h);
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const float2 fb = *reinterpret_cast<const float2 *>(pb + 8 * j * FT_PITCH + 2 * h);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i][j] = fmaf(fa[i].x, fb.x, acc[i][j]);
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i][j] = fmaf(fa[i].y, fb.y, acc[i][j]);
            }
        }
    }
    pdl_trigger();
    tc::cp_async_wait<0>();
    __syncthreads();
    // the warps' sums; the banks of rows tm, columns tn are 4 x 8 different ones
    float *red = sm;                                            // [8 warps][FT_M][FT_N]
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) red[(warp * FT_M + tm + 4 * i) * FT_N + ((tn + 8 * j) ^ (8 * tm))] = acc[i][j];
    __syncthreads();
    float *mine = sm + FT_STAGES * FT_STAGE_FLOATS;
#pragma unroll 1
    for (int q = 0; q < FT_M * FT_N / FT_THREADS; ++q) {
        const int e = tid + FT_THREADS * q, row = e / FT_N, col = e % FT_N, at = row * FT_N + (col ^ (8 * (row & 3)));
        float v = 0.f;
#pragma unroll
        for (int wp = 0; wp < 8; ++wp) v += red[wp * FT_M * FT_N + at];
        if (SPLIT > 1) {
            mine[e] = v;
        } else {
            const int b = b0 + row, n = n0 + col;
            if (b < B && n < N) logits[(long)b * N + n] = v + (bias ? __ldg(bias + n) : 0.f);
        }
    }
    if (SPLIT > 1) {
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
        for (int e = rank * (FT_M * FT_N / SPLIT) + tid; e < (rank + 1) * (FT_M * FT_N / SPLIT); e += FT_THREADS) {
            const int b = b0 + e / FT_N, n = n0 + e % FT_N;
            const uint32_t at = tc::smem_u32(mine + e);
            float v = 0.f;
#pragma unroll
            for (uint32_t r = 0; r < (uint32_t)SPLIT; ++r) {
                uint32_t there;
                float t;
                asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(there) : "r"(at), "r"(r));
                asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(t) : "r"(there) : "memory");
                v += t;
            }
            if (b < B && n < N) logits[(long)b * N + n] = v + (bias ? __ldg(bias + n) : 0.f);
        }
        // the others have read this CTA's sums
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

// logits[b][n] = sum_c pooled[b][c] * w[n][c] + bias[n].  A CTA takes FC_IMAGES images (their pooled rows in shared
// memory) and all outputs; a warp takes outputs warp, warp + 8, ...: lanes stride over c with 16-byte weight loads
// (each weight row is read once per CTA), then a shuffle reduction.
constexpr int FC_IMAGES = 4, FC_U = 4;     // images per CTA; 16-byte weight loads in flight per lane
__global__ void __launch_bounds__(256)
fc_kernel(const float *pooled, const float *w, const float *bias, float *logits, int B, int C, int N)
{
    extern __shared__ __align__(16) float fc_smem[];           // [FC_IMAGES][C]
    pdl_wait();
    const int b0 = blockIdx.x * FC_IMAGES;
    const int nb = min(FC_IMAGES, B - b0);
    for (int i = threadIdx.x; i < FC_IMAGES * C; i += blockDim.x)
        fc_smem[i] = (i / C) < nb ? __ldg(pooled + (long)b0 * C + i) : 0.f;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // blockIdx.y takes every gridDim.y-th group of eight outputs
    for (int n = blockIdx.y * 8 + warp; n < N; n += 8 * gridDim.y) {
        float acc[FC_IMAGES] = {0.f, 0.f, 0.f, 0.f};
        const float4 *wr = reinterpret_cast<const float4 *>(w + (long)n * C);
        for (int c0 = lane; c0 < C / 4; c0 += 32 * FC_U) {
            float4 wv[FC_U];
#pragma unroll
            for (int u = 0; u < FC_U; ++u) wv[u] = c0 + 32 * u < C / 4 ? __ldg(wr + c0 + 32 * u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int u = 0; u < FC_U; ++u) {
                if (c0 + 32 * u >= C / 4) break;
#pragma unroll
                for (int im = 0; im < FC_IMAGES; ++im) {
                    const float4 pv = reinterpret_cast<const float4 *>(fc_smem + im * C)[c0 + 32 * u];
                    acc[im] = fmaf(pv.x, wv[u].x, fmaf(pv.y, wv[u].y, fmaf(pv.z, wv[u].z, fmaf(pv.w, wv[u].w, acc[im]))));
                }
            }
        }
#pragma unroll
        for (int im = 0; im < FC_IMAGES; ++im) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) acc[im] += __shfl_xor_sync(0xffffffffu, acc[im], off);
        }
        float v = acc[0];
        if (lane == 1) v = acc[1];
        if (lane == 2) v = acc[2];
        if (lane == 3) v = acc[3];
        if (lane < nb) logits[(long)(b0 + lane) * N + n] = v + (bias ? __ldg(bias + n) : 0.f);
    }
    pdl_trigger();          // late: blocks of the next kernel that came in beside these ones would end up unevenly spread
}

}  // namespace

int launch_dwconv3x3_module(const uint16_t *x, const float *w, const float *scale, const float *shift, const float *slope,
                            const float *next_bias, uint16_t *y, uint8_t *y_bits, int B, int H, int W, int C_in, int R, int S,
                            cudaStream_t stream)
{
    const int C = C_in * R, OH = (H + 2 - 3) / S + 1, OW = (W + 2 - 3) / S + 1;
    const int groups = C / 8;
    const int smem = 13 * C * 4;
    if (groups > 256 || smem > 200 * 1024) return BCNN_ERR_UNSUPPORTED;      // more than 2048 channels
    if ((long)B * OH * OW >= (1L << 31)) return BCNN_ERR_UNSUPPORTED;         // pixel indices are 32-bit
    // tiles of 8 x 16 output pixels at stride 1 (8 x 8 where that covers the row with less waste, and at stride 2: the halo is
    // 17 x 17 pixels); 64 channels, or 32 where 64 do not divide the input's channels
    const int CB = C_in % 64 == 0 ? 64 : 32;
    if (S <= 2 && (R == 1 || C_in % CB == 0) && (long)B * ((OH + 7) / 8) * ((OW + 7) / 8) < (1L << 30)) {
        const bool narrow = S == 2 || (OW + 7) / 8 * 8 < (OW + 15) / 16 * 16;
        if (S == 1 && narrow) return CB == 64 ? launch_dw_tile<1, 8, 64>(x, w, scale, shift, slope, next_bias, y, y_bits, B, H, W, C_in, C, OH, OW, stream)
                                              : launch_dw_tile<1, 8, 32>(x, w, scale, shift, slope, next_bias, y, y_bits, B, H, W, C_in, C, OH, OW, stream);
        if (S == 1) return CB == 64 ? launch_dw_tile<1, 16, 64>(x, w, scale, shift, slope, next_bias, y, y_bits, B, H, W, C_in, C, OH, OW, stream)
                                    : launch_dw_tile<1, 16, 32>(x, w, scale, shift, slope, next_bias, y, y_bits, B, H, W, C_in, C, OH, OW, stream);
        return CB == 64 ? launch_dw_tile<2, 8, 64>(x, w, scale, shift, slope, next_bias, y, y_bits, B, H, W, C_in, C, OH, OW, stream)
                        : launch_dw_tile<2, 8, 32>(x, w, scale, shift, slope, next_bias, y, y_bits, B, H, W, C_in, C, OH, OW, stream);
    }
    const int threads = (256 / groups) * groups;                            // <= 256, a multiple of groups
    const long passes = ((long)B * OH * OW + threads / groups - 1) / (threads / groups);
    const int sms = sm_count();
    const long cap = (long)sms * 8;
    const unsigned blocks = (unsigned)(passes < cap ? passes : cap);
    if (!allow_smem((const void *)dwconv3x3_module_kernel, 200 * 1024)) return BCNN_ERR_CUDA;
    return launch(dwconv3x3_module_kernel, blocks, threads, smem, stream, x, w, scale, shift, slope, next_bias, y, y_bits,
                  B, H, W, C_in, C, S, OH, OW);
}

int launch_avgpool(const uint16_t *x, uint16_t *y, int B, int H, int W, int C_in, int R, int S, cudaStream_t stream)
{
    const long items = (long)B * (H / S) * (W / S) * (C_in / 8);
    if (items >= (1L << 31)) {                       // item numbers are 32-bit: whole images per launch
        const int part = (int)(((1L << 31) - 1) / (items / B));
        if (part < 1) return BCNN_ERR_UNSUPPORTED;
        for (int b = 0; b < B; b += part) {
            const int st = launch_avgpool(x + (long)b * H * W * C_in, y + (long)b * (H / S) * (W / S) * C_in * R, B - b < part ? B - b : part, H, W, C_in, R, S, stream);
            if (st != BCNN_OK) return st;
        }
        return BCNN_OK;
    }
    void (*k)(const uint16_t *, uint16_t *, unsigned, int, int, int, int, int) = S == 1 ? avgpool_kernel<1> : (S == 2 ? avgpool_kernel<2> : avgpool_kernel<0>);
    const long blocks = (items + 256 * AP - 1) / (256 * AP), cap = (long)sm_count() * blocks_per_sm((const void *)k, 256, 0);
    return launch(k, (unsigned)(blocks < cap ? blocks : cap), 256, 0, stream, x, y, (unsigned)items, H, W, C_in, R, S);
}

int launch_gap(const uint16_t *x, float *pooled, int B, int HW, int C, cudaStream_t stream)
{
    // channel groups of a block: the power of two that fits the channels, up to 32; fewer, and more pixels at a time, where that many
    // leave multiprocessors idle (8 images of 10 x 10 x 192: 4.0 -> 2.4 us, 4 of 9 x 9 x 2048 3.8 -> 2.7, 2 of 14 x 14 x 1600 6.9 -> 2.9;
    // 200 of 9 x 9 x 264 4.9 with 32, 5.2 with 8).  Not for so few pixels that a slice has no more than three: the slices' sums are added one after
    // the other (14 images of 2 x 2 x 1112 1.80 -> 2.07 us, 131 of 4 x 4 x 152 2.21 -> 2.50)
    const int groups = C / 8;
    int GX = 32;
    while (GX > 1 && GX / 2 >= groups) GX /= 2;
    while (GX > 8 && HW > 3 * (256 / GX) && (long)B * ((groups + GX - 1) / GX) < sm_count()) GX /= 2;
    const long blocks = (long)B * ((groups + GX - 1) / GX);
    if (blocks >= (1L << 31)) return BCNN_ERR_UNSUPPORTED;
    return launch(gap_kernel, (unsigned)blocks, 256, 0, stream, x, pooled, HW, C, GX);
}

// What a tile's launch asks for in shared memory: `alone`, so much that no second CTA comes in beside it.
template <int FT_N> constexpr int ft_ask(bool alone) { return alone && ft_smem(FT_N) < FT_ALONE ? FT_ALONE : ft_smem(FT_N); }

// Clusters of SPLIT CTAs, each alone on its multiprocessor, that run at a time.
template <int SPLIT, int FT_N>
static long fc_capacity()
{
    if (SPLIT == 1) return sm_count();
    auto k = fc_tile_kernel<SPLIT, FT_N>;
    if (!allow_smem((const void *)k, ft_ask<FT_N>(true))) return 0;
    return max_clusters((const void *)k, SPLIT, FT_THREADS, ft_ask<FT_N>(true));
}

template <int SPLIT, int FT_N>
static int launch_fc_tile(const float *pooled, const float *w, const float *bias, float *logits, int B, int C, int N, long tiles_n, long tiles_b, bool alone, cudaStream_t stream)
{
    auto k = fc_tile_kernel<SPLIT, FT_N>;
    if (!allow_smem((const void *)k, ft_ask<FT_N>(true))) return BCNN_ERR_CUDA;
    const int chunks = (C + FT_K - 1) / FT_K, per = (chunks + SPLIT - 1) / SPLIT;
    return launch<SPLIT>(k, dim3((unsigned)(tiles_n * SPLIT), (unsigned)tiles_b), FT_THREADS, ft_ask<FT_N>(alone), stream, pooled, w, bias, logits, B, C, N, per);
}

// A width and a split of K with the time they are expected to take, ns.
struct FcPlan {
    long ns;
    int split;
    bool alone;
};

template <int FT_N>
static FcPlan fc_plan(long tiles, int chunks)
{
    const long sms = sm_count();
    FcPlan best = {LONG_MAX, 1, false};
    for (int split = 1; split <= 8 && (split == 1 || split <= chunks); split *= 2) {
        // a split tile is one wave: a second one costs more than its shorter K saves
        const long fit = split == 1 ? fc_capacity<1, FT_N>() : split == 2 ? fc_capacity<2, FT_N>() : split == 4 ? fc_capacity<4, FT_N>() : fc_capacity<8, FT_N>();
        if (split > 1 && tiles > fit) break;
        const long per = (chunks + split - 1) / split;
        long ns;
        if (FT_N == 64) {
            ns = 160 + (split > 1 ? 790 : 0) + (tiles + sms - 1) / sms * (1845 + 529 * per);
        } else if (tiles <= fit) {
            ns = 1540 + (split > 1 ? 940 : 0) + 337 * per;
            if (ns < 2150) ns = 2150;
        } else {
            // two on a multiprocessor, the last wave's perhaps alone
            const long shared = tiles / (2 * sms), rest = tiles % (2 * sms);
            ns = 830 + (shared + (rest > sms)) * (1470 + 527 * per) + (rest > 0 && rest <= sms ? 1100 + 332 * per : 0);
        }
        if (ns < best.ns) best = {ns, split, tiles <= fit};
    }
    return best;
}

template <int FT_N>
static int launch_fc_tiles(const FcPlan &plan, const float *pooled, const float *w, const float *bias, float *logits, int B, int C, int N, long tiles_n, long tiles_b, cudaStream_t stream)
{
    switch (plan.split) {
    case 8: return launch_fc_tile<8, FT_N>(pooled, w, bias, logits, B, C, N, tiles_n, tiles_b, plan.alone, stream);
    case 4: return launch_fc_tile<4, FT_N>(pooled, w, bias, logits, B, C, N, tiles_n, tiles_b, plan.alone, stream);
    case 2: return launch_fc_tile<2, FT_N>(pooled, w, bias, logits, B, C, N, tiles_n, tiles_b, plan.alone, stream);
    default: return launch_fc_tile<1, FT_N>(pooled, w, bias, logits, B, C, N, tiles_n, tiles_b, plan.alone, stream);
    }
}

int launch_fc(const float *pooled, const float *w, const float *bias, float *logits, int B, int C, int N, cudaStream_t stream)
{
    // Tiles of 64 or 32 outputs, with the K of each over as many CTAs as run at a time, or the kernel below, which walks K in steps of 512 for
    // four images at a time.  Estimates in ns, fitted to 4462 heads drawn from 1 .. 512 images, 8 .. 4096 channels and 4 .. 6000 outputs (the choice
    // takes 1 % longer than the best of all variants in the mean); images x channels x outputs, us at 32 and 64 wide, streamed:
    // 32 x 580 x 2344 6.3, 8.7, 16.5; 203 x 516 x 274 5.9, 8.1, 12.8; 2 x 2328 x 1146 13.9, 13.4, 9.5; 4 x 2956 x 42 5.9, 7.0, 13;
    // 167 x 2480 x 2335 73, 92, 208; 446 x 24 x 15 2.1, 2.7, 1.8.  Tiles have to be 8 % ahead: the streaming estimate is the least sure.
    const int sms = sm_count(), chunks = (int)(((long)C + FT_K - 1) / FT_K);
    const long tiles_b = ((long)B + FT_M - 1) / FT_M, n32 = ((long)N + 31) / 32, n64 = ((long)N + 63) / 64, images = ((long)B + FC_IMAGES - 1) / FC_IMAGES;
    const long smem = (long)FC_IMAGES * C * 4;
    const bool streams = smem <= 200 * 1024;
    // rows of more channels than the kernel below can hold (12800) are taken in large products only
    if (!streams && images * N <= 10600 * ((n32 * tiles_b + 2 * sms - 1) / (2 * sms))) return BCNN_ERR_UNSUPPORTED;
    int ny = 1;                                     // (streaming) enough CTAs to fill the GPU a few times over
    while (images * ny < 592 && ny * 8 < N) ny *= 2;
    const long outs = (N + 8L * ny - 1) / (8L * ny);                         // of a warp
    const long streamed = streams ? 1250 + (B < FC_IMAGES ? B : FC_IMAGES) * 94L * C / 100 + outs * ((C + 511) / 512) * 250 + images * N * (180 + 3 * C / 4) / 1000 : LONG_MAX;
    if (tiles_b < 65536 && n32 < (1L << 27)) {
        const FcPlan narrow = fc_plan<32>(n32 * tiles_b, chunks), wide = fc_plan<64>(n64 * tiles_b, chunks);
        const long tiled = narrow.ns < wide.ns ? narrow.ns : wide.ns;
        if (!streams || tiled * 27 / 25 < streamed)
            return narrow.ns <= wide.ns ? launch_fc_tiles<32>(narrow, pooled, w, bias, logits, B, C, N, n32, tiles_b, stream)
                                        : launch_fc_tiles<64>(wide, pooled, w, bias, logits, B, C, N, n64, tiles_b, stream);
    }
    if (!streams) return BCNN_ERR_UNSUPPORTED;
    if (!allow_smem((const void *)fc_kernel, 200 * 1024)) return BCNN_ERR_CUDA;
    return launch(fc_kernel, dim3((unsigned)images, (unsigned)ny), 256, (size_t)smem, stream, pooled, w, bias, logits, B, C, N);
}

}  // namespace bcnn
