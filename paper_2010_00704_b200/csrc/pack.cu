// Binarize + pack kernel: real NHWC fp32 -> sign bits (bit 1 = +1), with optional
// per-channel bias and channel replication (paper Section 4.2.1 bias + sign, Section
// 4.2.2 replication by bookkeeping).  A pure HBM stream: 4 bytes read per input value,
// 1 bit written per output channel.
#include "bcnn_common.cuh"

namespace bcnn {

// Streaming path, no replication, C_in % 32 == 0: the tensor is a flat array of fp32 values and every aligned group of 32
// becomes one output word.  A thread takes four consecutive values (one 16-byte load) and leaves a nibble; eight lanes make a
// word, a warp stores four.  PACK_U loads are in flight per thread, `stride` quads apart.  FIXED: the stride is a multiple of
// the C_in / 4 quads of a pixel, so a thread keeps its four biases in registers; else one 32-bit remainder per load (the
// 64-bit remainder per 32 values of the kernel before this one held 28x28x256 at batch 128 to 2.2 TB/s).
constexpr int PACK_U = 4;
template <bool FIXED>
__global__ void __launch_bounds__(256)
pack_stream_kernel(const float4 *__restrict__ x, const float4 *__restrict__ bias, uint32_t *__restrict__ out, long quads, unsigned q)
{
    pdl_trigger();
    const long stride = (long)gridDim.x * 256, first = (long)blockIdx.x * 256 + threadIdx.x;
    const unsigned lane = threadIdx.x & 31u;
    pdl_wait();
    float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
    if (FIXED && bias) b = __ldg(bias + (unsigned)(first % q));
    for (long i0 = first; i0 - lane < quads; i0 += PACK_U * stride) {           // warp-uniform: quads is a multiple of 8
        float4 v[PACK_U];
#pragma unroll
        for (int u = 0; u < PACK_U; ++u) {
            const long i = i0 + u * stride;
            v[u] = i < quads ? __ldcs(x + i) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < PACK_U; ++u) {
            const long i = i0 + u * stride;
            if (!FIXED) b = i < quads ? __ldg(bias + (unsigned)((unsigned long)i < (1ul << 32) ? (unsigned)i % q : i % q)) : b;
            // without a bias b is zero: x + 0 >= 0 decides like x >= 0 (NaN and -0 included)
            uint32_t w = (__fadd_rn(v[u].x, b.x) >= 0.f ? 1u : 0u) | (__fadd_rn(v[u].y, b.y) >= 0.f ? 2u : 0u) |
                         (__fadd_rn(v[u].z, b.z) >= 0.f ? 4u : 0u) | (__fadd_rn(v[u].w, b.w) >= 0.f ? 8u : 0u);
            w <<= 4 * (lane & 7u);
            w |= __shfl_xor_sync(0xffffffffu, w, 1);
            w |= __shfl_xor_sync(0xffffffffu, w, 2);
            w |= __shfl_xor_sync(0xffffffffu, w, 4);
            if ((lane & 7u) == 0 && i < quads) __stcs(out + (i >> 3), w);
        }
    }
}

// General path: any C_in and replication factor R with R*C_in % 32 == 0.  A warp takes PACK_P pixels at a time (as many loads
// in flight) and walks their words; lane l evaluates channel c = 32*word + l, which reads input channel c mod C_in.  NV: where
// a lane meets only NV different input channels (C_in a divisor of 32: 1; 64: 2; 128: 4) they are read once per pixel, else
// (NV = 0) once per word.
constexpr int PACK_P = 8;
template <int NV>
__global__ void __launch_bounds__(256)
pack_general_kernel(const float *__restrict__ x, const float *__restrict__ bias, uint32_t *__restrict__ out, long npix, int C_in, int cwords)
{
    pdl_trigger();
    const int lane = threadIdx.x & 31;
    const long warp = (long)blockIdx.x * 8 + (threadIdx.x >> 5), nwarps = (long)gridDim.x * 8;
    const int adv = 32 % C_in;
    pdl_wait();
    for (long p0 = warp * PACK_P; p0 < npix; p0 += nwarps * PACK_P) {
        int ci = lane % C_in;
        float v[NV ? NV : 1][PACK_P];
        auto load = [&](float (&d)[PACK_P], int c) {
#pragma unroll
            for (int u = 0; u < PACK_P; ++u) d[u] = p0 + u < npix ? __ldg(x + (p0 + u) * C_in + c) : -1.f;
        };
        if (NV)
#pragma unroll
            for (int k = 0; k < NV; ++k) load(v[k], ci + 32 * k);
        for (int w0 = 0; w0 < cwords; w0 += NV ? NV : 1) {      // cwords is a multiple of NV
#pragma unroll
            for (int k = 0; k < (NV ? NV : 1); ++k) {
                const int w = w0 + k;
                if (!NV) load(v[0], ci);
                const float b = bias ? __ldg(bias + 32 * w + lane) : 0.f;
                uint32_t mine = 0;
#pragma unroll
                for (int u = 0; u < PACK_P; ++u) {
                    const uint32_t word = __ballot_sync(0xffffffffu, __fadd_rn(v[k][u], b) >= 0.f);
                    if (lane == u) mine = word;
                }
                if (lane < PACK_P && p0 + lane < npix) out[(p0 + lane) * cwords + w] = mine;
            }
            ci += adv;
            if (ci >= C_in) ci -= C_in;
        }
    }
}

// Stem path (Table 1 "stem replicate": 4 real channels replicated 8x to 32 sign channels): one
// thread per pixel reads its 4 values as one 16-byte load and emits the pixel's single 32-bit word.
//
// Fast path (all biases finite).  For finite b, fl(x + b) >= 0 exactly when x >= -b (a sum of two
// floats never rounds to zero unless it is zero, and NaN / infinite x behave the same on both sides),
// so input value i only has to be ranked among its 8 thresholds -b[4r+i]: they are sorted once per
// CTA, a 4-compare search counts how many are <= x, and a 9-entry table per input gives the bits.
// That is ~13 instructions per input value instead of 3 per output channel; the kernel becomes
// HBM-bound.  With a NaN or infinite bias (inf - inf = NaN -> -1) the plain per-channel path runs.
__global__ void __launch_bounds__(256)
pack_c4r8_kernel(const float4 *__restrict__ x, const float *__restrict__ bias,
                 uint32_t *__restrict__ out, long npix)
{
    pdl_trigger();
    pdl_wait();
    constexpr int U = 4;                       // pixels in flight per thread
    __shared__ float sb[32];
    __shared__ float sts[4][8];                // sorted thresholds of input i
    __shared__ uint32_t lut[4][9];             // bits set when c thresholds are <= x
    __shared__ int all_finite;
    if (threadIdx.x == 0) all_finite = 1;
    __syncthreads();
    if (threadIdx.x < 32) {
        const float b = bias ? bias[threadIdx.x] : 0.0f;
        sb[threadIdx.x] = b;
        if (!(fabsf(b) <= 3.402823466e38f)) all_finite = 0;      // NaN or infinity
    }
    __syncthreads();
    if (threadIdx.x < 4 && all_finite) {
        const int i = threadIdx.x;
        float t[8];
        int r[8];
        for (int k = 0; k < 8; ++k) { t[k] = -sb[4 * k + i]; r[k] = k; }
        for (int a = 1; a < 8; ++a)            // insertion sort, ascending
            for (int k = a; k > 0 && t[k] < t[k - 1]; --k) {
                const float tf = t[k]; t[k] = t[k - 1]; t[k - 1] = tf;
                const int ti = r[k]; r[k] = r[k - 1]; r[k - 1] = ti;
            }
        uint32_t m = 0;
        lut[i][0] = 0;
        for (int k = 0; k < 8; ++k) {
            sts[i][k] = t[k];
            m |= 1u << (4 * r[k] + i);
            lut[i][k + 1] = m;
        }
    }
    __syncthreads();
    const long stride = (long)gridDim.x * blockDim.x;
    if (all_finite) {
        float ts[4][8];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int k = 0; k < 8; ++k) ts[i][k] = sts[i][k];
        for (long p0 = (long)blockIdx.x * blockDim.x + threadIdx.x; p0 < npix; p0 += stride * U) {
            float4 v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long p = p0 + u * stride;
                v[u] = (p < npix) ? __ldcs(x + p) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const long p = p0 + u * stride;
                const float f[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
                uint32_t word = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float xv = f[i];
                    const bool pp = xv >= ts[i][3];
                    const bool qq = xv >= (pp ? ts[i][5] : ts[i][1]);
                    const float tl = pp ? (qq ? ts[i][6] : ts[i][4]) : (qq ? ts[i][2] : ts[i][0]);
                    const bool rr = xv >= tl;
                    const int c = (pp ? 4 : 0) + (qq ? 2 : 0) + (rr ? 1 : 0) + (xv >= ts[i][7] ? 1 : 0);
                    word |= lut[i][c];
                }
                if (p < npix) __stcs(out + p, word);
            }
        }
        return;
    }
    float b[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) b[c] = sb[c];
    for (long p0 = (long)blockIdx.x * blockDim.x + threadIdx.x; p0 < npix; p0 += stride * U) {
        float4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long p = p0 + u * stride;
            v[u] = (p < npix) ? __ldcs(x + p) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long p = p0 + u * stride;
            const float f[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
            uint32_t word = 0;
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                const float s = __fadd_rn(f[c & 3], b[c]);
                word |= (s >= 0.0f ? 1u : 0u) << c;
            }
            if (p < npix) __stcs(out + p, word);
        }
    }
}

int launch_pack(const float *x, const float *bias, uint32_t *out, long npix, int C_in, int R,
                cudaStream_t stream)
{
    const int C = C_in * R;
    const int cwords = C / 32;
    const long nwords = npix * cwords;
    const int sms = sm_count();
    const int threads = 256;
    if (R == 1 && C_in % 32 == 0) {
        const long quads = nwords * 8;
        const unsigned q = (unsigned)C_in / 4;
        long blocks = (quads + threads * PACK_U - 1) / (threads * PACK_U);
        const long cap = (long)sms * 8;
        if (blocks > cap) blocks = cap;
        // blocks such that a pass is a whole number of pixels
        unsigned m = q;                                  // q / gcd(q, 256)
        for (int i = 0; i < 8 && m % 2 == 0; ++i) m /= 2;
        const bool fixed = !bias || (long)m <= blocks;
        if (bias && fixed) blocks -= blocks % m;
        return launch(fixed ? pack_stream_kernel<true> : pack_stream_kernel<false>, (unsigned)blocks, threads, 0, stream,
                      reinterpret_cast<const float4 *>(x), reinterpret_cast<const float4 *>(bias), out, quads, q);
    } else if (C_in == 4 && R == 8) {
        long blocks = (npix + threads * 4 - 1) / (threads * 4);
        const long cap = (long)sms * blocks_per_sm((const void *)pack_c4r8_kernel, threads, 0);       // one wave of resident CTAs, grid-stride inside
        if (blocks > cap) blocks = cap;
        if (blocks < 1) blocks = 1;
        return launch(pack_c4r8_kernel, (unsigned)blocks, threads, 0, stream, reinterpret_cast<const float4 *>(x), bias, out, npix);
    } else {
        long blocks = (npix + 8 * PACK_P - 1) / (8 * PACK_P);
        const long cap = (long)sms * 8;
        if (blocks > cap) blocks = cap;
        auto k = 32 % C_in == 0 ? pack_general_kernel<1> : (C_in == 64 ? pack_general_kernel<2> : (C_in == 128 ? pack_general_kernel<4> : pack_general_kernel<0>));
        return launch(k, (unsigned)blocks, threads, 0, stream, x, bias, out, npix, C_in, cwords);
    }
}

}  // namespace bcnn
