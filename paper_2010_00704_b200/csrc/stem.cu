// Fused stem: binarize + pack (Section 4.2.1 bias + sign, Table 1 "stem replicate": 4 real channels
// replicated 8x to 32 sign channels) followed by the first binary 1x1 convolution (32 -> 32 channels)
// with its threshold epilogue, in one pass over the real input.  The 32-channel sign tensor is never
// written: per pixel the kernel reads 16 bytes and writes the 4 bytes of the convolution's packed output.
//
// Why a table.  Sign channel c = 4r + i is (x_i + bias_c >= 0): the 8 replicas of real channel i are a
// thermometer code of x_i against its 8 thresholds -bias, so a pixel's 32 sign bits are fixed by four
// levels c_i in 0..8 (how many thresholds of channel i are <= x_i): 9^4 = 6561 distinct sign words.  The
// whole 1x1 layer - K - 2 popc(word XOR w_n) >= thr_n for the 32 outputs n - is therefore a function of
// e = c_0 + 9 c_1 + 81 c_2 + 729 c_3, tabulated once per CTA in shared memory (26 KB); the pixel loop is
// the level search of the pack kernel plus one table read.  The result is bit-identical to bcnn_pack
// followed by bcnn_conv2d_b1_fused.
//
// Table build (per CTA, ~2 us): mismatches split as popc over channels {0,1} + popc over channels {2,3};
// two 81-entry tables of 32 byte fields (one per output n: word n % 8, byte n / 8) are added word-wise; the first
// carries 127 - theta_n, theta_n = floor((32 - thr_n) / 2) clamped to [-1, 32], so that bit 7 of field n
// is set exactly when mismatches > theta_n, i.e. when the output bit is 0.  The thresholds are ranked by 32 lanes at once.
//
// Bound by memory (16 bytes per pixel in, 4 out).  A thread that loads its own pixels has nothing in flight while it computes
// (about 70 instructions a pixel, half of the time), so the pixels arrive by bulk copies into a ring in shared memory: 155 KB
// in flight per multiprocessor, the first of them while the tables are built.  256 images of 224 x 224: 51.5 us with loads by
// the threads, 46.3 with the ring, 42.5 - 43.8 (5.9 - 6.05 TB/s; a copy reaches 6.5) with the shorter table build; 16 images 9.6 -> 7.9.
//
// The table pays for itself only when a CTA has many pixels: up to PLAIN_PIXELS per multiprocessor the plain per-channel path
// runs in a kernel of its own, spread over all of them (one 224 x 224 image 2.5 us against 6.0, four 5.4 against 6.1).
// With a NaN or infinite bias the thermometer argument fails (inf - inf = NaN -> -1): the plain
// per-channel path runs instead (32 fp32 adds + compares, 32 popcounts per pixel).
#include "bcnn_common.cuh"
#include "tc_slot.cuh"

namespace bcnn {

using namespace tc;

namespace {

constexpr int STEM_THREADS = 1024;         // 31 warps that compute, a loader warp
constexpr int STEM_WORKERS = STEM_THREADS - 32;
constexpr int STEM_U = 2;                  // pixels of a thread per chunk
constexpr int STEM_CHUNK = STEM_U * STEM_WORKERS;      // pixels per bulk copy
constexpr int STEM_RING = 5;
constexpr int STEM_RING_BYTES = STEM_RING * STEM_CHUNK * 16;
constexpr int ERR_STEM_LOADER_TIMEOUT = 181;     // loader: a chunk was not consumed
constexpr int ERR_STEM_WORKER_TIMEOUT = 182;     // worker: a chunk did not arrive
constexpr long PLAIN_PIXELS = 2304;        // per multiprocessor (crossover: seven 224 x 224 images, 6.9 us either way)
constexpr int STEM_LEVELS = 9 * 9 * 9 * 9;

// One pixel, every sign channel evaluated as written, then 32 XOR + popcount.
__device__ __forceinline__ uint32_t stem_pixel(const float4 &v, const float *sb, const uint32_t *sw, const int *stheta)
{
    const float f[4] = {v.x, v.y, v.z, v.w};
    uint32_t word = 0;
#pragma unroll
    for (int c = 0; c < 32; ++c) {
        const float s = __fadd_rn(f[c & 3], sb[c]);
        word |= (s >= 0.0f ? 1u : 0u) << c;
    }
    uint32_t o = 0;
#pragma unroll 8
    for (int n = 0; n < 32; ++n) o |= (__popc(word ^ sw[n]) <= stheta[n] ? 1u : 0u) << n;
    return o;
}
// out bit n = (32 - 2*mism >= thr)  <=>  mism <= floor((32 - thr) / 2)
__device__ __forceinline__ int stem_theta(int thr)
{
    const long long th = (32LL - (long long)thr) >> 1;
    return (int)(th < -1 ? -1 : (th > 32 ? 32 : th));
}

__global__ void __launch_bounds__(256)
stem_plain_kernel(const float4 *__restrict__ x, const float *__restrict__ bias, const uint32_t *__restrict__ w,
                  const int32_t *__restrict__ thr, uint32_t *__restrict__ out, long npix)
{
    __shared__ float sb[32];
    __shared__ uint32_t sw[32];
    __shared__ int stheta[32];
    pdl_trigger();
    const long p = (long)blockIdx.x * 256 + threadIdx.x;
    pdl_wait();
    const float4 v = p < npix ? __ldcs(x + p) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (threadIdx.x < 32) {
        sb[threadIdx.x] = bias ? bias[threadIdx.x] : 0.0f;
        sw[threadIdx.x] = w[threadIdx.x];
        stheta[threadIdx.x] = stem_theta(thr[threadIdx.x]);
    }
    __syncthreads();
    if (p < npix) __stcs(out + p, stem_pixel(v, sb, sw, stheta));
}

__global__ void __launch_bounds__(STEM_THREADS, 1)
stem_c4r8_k32_kernel(const float4 *__restrict__ x, const float *__restrict__ bias, const uint32_t *__restrict__ w,
                     const int32_t *__restrict__ thr, uint32_t *__restrict__ out, long npix, int *err)
{
    extern __shared__ __align__(16) unsigned char ring_raw[];   // [STEM_RING][STEM_CHUNK] pixels
    __shared__ __align__(8) unsigned long long bars[2 * STEM_RING];
    __shared__ int abort_flag_smem;
    __shared__ float sb[32];
    __shared__ float sts[4][8];                 // sorted thresholds of input i
    __shared__ uint32_t lut[4][9];              // sign bits of input i set at level c
    __shared__ uint32_t sw[32];                 // weight word of output n
    __shared__ int stheta[32];
    __shared__ __align__(16) uint32_t ta[81][8];  // byte field n: 127 - theta_n + mismatches over channels {0, 1}
    __shared__ __align__(16) uint32_t tb[81][8];  // byte field n: mismatches over channels {2, 3}
    __shared__ uint32_t table[STEM_LEVELS];     // output word of the level tuple e
    __shared__ int all_finite;

    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t ring = smem_u32(ring_raw), bar0 = smem_u32(bars);
    auto full = [&](int st) { return bar0 + 8u * st; };
    auto empty = [&](int st) { return bar0 + 8u * (STEM_RING + st); };
    volatile int *abort_flag = &abort_flag_smem;
    // this CTA's chunks: blockIdx.x + k * gridDim.x
    const long chunks = (npix + STEM_CHUNK - 1) / STEM_CHUNK;
    auto load = [&](long c, int st) {           // one thread
        const long left = npix - c * STEM_CHUNK;
        const uint32_t bytes = (uint32_t)(left < STEM_CHUNK ? left : STEM_CHUNK) * 16u;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full(st)), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(ring + (uint32_t)(st * STEM_CHUNK * 16)), "l"(x + c * STEM_CHUNK), "r"(bytes), "r"(full(st)) : "memory");
    };
    if (tid == 0) {
        abort_flag_smem = 0;
        for (int st = 0; st < STEM_RING; ++st) {
            mbar_init(full(st), 1);             // the loader's arrive (+ the copy's bytes)
            mbar_init(empty(st), STEM_WORKERS / 32);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    pdl_trigger();
    pdl_wait();
    // the first chunks arrive while the tables are built
    if (tid == STEM_WORKERS)
        for (int k = 0; k < STEM_RING && (long)blockIdx.x + (long)k * gridDim.x < chunks; ++k) load(blockIdx.x + (long)k * gridDim.x, k);
    if (tid < 32) {
        const float b = bias ? bias[tid] : 0.0f;
        sb[tid] = b;
        sw[tid] = w[tid];
        stheta[tid] = stem_theta(thr[tid]);
        const bool finite = __all_sync(0xffffffffu, fabsf(b) <= 3.402823466e38f);      // no NaN or infinity
        if (tid == 0) all_finite = finite;
        // rank of sign channel tid = 4 k + i among the eight thresholds of input i; a level's sign bits are then a vote
        const float t = -b;
        int rank = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int other = 4 * k + (tid & 3);
            const float o = __shfl_sync(0xffffffffu, t, other);
            rank += (o < t || (o == t && other < tid)) ? 1 : 0;
        }
        sts[tid & 3][rank] = t;
#pragma unroll
        for (int c = 0; c <= 8; ++c) {
            const uint32_t m = __ballot_sync(0xffffffffu, rank < c);
            if (tid < 4) lut[tid][c] = m & (0x11111111u << tid);
        }
    }
    __syncthreads();
    // the two half tables: entry (c_lo + 9 c_hi), output n -> one byte
    for (int idx = tid; idx < 2 * 81 * 32; idx += STEM_THREADS) {
        const int half = idx / (81 * 32), rem = idx - half * (81 * 32);
        const int e = rem >> 5, n = rem & 31;
        const int clo = e % 9, chi = e / 9;
        const uint32_t word = lut[2 * half][clo] | lut[2 * half + 1][chi];
        const uint32_t mask = half ? 0xCCCCCCCCu : 0x33333333u;    // sign channels c with c % 4 in {2,3} / {0,1}
        int v = __popc((word ^ sw[n]) & mask);
        if (half == 0) v += 127 - stheta[n];
        unsigned char *dst = reinterpret_cast<unsigned char *>(half ? &tb[e][0] : &ta[e][0]);
        dst[4 * (n & 7) + (n >> 3)] = (unsigned char)v;                // word n % 8, byte n / 8
    }
    __syncthreads();
    for (int e = tid; e < STEM_LEVELS; e += STEM_THREADS) {
        const int e01 = e % 81, e23 = e / 81;
        uint32_t o = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t v = ta[e01][k] + tb[e23][k];            // fields stay below 256: no carries between them
            o |= ~(v >> (7 - k)) & (0x01010101u << k);                 // bit 7 of byte j of word k clear -> output bit 8j + k set
        }
        table[e] = o;
    }
    __syncthreads();

    if (warp == STEM_WORKERS / 32) {
        // ---- loader: refills a stage once the workers have read it
        int k = 0;
        for (long c = blockIdx.x; c < chunks; c += gridDim.x, ++k) {
            if (k < STEM_RING) continue;        // on its way since the start
            if (!pw_wait<64>(empty(k % STEM_RING), (uint32_t)(k / STEM_RING - 1) & 1u, abort_flag, err, ERR_STEM_LOADER_TIMEOUT)) break;
            if (tid == STEM_WORKERS) load(c, k % STEM_RING);
            __syncwarp();
        }
        // after a time-out elsewhere: copies still in flight must land before the CTA's shared memory goes away
        if (*abort_flag)
            for (int q = k > STEM_RING ? k - STEM_RING : 0; q < k; ++q)
                pw_wait(full(q % STEM_RING), (uint32_t)(q / STEM_RING) & 1u, abort_flag, nullptr, 0);
        return;
    }
    // ---- workers: chunk k of this CTA, STEM_U pixels per thread
    const uint32_t lane0 = (tid & 31) == 0 ? 1u : 0u;
    auto walk = [&](auto pixel) {
        int k = 0;
        for (long c = blockIdx.x; c < chunks; c += gridDim.x, ++k) {
            const int stage = k % STEM_RING;
            if (!pw_wait(full(stage), (uint32_t)(k / STEM_RING) & 1u, abort_flag, err, ERR_STEM_WORKER_TIMEOUT)) return;
            float4 v[STEM_U];
#pragma unroll
            for (int u = 0; u < STEM_U; ++u)    // (what lies beyond the last pixel is read and not used)
                asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v[u].x), "=f"(v[u].y), "=f"(v[u].z), "=f"(v[u].w)
                             : "r"(ring + (uint32_t)((stage * STEM_CHUNK + u * STEM_WORKERS + tid) * 16)) : "memory");
            const long p0 = c * STEM_CHUNK + tid;
#pragma unroll
            for (int u = 0; u < STEM_U; ++u) {
                const uint32_t o = pixel(v[u]);
                if (p0 + u * STEM_WORKERS < npix) __stcs(out + p0 + u * STEM_WORKERS, o);
            }
            // The stage may be refilled: its words have been used.  (With the arrival right behind the loads a refill can overtake
            // them: seen in conv_tc_pn.cu, a few rows wrong in one launch of fifteen.)
            __syncwarp();
            mbar_arrive_pred(empty(stage), lane0);
        }
    };
    if (!all_finite) {
        walk([&](const float4 &v) { return stem_pixel(v, sb, sw, stheta); });
        return;
    }
    float ts[4][8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int k = 0; k < 8; ++k) ts[i][k] = sts[i][k];
    walk([&](const float4 &v) {
        const float f[4] = {v.x, v.y, v.z, v.w};
        // level of value i = how many of its sorted thresholds are <= x: eight compares that yield 1.0f / 0.0f
        // and a sum on the fp32 pipe (cheaper than a search made of selects on the integer pipe); the tuple index
        // c_0 + 9 c_1 + 81 c_2 + 729 c_3 <= 6560 is exact in fp32
        float ef = 0.0f;
#pragma unroll
        for (int i = 3; i >= 0; --i) {
            const float xv = f[i];
            float c = 0.0f;
#pragma unroll
            for (int k = 0; k < 8; ++k) c += (xv >= ts[i][k]) ? 1.0f : 0.0f;
            ef = fmaf(ef, 9.0f, c);
        }
        return table[__float2int_rn(ef)];
    });
}

}  // namespace

int launch_stem_c4r8_k32(const float *x, const float *bias, const uint32_t *w, const int32_t *thr, uint32_t *out,
                         long npix, cudaStream_t stream)
{
    const int sms = sm_count();
    if (npix <= sms * PLAIN_PIXELS)
        return launch(stem_plain_kernel, (unsigned)((npix + 255) / 256), 256, 0, stream, reinterpret_cast<const float4 *>(x), bias, w, thr, out, npix);
    long blocks = (npix + STEM_CHUNK - 1) / STEM_CHUNK;
    if (blocks > sms) blocks = sms;             // one resident CTA per SM builds the table once
    if (!allow_smem((const void *)stem_c4r8_k32_kernel, STEM_RING_BYTES)) return BCNN_ERR_CUDA;
    return launch(stem_c4r8_k32_kernel, (unsigned)blocks, STEM_THREADS, STEM_RING_BYTES, stream, reinterpret_cast<const float4 *>(x), bias, w, thr, out, npix,
                  device_error_word());
}

}  // namespace bcnn
