// 4+4-bit quantiser of the voltage stream (precision variant of the voltage
// path; the paper itself works with unquantised voltages).
//
// Per channel: rms = sqrt(sum(re^2 + im^2) / (2 T N)) accumulated in FP64,
// scale = (float)(3 / rms) so that each component has an RMS of 3 levels,
// q = clip(round_half_away(x * scale), -7, 7) with the product rounded to
// float, byte = (q_re << 4) | (q_im & 15).  The FP64 sum is formed in a
// fixed order (block partials, then a sequential sum), so a channel's scale
// does not depend on the launch.
#include <algorithm>

#include "gc_f32x2.h"
#include "gc_internal.h"

namespace {

constexpr int kQThreads = 256;

// Running sums of squares of two neighbouring components as unevaluated triples
// s + c + d of floats.  The product x x is p + e (e its exact rounding error, by
// fma); p is added to s by the exact two-term sum (Knuth), its error and e to c
// likewise, and only what is left of those is rounded, in d: about 66 bits, more
// than an FP64 sum keeps.  (A pair s + c rounds e away: the low bits of squares
// are not symmetric, and sums came out 6e-16 low.)  Packed: 24 operations for two.
struct Sum3 {
    f2 s = 0, c = 0, d = 0;
    // a + b = t + the value returned
    static __device__ __forceinline__ f2 two_sum(f2 a, f2 b, f2 &t) {
        t = padd(a, b);
        const f2 z = psub(t, a);
        return padd(psub(a, psub(t, z)), psub(b, z));
    }
    __device__ __forceinline__ void square(float x0, float x1) {
        const float2 q = make_float2(__fmul_rn(x0, x0), __fmul_rn(x1, x1));
        const f2 p = p2(q.x, q.y), e = p2(__fmaf_rn(x0, x0, -q.x), __fmaf_rn(x1, x1, -q.y));
        const f2 r = two_sum(c, two_sum(s, p, s), c);
        d = padd(d, padd(two_sum(c, e, c), r));
    }
    __device__ __forceinline__ double value() const {
        const float2 x = u2(s), y = u2(c), z = u2(d);
        return ((double)x.x + ((double)y.x + z.x)) + ((double)x.y + ((double)y.y + z.y));
    }
};

// Each thread sums its squares in such triples, the threads' sums are added in
// FP64: rms error of a thread's sum of 256 squares 4e-17, 1e-15 with FP64
// additions.  An FP64 fma of every component is bound by this part's FP64 rate (1.05
// TFLOP/s, 1/74 of FP32): the whole quantiser takes 1357 us with it on 64 channels
// of 2048 x 1024 voltages (1.07 GB), 435 us so, near the HBM reads of both passes
// (109 and 53 us on a sixteenth of that, in L2, where the FP32 issue bounds it).
// Four loads a thread are in flight; four CTAs an SM leave the registers for them (435 us;
// 452 at three, 472 at five, which spills).
__global__ void __launch_bounds__(kQThreads, 4)
quant_sumsq(const float4 *__restrict__ v, size_t n4_per_ch, int nblk, double *__restrict__ part) {
    const int c = blockIdx.y, b = blockIdx.x;
    const float4 *src = v + (size_t)c * n4_per_ch;
    const size_t per = (n4_per_ch + nblk - 1) / nblk;
    const size_t lo = min(n4_per_ch, (size_t)b * per), hi = min(n4_per_ch, lo + per);
    constexpr int U = 4;
    Sum3 xy, zw;
    unsigned bits = 0u;   // of all values: 0 or the sign alone when all are zero
    auto take = [&](float4 q) {
        xy.square(q.x, q.y);
        zw.square(q.z, q.w);
        bits |= __float_as_uint(q.x) | __float_as_uint(q.y);
        bits |= __float_as_uint(q.z) | __float_as_uint(q.w);
    };
    size_t i = lo + threadIdx.x;
    for (; i + (U - 1) * kQThreads < hi; i += U * kQThreads) {
        float4 q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = src[i + u * kQThreads];
#pragma unroll
        for (int u = 0; u < U; ++u) take(q[u]);
    }
    for (; i < hi; i += kQThreads) take(src[i]);
    double s = xy.value() + zw.value();
    // sums near the ends of FP32's range (|x| above 1e17 or all below 1e-12,
    // non-finite values among them) are made in FP64; zeros are what they are
    if (!(s > 1e-24 && s < 1e34) && (bits & 0x7fffffffu) != 0u) {
        s = 0.0;
        for (size_t k = lo + threadIdx.x; k < hi; k += kQThreads) {
            const float4 q = src[k];
            s += (double)q.x * q.x + (double)q.y * q.y + (double)q.z * q.z + (double)q.w * q.w;
        }
    }
    __shared__ double red[kQThreads];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = kQThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[(size_t)c * nblk + b] = red[0];
}

__global__ void quant_scale(const double *__restrict__ part, int nblk, int C, double n_components,
                            float *__restrict__ scale) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    double s = 0.0;
    for (int b = 0; b < nblk; ++b) s += part[(size_t)c * nblk + b];
    const double rms = sqrt(s / n_components);
    scale[c] = rms > 0.0 ? (float)(3.0 / rms) : 0.0f;
}

__device__ __forceinline__ int q4(float x) {
    const float a = fabsf(x);
    float f = floorf(a);
    if (a - f >= 0.5f) f += 1.0f;
    int q = (int)f;
    q = q > 7 ? 7 : q;
    return x < 0.0f ? -q : q;
}

__global__ void __launch_bounds__(kQThreads)
quant_apply(const float4 *__restrict__ v, size_t n2_per_ch, int C, const float *__restrict__ scale,
            uint16_t *__restrict__ out) {
    // each thread packs two antenna-samples (one float4) into two bytes
    const size_t total = n2_per_ch * C;
    for (size_t i = blockIdx.x * (size_t)kQThreads + threadIdx.x; i < total; i += (size_t)gridDim.x * kQThreads) {
        const int c = (int)(i / n2_per_ch);
        const float s = scale[c];
        const float4 q = v[i];
        const int r0 = q4(__fmul_rn(q.x, s)), i0 = q4(__fmul_rn(q.y, s));
        const int r1 = q4(__fmul_rn(q.z, s)), i1 = q4(__fmul_rn(q.w, s));
        const unsigned b0 = ((unsigned)(r0 & 15) << 4) | (unsigned)(i0 & 15);
        const unsigned b1 = ((unsigned)(r1 & 15) << 4) | (unsigned)(i1 & 15);
        out[i] = (uint16_t)(b0 | (b1 << 8));
    }
}

}  // namespace

extern "C" gc_status gc_quantize(gc_ctx *ctx, const float *volt, int C, int T, int N, uint8_t *out, float *scales,
                                 void *stream) {
    if (!ctx) return GC_EINVAL;
    ctx->last_error.clear();
    if (!volt || !out) return gc_fail(ctx, GC_EINVAL, "gc_quantize: null buffer");
    if (C < 1 || T < 1 || N < 1 || ((size_t)T * N) % 2 != 0)
        return gc_fail(ctx, GC_EINVAL, "gc_quantize: need C, T, N >= 1 and T*N even");
    if (!gc_aligned(volt, 16) || !gc_aligned(out, 2) || (scales && !gc_aligned(scales, 4)))
        return gc_fail(ctx, GC_EINVAL, "gc_quantize: misaligned buffer");
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return gc_cuda_fail(ctx, e, "cudaSetDevice");
    const size_t n2 = (size_t)T * N / 2;        // float4 (two complex) per channel
    const int nblk = (int)std::max<size_t>(1, std::min<size_t>(64, n2 / 4096));
    const size_t need = (size_t)C * nblk * sizeof(double) + (size_t)C * sizeof(float) + 256;
    gc_status st = gc_scratch_reserve(ctx, need);
    if (st != GC_OK) return st;
    double *part = static_cast<double *>(ctx->scratch);
    float *sc = scales ? scales
                       : reinterpret_cast<float *>(static_cast<char *>(ctx->scratch) +
                                                   (((size_t)C * nblk * sizeof(double) + 255) / 256) * 256);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const float4 *v4 = reinterpret_cast<const float4 *>(volt);
    int rec = gc_prof_begin(ctx, s, "quant_sumsq");
    quant_sumsq<<<dim3(nblk, C), kQThreads, 0, s>>>(v4, n2, nblk, part);
    gc_prof_end(ctx, s, rec);
    quant_scale<<<(C + 127) / 128, 128, 0, s>>>(part, nblk, C, 2.0 * (double)T * N, sc);
    const size_t total = n2 * C;
    const int grid = (int)std::min<size_t>((total + kQThreads - 1) / kQThreads, (size_t)ctx->sm_count * 16);
    rec = gc_prof_begin(ctx, s, "quant_apply");
    quant_apply<<<grid, kQThreads, 0, s>>>(v4, n2, C, sc, reinterpret_cast<uint16_t *>(out));
    gc_prof_end(ctx, s, rec);
    e = cudaGetLastError();
    if (e != cudaSuccess) return gc_cuda_fail(ctx, e, "launch quantiser");
    return GC_OK;
}
