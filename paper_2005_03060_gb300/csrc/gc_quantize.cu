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

#include "gc_internal.h"

namespace {

constexpr int kQThreads = 256;

// Running sum of squares as an unevaluated pair s + c of floats: the product
// x x as p + e (e its exact rounding error, by fma), then the exact two-term
// sum of s and p (Knuth), with every rounding error collected in c.  About 44
// bits, ten FP32 operations a component.
struct Sum2 {
    float s = 0.f, c = 0.f;
    __device__ __forceinline__ void square(float x) {
        const float p = __fmul_rn(x, x), e = __fmaf_rn(x, x, -p);
        const float t = __fadd_rn(s, p), b = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(p, b)), e));
        s = t;
    }
};

// Squares summed per thread in float pairs, the threads' sums in FP64.  An
// FP64 fma of every component is bound by this part's FP64 rate (1.05 TFLOP/s,
// 1/74 of FP32): 1117 us for 64 channels of 2048 x 1024 voltages (1.07 GB)
// against 212 us for the pairs (5.1 TB/s), which the HBM read bounds.  Four loads a
// thread are in flight.
__global__ void __launch_bounds__(kQThreads)
quant_sumsq(const float4 *__restrict__ v, size_t n4_per_ch, int nblk, double *__restrict__ part) {
    const int c = blockIdx.y, b = blockIdx.x;
    const float4 *src = v + (size_t)c * n4_per_ch;
    const size_t per = (n4_per_ch + nblk - 1) / nblk;
    const size_t lo = min(n4_per_ch, (size_t)b * per), hi = min(n4_per_ch, lo + per);
    constexpr int U = 4;
    Sum2 acc[4];   // one per component of the float4: independent chains
    size_t i = lo + threadIdx.x;
    for (; i + (U - 1) * kQThreads < hi; i += U * kQThreads) {
        float4 q[U];
#pragma unroll
        for (int u = 0; u < U; ++u) q[u] = src[i + u * kQThreads];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            acc[0].square(q[u].x);
            acc[1].square(q[u].y);
            acc[2].square(q[u].z);
            acc[3].square(q[u].w);
        }
    }
    for (; i < hi; i += kQThreads) {
        const float4 q = src[i];
        acc[0].square(q.x);
        acc[1].square(q.y);
        acc[2].square(q.z);
        acc[3].square(q.w);
    }
    double s = 0.0;
    bool fine = true;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        // squares near the ends of FP32's range (|x| above 1e17 or all below
        // 1e-12, zeros and non-finite values among them) are summed in FP64
        fine = fine && acc[k].s > 1e-24f && acc[k].s < 1e34f;
        s += (double)acc[k].s + (double)acc[k].c;
    }
    if (!fine) {
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
