// Reduced X-engine over pair lists (paper Fig. 1, calibrator step (a); Sec. 4):
// selections with several integration windows, i.e. low-cadence calibration,
// where every baseline-type of the array is correlated in one of many short
// windows.
//
// One CTA takes (channel, window, block of the window's entries, time slice).
// The window's entries are listed once per selection: its pairs, ordered so
// that half a warp reads distinct banks, and then one entry (j, j) per
// antenna, whose sum is the window's autocorrelation.  A thread owns up to KP
// entries, holds their shared-memory offsets and sums in registers, and walks
// the samples, which TMA stages (two buffers; grid rows on a padded pitch
// where the plain one would repeat the banks).
//
// Why lists: owning antennas instead (xeng_accumulate) leaves lanes idle
// wherever j + d falls off the grid, three quarters of them over all types of
// a square array, and re-stages the samples per group of 16 types.  What
// bounds this form is shared-memory bandwidth, two operand reads a product:
// 32x32 antennas, 64 channels of 4096 complex64 samples (2.6e9 products) need
// 1.13 ms of reads at 128 B/clk/SM.  Measured there: 1890 us (2650 us with the
// pairs in type order, where bank conflicts were 41 % of the wavefronts),
// 4450 us for the antenna form with its separate slice sum.
//
// 4+4-bit voltages are expanded per stage into signed-byte words for dp4a, two
// samples a word as in xeng_accumulate (W for the first member, W and Wx for
// the second), in planes of 8 bytes per antenna so that consecutive antennas
// fall on distinct banks; sums are exact int32.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "gc_sel.h"

namespace {

constexpr int kPThreads = 512;

struct PParams {
    const unsigned char *volt;   // [C][T][N]
    int L, N, C, T, P;
    int pitch;                   // elements per grid row in what the products read
    int n_windows, n_blk, per_blk, n_tsplit, n_items;
    int ns;                      // samples per stage
    int autos;                   // 1: the (j, j) entries too
    const int32_t *wp_entry;     // window entries: pair index q < P, or P + antenna
    const int32_t *wp_off;       // [n_windows + 1]
    const int32_t *win_t0, *win_t1;   // [n_windows]
    const int32_t *pair_i, *pair_j;
    void *out;                   // [n_tsplit][C][P] float2 / int2 (V^reduced itself with one slice)
    void *apart;                 // [n_windows * n_tsplit][C][N] float / int, or null
    unsigned int *status;
    size_t stage_stride;
    int use_tma;                 // 0 plain loads, 1 bulk copies, 2 tiled copies (padded rows)
};

template <int VF, int KP>
__global__ void __launch_bounds__(kPThreads) xeng_pairs(const __grid_constant__ CUtensorMap tmap, const PParams p) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint64_t bars[2];
    __shared__ int s_err;
    constexpr bool kI4 = VF == GC_I4C;
    constexpr int esz = VF == GC_C64 ? 8 : (VF == GC_C32H ? 4 : 1);
    constexpr int kOff = kI4 ? 8 : esz;   // bytes per antenna in what the products read
    const int tid = threadIdx.x, nt = blockDim.x, N = p.N;
    const size_t sample_bytes = (size_t)N * esz;
    const unsigned staged = p.use_tma == 2 ? (unsigned)(p.L * p.pitch * esz) : (unsigned)sample_bytes;   // per sample
    // 4+4-bit: planes [sample quad][W | Wx][antenna] of 8 bytes after the raw stages
    unsigned char *planes = smem + 2 * p.stage_stride;
    const unsigned plane = 8u * (unsigned)(p.L * p.pitch);
    if (tid == 0) {
        s_err = 0;
        gc_mbar_init(&bars[0], 1);
        gc_mbar_init(&bars[1], 1);
        gc_fence_mbar_init();
    }
    __syncthreads();
    uint32_t ld_count = 0, use_count = 0;

    for (int item = blockIdx.x; item < p.n_items; item += gridDim.x) {
        // time slice fastest, then block, window, channel: blocks of one
        // window share its samples in L2
        const int ts = item % p.n_tsplit;
        const int b = (item / p.n_tsplit) % p.n_blk;
        const int w = (item / (p.n_tsplit * p.n_blk)) % p.n_windows;
        const int c = item / (p.n_tsplit * p.n_blk * p.n_windows);
        const int w0 = p.win_t0[w], w1 = p.win_t1[w];
        const int len = (w1 - w0 + p.n_tsplit - 1) / p.n_tsplit;
        const int ta = min(w1, w0 + ts * len), tb = min(w1, ta + len);
        const int e0 = p.wp_off[w] + b * p.per_blk;
        const int e1 = min(p.wp_off[w + 1] - (p.autos ? 0 : N), e0 + p.per_blk);
        const unsigned char *vc = p.volt + (size_t)c * p.T * sample_bytes;
        const int n_st = (tb - ta + p.ns - 1) / p.ns;
        auto issue = [&](int t) {
            const uint32_t bb = ld_count & 1u;
            if (p.use_tma == 2) {   // whole boxes: what lies past a row or past T is zero filled
                gc_mbar_expect_tx(&bars[bb], staged * p.ns);
                gc_tma_load_4d(smem + bb * p.stage_stride, &tmap, &bars[bb], 0, 0, t, c);
            } else {
                const uint32_t bytes = (uint32_t)(min(p.ns, tb - t) * sample_bytes);
                gc_mbar_expect_tx(&bars[bb], bytes);
                gc_bulk_load(smem + bb * p.stage_stride, vc + (size_t)t * sample_bytes, bytes, &bars[bb]);
            }
            ++ld_count;
        };
        if (e0 >= e1) continue;   // uniform: the last window may be shorter
        if (p.use_tma && tid == 0)
            for (int k = 0; k < 2 && k < n_st; ++k) issue(ta + k * p.ns);
        // this thread's entries: offsets of both members, zero sums (entries
        // past the end read antenna 0 and are not stored)
        unsigned oi[KP], oj[KP];
        float2 acc[kI4 ? 1 : KP];
        int ire[kI4 ? KP : 1], iim[kI4 ? KP : 1];
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            const int e = e0 + tid + k * nt;
            int i = 0, j = 0;
            if (e < e1) {
                const int q = p.wp_entry[e];
                i = q < p.P ? p.pair_i[q] : q - p.P;
                j = q < p.P ? p.pair_j[q] : q - p.P;
            }
            oi[k] = (unsigned)((i + (p.pitch - p.L) * (i / p.L)) * kOff);
            oj[k] = (unsigned)((j + (p.pitch - p.L) * (j / p.L)) * kOff);
            if constexpr (kI4) {
                ire[k] = 0;
                iim[k] = 0;
            } else {
                acc[k] = make_float2(0.f, 0.f);
            }
        }
        for (int st = 0; st < n_st; ++st) {
            const int t = ta + st * p.ns;
            const int cnt = min(p.ns, tb - t);
            const unsigned char *stage = smem;
            if (p.use_tma) {
                const uint32_t bb = use_count & 1u;
                stage = smem + bb * p.stage_stride;
                if (!gc_mbar_wait(&bars[bb], (use_count >> 1) & 1u, GC_WAIT_LIMIT_NS)) {
                    atomicOr(p.status, GC_DEV_TIMEOUT_XENG);
                    s_err = 1;
                } else {
                    ++use_count;
                }
                __syncthreads();
                if (s_err) break;
            } else {
                const size_t bytes = cnt * sample_bytes;
                const unsigned char *src = vc + (size_t)t * sample_bytes;
                if constexpr (VF == GC_C64) {
                    for (size_t i = tid; i < bytes / 8; i += nt)
                        reinterpret_cast<uint2 *>(smem)[i] = reinterpret_cast<const uint2 *>(src)[i];
                } else if constexpr (VF == GC_C32H) {
                    for (size_t i = tid; i < bytes / 4; i += nt)
                        reinterpret_cast<uint32_t *>(smem)[i] = reinterpret_cast<const uint32_t *>(src)[i];
                } else {
                    for (size_t i = tid; i < bytes; i += nt) smem[i] = src[i];
                }
                __syncthreads();
            }
            if constexpr (kI4) {
                // signed-byte words of four samples per antenna (zero past cnt)
                for (int u = tid; u < N * ((cnt + 3) / 4); u += nt) {
                    const int qd = u / N, a = u - qd * N;
                    uint32_t X = 0u;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (4 * qd + i < cnt) X |= (uint32_t)stage[(size_t)(4 * qd + i) * N + a] << (8 * i);
                    // (n ^ 8) + 0x78 never carries out of a byte and ^ 0x80 turns
                    // it into n as int8; 0x88 - (n ^ 8), then ^ 0x80, gives -n
                    const uint32_t ux = (X & 0x0F0F0F0Fu) ^ 0x08080808u;
                    const uint32_t vx = ((X >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
                    const uint32_t im = (ux + 0x78787878u) ^ 0x80808080u;
                    const uint32_t nim = (0x88888888u - ux) ^ 0x80808080u;
                    const uint32_t re = (vx + 0x78787878u) ^ 0x80808080u;
                    unsigned char *dst = planes + (size_t)(2 * qd) * plane + 8 * (a + (p.pitch - p.L) * (a / p.L));
                    *reinterpret_cast<uint2 *>(dst) =
                        make_uint2(__byte_perm(re, im, 0x5140), __byte_perm(re, im, 0x7362));
                    *reinterpret_cast<uint2 *>(dst + plane) =
                        make_uint2(__byte_perm(nim, re, 0x5140), __byte_perm(nim, re, 0x7362));
                }
                __syncthreads();
                if (p.use_tma && tid == 0 && st + 2 < n_st) {   // the raw stage is free again
                    gc_fence_proxy_async();
                    issue(ta + (st + 2) * p.ns);
                }
                for (int qd = 0; qd < (cnt + 3) / 4; ++qd) {
                    const unsigned char *W = planes + (size_t)(2 * qd) * plane, *X = W + plane;
#pragma unroll
                    for (int k = 0; k < KP; ++k) {
                        const int2 wi = *reinterpret_cast<const int2 *>(W + oi[k]);
                        const int2 wj = *reinterpret_cast<const int2 *>(W + oj[k]);
                        const int2 xj = *reinterpret_cast<const int2 *>(X + oj[k]);
                        ire[k] = __dp4a(wi.y, wj.y, __dp4a(wi.x, wj.x, ire[k]));
                        iim[k] = __dp4a(wi.y, xj.y, __dp4a(wi.x, xj.x, iim[k]));
                    }
                }
                __syncthreads();
            } else {
                for (int u = 0; u < cnt; ++u) {
                    const unsigned char *sv = stage + u * staged;
#pragma unroll
                    for (int k = 0; k < KP; ++k) {
                        float2 a, v;
                        if constexpr (VF == GC_C64) {
                            a = *reinterpret_cast<const float2 *>(sv + oi[k]);
                            v = *reinterpret_cast<const float2 *>(sv + oj[k]);
                        } else {
                            a = __half22float2(*reinterpret_cast<const __half2 *>(sv + oi[k]));
                            v = __half22float2(*reinterpret_cast<const __half2 *>(sv + oj[k]));
                        }
                        // a * conj(v)
                        acc[k].x = fmaf(a.x, v.x, fmaf(a.y, v.y, acc[k].x));
                        acc[k].y = fmaf(a.y, v.x, fmaf(-a.x, v.y, acc[k].y));
                    }
                }
                __syncthreads();
                if (p.use_tma && tid == 0 && st + 2 < n_st) {
                    gc_fence_proxy_async();
                    issue(ta + (st + 2) * p.ns);
                }
            }
        }
        if (s_err) break;
        const size_t orow = ((size_t)ts * p.C + c) * p.P, arow = ((size_t)(w * p.n_tsplit + ts) * p.C + c) * N;
#pragma unroll
        for (int k = 0; k < KP; ++k) {
            const int e = e0 + tid + k * nt;
            if (e >= e1) continue;
            const int q = p.wp_entry[e];
            if constexpr (kI4) {
                if (q < p.P) static_cast<int2 *>(p.out)[orow + q] = make_int2(ire[k], iim[k]);
                else static_cast<int *>(p.apart)[arow + q - p.P] = ire[k];
            } else if (q < p.P) {
                if (!isfinite(acc[k].x) || !isfinite(acc[k].y)) atomicOr(p.status, GC_DEV_BADINPUT);
                static_cast<float2 *>(p.out)[orow + q] = acc[k];
            } else {
                static_cast<float *>(p.apart)[arow + q - p.P] = acc[k].x;
            }
        }
    }
    if (p.use_tma && s_err && tid == 0) {
        // copies still in flight land before the CTA exits (bounded)
        while (use_count < ld_count) {
            gc_mbar_wait(&bars[use_count & 1u], (use_count >> 1) & 1u, GC_WAIT_LIMIT_NS / 10);
            ++use_count;
        }
    }
}

// Entries per thread.  22 is the most whose offsets and sums fit 128 registers (the
// limit at 512 threads): 23 spill in every format.
constexpr int kKp[] = {22, 16, 12, 8, 4};

template <int VF>
const void *pick_pairs(int kp) {
    switch (kp) {
        case 22: return (const void *)xeng_pairs<VF, 22>;
        case 16: return (const void *)xeng_pairs<VF, 16>;
        case 12: return (const void *)xeng_pairs<VF, 12>;
        case 8: return (const void *)xeng_pairs<VF, 8>;
        default: return (const void *)xeng_pairs<VF, 4>;
    }
}

int elem_size(int vfmt) { return vfmt == GC_C64 ? 8 : (vfmt == GC_C32H ? 4 : 1); }

// samples per stage: up to 16 in 32 KB of raw voltages; for 4+4 bits up to 32,
// whole quads, whose expanded words take 32 KB
int stage_samples(int vfmt, size_t sample_bytes) {
    if (vfmt == GC_I4C) return 4 * (int)std::max<size_t>(1, std::min<size_t>(8, 2048 / sample_bytes));
    return (int)std::max<size_t>(1, std::min<size_t>(16, (32u << 10) / sample_bytes));
}

// Padded rows: complex64 through a tiled copy (rows of whole 16-byte units), the
// expanded words of 4+4 bits always; binary16 pairs are staged as they are.
int pairs_pitch(int vfmt, int L) { return vfmt == GC_C32H ? L : gc_xeng_pairs_pitch(L); }

size_t pairs_smem(int vfmt, int L, size_t &stride) {
    const int pitch = pairs_pitch(vfmt, L);
    const size_t sample = (size_t)L * (vfmt == GC_C64 ? pitch : L) * elem_size(vfmt);
    const int ns = stage_samples(vfmt, (size_t)L * L * elem_size(vfmt));
    stride = (sample * ns + 127) / 128 * 128;
    return 2 * stride + (vfmt == GC_I4C ? (size_t)(ns / 4) * 16 * L * pitch : 0);
}

}  // namespace

// Several windows, and two samples of the grid fit the stages.  Not: binary16 on
// rows of a multiple of 32 (staged as they lie, columns share banks) where few
// channels have long windows -- 32x32 antennas, 4096 samples, one channel 111 us,
// 91 in the antenna form; two 181 and 168; four 316 and 322.
bool gc_xeng_pairs_eligible(const gc_ctx *ctx, const gc_sel *sel, int vfmt, int C) {
    size_t stride;
    if (sel->masked && sel->nbr.empty()) return false;   // refused without the pair table
    if (sel->wp_entry.empty() || pairs_smem(vfmt, sel->L, stride) > 200u * 1024u) return false;
    return !(vfmt == GC_C32H && sel->L % 32 == 0 && (long)C * sel->n_windows < ctx->sm_count && sel->t_int >= 64);
}

// Staged by copy engines: whole 16-byte units a sample.
bool gc_xeng_pairs_bulk(const gc_sel *sel, int vfmt, const void *volt) {
    return gc_aligned(volt, 16) && ((size_t)sel->L * sel->L * elem_size(vfmt)) % 16 == 0;
}

namespace {

// Entries per thread, threads and blocks of a window of `most` entries in at
// least `least` blocks: the fewest idle slots among the shapes of at least 128
// threads (more entries a thread hide the read latency better and are listed
// first); a window past 512 threads is split into blocks.
void pairs_blocks(int most, int least, gc_xeng_pairs_shape *sh) {
    const int per1 = (most + least - 1) / least;
    sh->kp = 4;
    sh->nthr = std::min(kPThreads, std::max(32, ((per1 + 3) / 4 + 31) / 32 * 32));
    long best = -1;
    for (int kp : kKp) {
        const int nb = std::max(least, (most + kPThreads * kp - 1) / (kPThreads * kp));
        const int per = (most + nb - 1) / nb;
        const int nthr = ((per + kp - 1) / kp + 31) / 32 * 32;
        if (nthr < 128 && kp > 4) continue;
        const long slots = (long)nb * nthr * kp;
        if (best < 0 || slots < best) {
            best = slots;
            sh->kp = kp;
            sh->nthr = nthr;
        }
    }
    sh->per_blk = sh->nthr * sh->kp;
    sh->n_blk = (most + sh->per_blk - 1) / sh->per_blk;
}

// Cycles that a reduction whose items all fit the chip takes in ts time slices: an
// item's start (first copies, then entry lists and scattered stores), its samples,
// each with the products' latency, the shared-memory reads of the SM's `live` CTAs
// at 128 B a cycle (16, 8 or 6 bytes an entry) and what the threads themselves
// stage or expand; then the partial sums of the slices, and the autocorrelations
// of all windows and slices.  The constants are from runs of few channels, 3x3 to 32x32 antennas.
double pairs_cycles(const gc_sel *sel, int vfmt, int C, int sms, int max_win, bool bulk, const gc_xeng_pairs_shape &sh,
                    int ts) {
    const int N = sel->L * sel->L;
    const double bytes = vfmt == GC_C64 ? 16.0 : (vfmt == GC_C32H ? 8.0 : 6.0);
    const double live = (double)(((long)C * sel->n_windows * sh.n_blk * ts + sms - 1) / sms);
    double sample = 150.0 + live * sh.per_blk * bytes / 128.0;
    if (vfmt == GC_I4C) sample += 100.0 + 8.0 * N / sh.nthr;
    if (!bulk) sample += 20.0 * N / sh.nthr;
    double t = 5000.0 + 2.5 * live * sh.per_blk + (double)((max_win + ts - 1) / ts) * sample;
    if (ts > 1) t += 100.0 * ts + (double)ts * C * sel->P * 16.0 / 3500.0;
    return t + 40.0 * ts * sel->n_windows;
}

}  // namespace

gc_status gc_xeng_pairs_plan(gc_ctx *ctx, const gc_sel *sel, int vfmt, int C, bool autos, bool bulk, gc_xeng_pairs_shape *sh) {
    int most = 0, max_win = 0;   // (window's pairs and autocorrelations)
    for (int w = 0; w < sel->n_windows; ++w) {
        most = std::max(most, sel->wp_off[w + 1] - sel->wp_off[w]);
        max_win = std::max(max_win, sel->wp_t1[w] - sel->wp_t0[w]);
    }
    pairs_blocks(most, 1, sh);
    sh->smem = pairs_smem(vfmt, sel->L, sh->stage_stride);
    sh->ns = stage_samples(vfmt, (size_t)sel->L * sel->L * elem_size(vfmt));
    int occ = 0;
    auto resident = [&]() {
        sh->kern = vfmt == GC_C64 ? pick_pairs<GC_C64>(sh->kp)
                                  : (vfmt == GC_C32H ? pick_pairs<GC_C32H>(sh->kp) : pick_pairs<GC_I4C>(sh->kp));
        cudaError_t e = cudaFuncSetAttribute(sh->kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return gc_cuda_fail(ctx, e, "cudaFuncSetAttribute(xeng_pairs)");
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, sh->kern, sh->nthr, sh->smem);
        if (e != cudaSuccess || occ < 1) return gc_cuda_fail(ctx, e, "occupancy(xeng_pairs)");
        return GC_OK;
    };
    gc_status st = resident();
    if (st != GC_OK) return st;
    // split long windows in time so that the items fill whole waves of the
    // resident CTAs (slices of at least 64 samples)
    const int slots = occ * ctx->sm_count;
    const long base = (long)C * sel->n_windows;
    sh->n_tsplit = 1;
    double top = -1.0;
    for (int ts = 1; ts <= 16 && (ts == 1 || max_win / ts >= 64); ++ts) {
        const long items = base * sh->n_blk * ts, waves = (items + slots - 1) / slots;
        const double eff = (double)items / ((double)waves * slots) - 0.01 * ts;   // prefer fewer slices
        if (eff > top) {
            top = eff;
            sh->n_tsplit = ts;
        }
    }
    // Where that leaves SMs idle (few channels: there the 0.01 outweighs the fill):
    // slices down to 16 samples, and blocks of a window on several SMs, each of
    // which stages the window's samples again, by the cycles they are reckoned to
    // take and if these are fewer by a quarter.  One channel, without / so / in the
    // antenna form: 8x8 antennas, 8192 complex64 samples 133 / 29 / 33 us; 6x6, 8192
    // samples of 4+4 bits 289 / 25 / 25; 32x32, 4096 complex64 samples 93 / 64 / 85.
    if (base * sh->n_blk * sh->n_tsplit < ctx->sm_count) {
        gc_xeng_pairs_shape best = *sh;
        double least = 0.75 * pairs_cycles(sel, vfmt, C, ctx->sm_count, max_win, bulk, *sh, sh->n_tsplit);
        for (int nb = sh->n_blk; nb <= 16; nb *= 2) {
            gc_xeng_pairs_shape more = *sh;
            if (nb > sh->n_blk) pairs_blocks(most, nb, &more);
            if (nb > sh->n_blk && more.nthr < 128) break;
            const long fit = nb > sh->n_blk ? ctx->sm_count : slots;
            for (int ts = 1; ts <= 64 && (ts == 1 || max_win / ts >= 16) && base * more.n_blk * ts <= fit; ++ts) {
                const double t = pairs_cycles(sel, vfmt, C, ctx->sm_count, max_win, bulk, more, ts);
                if (t < least) {
                    least = t;
                    best = more;
                    best.n_tsplit = ts;
                }
            }
        }
        *sh = best;
        st = resident();
        if (st != GC_OK) return st;
    }
    // without autocorrelations the same slices (the same sums, bit for bit) in smaller blocks
    if (!autos) {
        pairs_blocks(most - sel->L * sel->L, sh->n_blk, sh);
        st = resident();
        if (st != GC_OK) return st;
    }
    if (ctx->tune[GC_TUNE_XENG_TSPLIT] > 0) sh->n_tsplit = std::min(ctx->tune[GC_TUNE_XENG_TSPLIT], 64);
    sh->n_items = (long)C * sel->n_windows * sh->n_blk * sh->n_tsplit;
    sh->grid = (int)std::min<long>(sh->n_items, (long)occ * ctx->sm_count);
    return GC_OK;
}

gc_status gc_xeng_pairs_launch(gc_ctx *ctx, const void *volt, int vfmt, int C, int T, const gc_sel *sel,
                               const gc_xeng_pairs_shape &sh, void *out, void *apart, cudaStream_t s) {
    PParams p;
    p.volt = static_cast<const unsigned char *>(volt);
    p.L = sel->L;
    p.N = sel->L * sel->L;
    p.C = C;
    p.T = T;
    p.P = sel->P;
    p.n_windows = sel->n_windows;
    p.n_blk = sh.n_blk;
    p.per_blk = sh.per_blk;
    p.n_tsplit = sh.n_tsplit;
    p.n_items = (int)sh.n_items;
    p.ns = sh.ns;
    p.autos = apart ? 1 : 0;
    p.wp_entry = sel->d_wp_entry;
    p.wp_off = sel->d_wp_off;
    p.win_t0 = sel->d_wp_t0;
    p.win_t1 = sel->d_wp_t1;
    p.pair_i = sel->d_pair_i;
    p.pair_j = sel->d_pair_j;
    p.out = out;
    p.apart = apart;
    p.status = ctx->status_dev;
    p.stage_stride = sh.stage_stride;
    p.use_tma = gc_xeng_pairs_bulk(sel, vfmt, volt) ? 1 : 0;
    p.pitch = pairs_pitch(vfmt, p.L);
    CUtensorMap tmap;
    memset(&tmap, 0, sizeof tmap);
    if (vfmt == GC_C64 && p.pitch != p.L) {
        if (p.use_tma) {
            const uint64_t dims[4] = {(uint64_t)p.L, (uint64_t)p.L, (uint64_t)T, (uint64_t)C};
            const uint64_t strides[3] = {(uint64_t)p.L * 8, (uint64_t)p.N * 8, (uint64_t)T * p.N * 8};
            const uint32_t box[4] = {(uint32_t)p.pitch, (uint32_t)p.L, (uint32_t)p.ns, 1u};
            const gc_status st = gc_encode_tiled(ctx, &tmap, CU_TENSOR_MAP_DATA_TYPE_UINT64, 4,
                                                 const_cast<void *>(volt), dims, strides, box);
            if (st != GC_OK) return st;
            p.use_tma = 2;
        } else {
            p.pitch = p.L;   // plain loads keep the rows as they are
        }
    }
    void *args[] = {&tmap, &p};
    const int rec = gc_prof_begin(ctx, s, "xeng_pairs");
    const cudaError_t e = cudaLaunchKernel(sh.kern, dim3(sh.grid), dim3(sh.nthr), args, sh.smem, s);
    gc_prof_end(ctx, s, rec);
    if (e != cudaSuccess) return gc_cuda_fail(ctx, e, "launch xeng_pairs");
    return GC_OK;
}
