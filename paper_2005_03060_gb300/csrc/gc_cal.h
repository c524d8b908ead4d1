// Device code shared by the calibration solvers (gc_calib.cu, gc_lincal.cu):
// parameters, observations, block reductions, the start point, the
// degeneracy convention and the end of a channel.
#pragma once

#include "gc_sel.h"

struct CalParams {
    const void *vred;            // c64 [C][P] float2 | i4c [C][P] int2
    int vfmt;
    const void *autos;           // c64 float | i4c int [C][N], or null
    int C, L, N, P, n_ubl;
    const int32_t *types, *type_ptr, *pair_i, *pair_j, *pair_type, *win_t0, *win_t1;
    const int32_t *nbr;          // [2][n_ubl][N] neighbour table or null
    int ax, ay;                  // indices of types (1,0) and (0,1)
    int stencil;                 // matrix-free operator by per-antenna gather (<= kStencilTypes types)
    int st_halo;                 // largest |dx| or |dy| of a type (stencil operator)
    int dense;                   // matrix-free operator as lag-plane correlations (selections of many types)
    // partly occupied lattice (null / L*L otherwise): occupancy [N], the
    // breadth-first start-point tree over the axis types, antennas
    const int32_t *mask, *tree_ant, *tree_pair, *tree_sign;
    int n_occ;
    int t_autos;                 // samples summed in autos
    float2 *gains;               // [C][N] (in: warm start when warm != 0)
    float2 *vmodel;              // [C][n_ubl]
    gc_calstats *stats;          // [C]
    int solver, max_iter, warm;
    double tol, damping, mu_rel;
    int band;                    // largest distance of a pair's antennas in row order (GC_LINCAL)
    char *work;
    size_t work_per_cta;
    unsigned int *counter;   // next channel to take (matrix-free kernels; zeroed before the launch)
    unsigned int *status;
    unsigned long long deadline_ns;   // per-channel time budget
    int red32;                   // matrix-free solver: every reduction in FP32 (the plain-FP32 form)
};

gc_status gc_lincal_run(gc_ctx *ctx, CalParams &p, bool fp64, cudaStream_t s);   // GC_LINCAL (gc_lincal.cu)

namespace {

__device__ __forceinline__ float2 vobs(const CalParams &p, int c, int pidx) {
    const int k = p.pair_type[pidx];
    const float inv = 1.0f / (float)(p.win_t1[k] - p.win_t0[k]);
    if (p.vfmt == GC_C64) {
        const float2 v = reinterpret_cast<const float2 *>(p.vred)[(size_t)c * p.P + pidx];
        return make_float2(v.x * inv, v.y * inv);
    }
    const int2 v = reinterpret_cast<const int2 *>(p.vred)[(size_t)c * p.P + pidx];
    return make_float2((float)v.x * inv, (float)v.y * inv);
}

__device__ __forceinline__ float auto_of(const CalParams &p, int c, int i) {
    if (!p.autos) return 1.0f;
    if (p.vfmt == GC_C64) return reinterpret_cast<const float *>(p.autos)[(size_t)c * p.N + i];
    return (float)reinterpret_cast<const int *>(p.autos)[(size_t)c * p.N + i];
}

// index of the pair (r_j + d_k, r_j) in the selection, or -1
__device__ __forceinline__ int pair_index(const CalParams &p, int k, int xj, int yj) {
    const int dx = p.types[2 * k], dy = p.types[2 * k + 1];
    const int L = p.L;
    const int xi = xj + dx, yi = yj + dy;
    if (xj < 0 || xj >= L || yj < 0 || yj >= L || xi < 0 || xi >= L || yi < 0 || yi >= L) return -1;
    const int xlo = max(0, -dx), ylo = max(0, -dy);
    return p.type_ptr[k] + (yj - ylo) * (L - abs(dx)) + (xj - xlo);
}

template <class R>
struct C2 {
    R x, y;
};
template <class R>
__device__ __forceinline__ C2<R> cm(C2<R> a, C2<R> b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <class R>
__device__ __forceinline__ C2<R> cj(C2<R> a) {
    return {a.x, -a.y};
}

// ----------------------------------------------------------------- block reductions
template <class R, int NV>
__device__ void block_sum(R (&v)[NV], R *red /* smem [32][NV] */) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    __syncthreads();
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) red[w * NV + q] = v[q];
    __syncthreads();
    const int nw = blockDim.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        R s = 0;
        for (int u = 0; u < nw; ++u) s += red[u * NV + q];
        v[q] = s;
    }
    __syncthreads();
}

// Has the channel used up its time?  One thread asks, ahead of a barrier that the
// iteration has anyway, and all threads read its answer after it: threads that
// read the timer for themselves could part in the limit's last instant, some
// leaving the iteration and some waiting at its barriers.
__device__ __forceinline__ bool out_of_time(const CalParams &p, uint64_t t_start) {
    return gc_globaltimer() - t_start > p.deadline_ns;
}

// ----------------------------------------------------------------- start point
// Spanning-tree phases over the (1,0) and (0,1) types (arg V_(1,0) = arg V_(0,1)
// = 0 fixes the slopes), unit amplitudes, V_alpha = group mean of V_p / (g_i g_j^*).
template <class R>
__device__ void start_point(const CalParams &p, int c, R *xg, R *xv, R *red, R *phi /* N reals of scratch */) {
    const int L = p.L, N = p.N;
    // the phase steps are taken by all threads (their loads are independent),
    // then summed along the tree in a fixed order
    if (p.tree_ant) {
        // partly occupied lattice: walk the breadth-first tree, phi_i - phi_j
        // = arg V_p along each linking pair p = (i, j); empty points get 0
        for (int i = threadIdx.x; i < N; i += blockDim.x) phi[i] = 0;
        __syncthreads();
        for (int h = 1 + threadIdx.x; h < p.n_occ; h += blockDim.x) {
            const float2 v = vobs(p, c, p.tree_pair[h]);
            phi[p.tree_ant[h]] = (R)atan2f(v.y, v.x);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int h = 1; h < p.n_occ; ++h) {
                const int a = p.tree_ant[h], q = p.tree_pair[h];
                const R arg = phi[a];
                phi[a] = p.tree_sign[h] > 0 ? phi[p.pair_j[q]] + arg : phi[p.pair_i[q]] - arg;
            }
        }
    } else {
        for (int i = threadIdx.x; i < N; i += blockDim.x) {
            const int x = i % L, y = i / L;
            R arg = 0;
            if (i > 0) {
                const float2 v = vobs(p, c, y == 0 ? pair_index(p, p.ax, x - 1, 0) : pair_index(p, p.ay, x, y - 1));
                arg = (R)atan2f(v.y, v.x);
            }
            phi[i] = arg;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int x = 1; x < L; ++x) phi[x] += phi[x - 1];
        __syncthreads();
        for (int x = threadIdx.x; x < L; x += blockDim.x) {
            R acc = phi[x];
            for (int y = 1; y < L; ++y) {
                acc += phi[y * L + x];
                phi[y * L + x] = acc;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        R s, co;
        if (sizeof(R) == 8) {
            double sd, cd;
            sincos((double)phi[i], &sd, &cd);
            s = (R)sd;
            co = (R)cd;
        } else {
            float sf, cf;
            sincosf((float)phi[i], &sf, &cf);
            s = (R)sf;
            co = (R)cf;
        }
        const bool occ = !p.mask || p.mask[i];   // empty points hold g = 0
        xg[2 * i] = occ ? co : (R)0;
        xg[2 * i + 1] = occ ? s : (R)0;
    }
    __syncthreads();
    // V_alpha: one warp per type
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int k = w; k < p.n_ubl; k += nw) {
        R sx = 0, sy = 0;
        for (int q = p.type_ptr[k] + lane; q < p.type_ptr[k + 1]; q += 32) {
            const int i = p.pair_i[q], j = p.pair_j[q];
            const float2 v = vobs(p, c, q);
            C2<R> gi{xg[2 * i], xg[2 * i + 1]}, gj{xg[2 * j], xg[2 * j + 1]};
            C2<R> e = cm(cj(gi), gj);   // 1 / (g_i g_j^*) for unit gains
            C2<R> t = cm(C2<R>{(R)v.x, (R)v.y}, e);
            sx += t.x;
            sy += t.y;
        }
        for (int o = 16; o > 0; o >>= 1) {
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
        }
        if (lane == 0) {
            const R n = (R)(p.type_ptr[k + 1] - p.type_ptr[k]);
            xv[2 * k] = sx / n;
            xv[2 * k + 1] = sy / n;
        }
    }
    __syncthreads();
}

// chi^2 = sum_p |so V_p - g_i g_j^* V_alpha|^2 over all pairs (one visit each)
template <class R>
__device__ R chi2_of(const CalParams &p, int c, const R *xg, const R *xv, R *red, R so = 1) {
    R s[1] = {0};
    for (int q = threadIdx.x; q < p.P; q += blockDim.x) {
        const int i = p.pair_i[q], j = p.pair_j[q], k = p.pair_type[q];
        const float2 v = vobs(p, c, q);
        C2<R> m = cm(cm(C2<R>{xg[2 * i], xg[2 * i + 1]}, cj(C2<R>{xg[2 * j], xg[2 * j + 1]})),
                     C2<R>{xv[2 * k], xv[2 * k + 1]});
        const R rx = (R)v.x * so - m.x, ry = (R)v.y * so - m.y;
        s[0] += rx * rx + ry * ry;
    }
    block_sum<R, 1>(s, red);
    return s[0];
}

// Solve G c = r for the 4 degeneracy coefficients from the packed lower
// triangle of the Gram matrix (acc[0..9]) and the right-hand side acc[10..13]
// (Cholesky; c = 0 when a direction vanishes).
template <class R>
__device__ void solve_gram4(const R (&acc)[14], R (&cvec)[4]) {
    R G[4][4], r[4];
    {
        int q = 0;
        for (int a = 0; a < 4; ++a)
            for (int b = 0; b <= a; ++b) {
                G[a][b] = acc[q];
                G[b][a] = acc[q];
                ++q;
            }
        for (int a = 0; a < 4; ++a) r[a] = acc[10 + a];
        // Cholesky with a guard
        R Lm[4][4] = {};
        bool ok = true;
        for (int a = 0; a < 4 && ok; ++a) {
            R s = G[a][a];
            for (int b = 0; b < a; ++b) s -= Lm[a][b] * Lm[a][b];
            if (!(s > (R)1e-30)) {
                ok = false;
                break;
            }
            Lm[a][a] = sqrt(s);
            for (int i = a + 1; i < 4; ++i) {
                R t = G[i][a];
                for (int b = 0; b < a; ++b) t -= Lm[i][b] * Lm[a][b];
                Lm[i][a] = t / Lm[a][a];
            }
        }
        if (ok) {
            R y[4];
            for (int a = 0; a < 4; ++a) {
                R s = r[a];
                for (int b = 0; b < a; ++b) s -= Lm[a][b] * y[b];
                y[a] = s / Lm[a][a];
            }
            for (int a = 3; a >= 0; --a) {
                R s = y[a];
                for (int b = a + 1; b < 4; ++b) s -= Lm[b][a] * cvec[b];
                cvec[a] = s / Lm[a][a];
            }
        } else {
            for (int a = 0; a < 4; ++a) cvec[a] = 0;
        }
    }
}

// Degeneracy convention of the output: mean ln|g| = 0, arg V_(1,0) =
// arg V_(0,1) = 0, arg g_0 = 0.  Works on float2 gains in place.
__device__ void output_convention(const CalParams &p, float2 *g, float2 *V, double *red) {
    // per antenna in FP32 (the gains are FP32 values), summed in FP64
    double s[1] = {0.0};
    for (int i = threadIdx.x; i < p.N; i += blockDim.x)
        if (!p.mask || p.mask[i]) s[0] += (double)logf(hypotf(g[i].x, g[i].y));
    block_sum<double, 1>(s, red);
    const double sc = exp(s[0] / p.n_occ);
    const double kx = atan2((double)V[p.ax].y, (double)V[p.ax].x);
    const double ky = atan2((double)V[p.ay].y, (double)V[p.ay].x);
    __syncthreads();
    for (int k = threadIdx.x; k < p.n_ubl; k += blockDim.x) {
        const double ph = -(kx * p.types[2 * k] + ky * p.types[2 * k + 1]);
        double sn, cs;
        sincos(ph, &sn, &cs);
        const double vx = V[k].x * sc * sc, vy = V[k].y * sc * sc;
        V[k] = make_float2((float)(vx * cs - vy * sn), (float)(vx * sn + vy * cs));
    }
    // phase of the first antenna after the slope change (antenna 0 of a full
    // grid, at x = y = 0; the first occupied point of a partly occupied one)
    const int r0 = p.tree_ant ? p.tree_ant[0] : 0;
    const double psi = atan2((double)g[r0].y, (double)g[r0].x) + kx * (r0 % p.L) + ky * (r0 / p.L);
    __syncthreads();
    // the ramp phase in FP64, reduced to [-pi, pi] there, then rotated in FP32
    constexpr double kTwoPi = 6.283185307179586, kInvTwoPi = 0.15915494309189535;
    const float isc = (float)(1.0 / sc);
    for (int i = threadIdx.x; i < p.N; i += blockDim.x) {
        const double ph = kx * (i % p.L) + ky * (i / p.L) - psi;
        float sn, cs;
        sincosf((float)(ph - kTwoPi * rint(ph * kInvTwoPi)), &sn, &cs);
        const float gx = g[i].x * isc, gy = g[i].y * isc;
        g[i] = make_float2(gx * cs - gy * sn, gx * sn + gy * cs);
    }
    __syncthreads();
}

template <class R>
__device__ void finish_channel(const CalParams &p, int c, const R *xg, const R *xv, int iters, int st,
                               double *red, int inner = 0) {
    float2 *g = p.gains + (size_t)c * p.N;
    float2 *V = p.vmodel + (size_t)c * p.n_ubl;
    for (int i = threadIdx.x; i < p.N; i += blockDim.x) g[i] = make_float2((float)xg[2 * i], (float)xg[2 * i + 1]);
    for (int k = threadIdx.x; k < p.n_ubl; k += blockDim.x) V[k] = make_float2((float)xv[2 * k], (float)xv[2 * k + 1]);
    __syncthreads();
    output_convention(p, g, V, red);
    // chi^2 and chi^2_r (Eq. redchi, Eq. dof) at the output point: the
    // model products in the solver's precision (FP32 for the FP32 solvers,
    // FP64 for the FP64 one), the sums in FP64; the noise weight
    // 1 / sigma_p^2 = t_p (t_a / a_i) (t_a / a_j) in FP32 (no FP64 division)
    double acc[2] = {0.0, 0.0};
    const float ta = (float)p.t_autos;
    for (int q = threadIdx.x; q < p.P; q += blockDim.x) {
        const int i = p.pair_i[q], j = p.pair_j[q], k = p.pair_type[q];
        const float2 v = vobs(p, c, q);
        double r2;
        if constexpr (sizeof(R) == sizeof(float)) {
            const float2 gi = g[i], gj = g[j], Vk = V[k];
            const float ex = gi.x * gj.x + gi.y * gj.y, ey = gi.y * gj.x - gi.x * gj.y;   // g_i conj(g_j)
            const float mx = ex * Vk.x - ey * Vk.y, my = ex * Vk.y + ey * Vk.x;
            const float rx = v.x - mx, ry = v.y - my;
            r2 = (double)rx * rx + (double)ry * ry;
        } else {
            const double gx = g[i].x, gy = g[i].y, hx = g[j].x, hy = -g[j].y;
            const double ex = gx * hx - gy * hy, ey = gx * hy + gy * hx;
            const double mx = ex * V[k].x - ey * V[k].y, my = ex * V[k].y + ey * V[k].x;
            const double rx = v.x - mx, ry = v.y - my;
            r2 = rx * rx + ry * ry;
        }
        acc[0] += r2;
        const float wp = (float)(p.win_t1[k] - p.win_t0[k]) * (ta / auto_of(p, c, i)) * (ta / auto_of(p, c, j));
        acc[1] += r2 * (double)wp;
    }
    block_sum<double, 2>(acc, red);
    if (threadIdx.x == 0) {
        gc_calstats s;
        s.chi2 = acc[0];
        s.dof = p.P - p.n_occ - p.n_ubl + 2;
        s.chi2r = p.autos && s.dof > 0 ? acc[1] / s.dof : -1.0;
        s.iters = iters;
        // observations or solution not finite: the channel has no result
        s.status = isfinite(acc[0]) ? st : GC_EINVAL;
        s.inner = inner;
        p.stats[c] = s;
    }
    __syncthreads();
}

}  // namespace
