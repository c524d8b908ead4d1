// lincal (paper Sec. 2: Gauss-Newton on the redundant model), the direct
// solver of GC_LINCAL.
//
// One CTA calibrates one channel at a time.  A step solves the normal
// equations of the linearised model; what decides the result is the gradient
// J^T r, evaluated in the caller's precision (FP64 by default), and the
// convergence test on the step.  The matrix only turns the gradient into a
// step, so it is formed and factorised in FP32 and kept while the iteration
// contracts; the fixed point, J^T r = 0, does not depend on it.
//
// Step coordinates.  With dg_i = u_i q_i, dV_k = v_k w_k (u, v the unit phases of
// g_i and V_k) the linearised model of pair (i, j) of type k is
//   dM = m/|m| (|g_j||V_k| q_i + |g_i||V_k| conj(q_j) + |g_i||g_j| w_k),
// with real factors, so the 2N + 2K real unknowns fall apart into an
// "amplitude" system (real parts, q_i + q_j + w_k) and a "phase" system
// (imaginary parts, q_i - q_j + w_k) of N + K unknowns each.  Antennas in row
// order give each a band of half-width D = max(dy L + dx) with the K model
// visibilities as a border: a fourth of the arithmetic of one real band of
// 2N rows and half-width 2D + 1, and two independent factorisations, one per
// half of the CTA.
//
// What bounds it: the serial chains of the factorisation (0.35 ms, three to
// four a solve) and of the block solves (0.07 ms), then the FP64 pipe (1.8
// FMA/clk/SM) in the gradient (24 operations a pair, 0.08 ms an iteration).
// Measured, 128 channels of 32x32 antennas (10 446 pairs, D = 66, 8 iterations):
// 4.2 ms, against 285 ms for an FP64 band factorisation with a barrier per
// column in every iteration; 8 channels of 48x48: 15.7 against 922 ms; 32 of
// 8x8: 0.40 against 9.9 ms.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "gc_cal.h"

namespace {

constexpr int kLThreads = 512;
constexpr int kNB = 16;         // block side of the band
constexpr int kPS = 20;         // row stride of a block in shared memory (floats): 16-byte pieces of
                                // eight consecutive rows on distinct banks
constexpr int kBS = kNB * kPS;  // floats of a block in shared memory
constexpr size_t kLSmem = 221 * 1024;   // dynamic shared memory of a CTA at most

template <class R>
struct alignas(2 * sizeof(R)) V2 {
    R x, y;
};

// Where a solve keeps what it reads over and over.  `fast`: vectors, panels and
// a ring of the last kRing block columns in shared memory (up to D = 96 antennas
// of band, i.e. 40 x 40 grids with the default selections; its own
// instantiation, so that they are read as shared memory).  Otherwise all of it
// is in the CTA's global (L2) workspace.
constexpr int kRing = 8;
struct LinShape {
    int npad, nblk, q;          // padded antennas, block columns, sub-diagonal blocks per column
    int fast;
};

__host__ __device__ inline LinShape lin_shape(int N, int D, int K) {
    LinShape s;
    s.npad = (N + kNB - 1) / kNB * kNB;
    s.nblk = s.npad / kNB;
    s.q = (D + kNB - 1) / kNB;
    const size_t types = (size_t)2 * (K * (K + 1) + K + kNB * K + kBS + 2 * 16 * kNB) * 4 + 4096;
    const size_t vec = (size_t)3 * s.npad * 4, panel = (size_t)2 * 2 * (s.q + 1) * kBS * 4;
    const size_t ring = (size_t)2 * kRing * ((s.q + 1) * kBS + kNB * K) * 4;
    s.fast = s.q <= kRing - 2 && types + vec + panel + ring <= kLSmem ? 1 : 0;
    return s;
}

// Bump allocator used on both sides: bytes on the host, pointers on the device.
struct Bump {
    char *base;
    size_t at = 0;
    __host__ __device__ explicit Bump(char *b) : base(b) {}
    template <class T>
    __host__ __device__ T *take(size_t n) {
        T *r = reinterpret_cast<T *>(base + at);
        at = (at + n * sizeof(T) + 127) / 128 * 128;
        return r;
    }
};

template <class R>
struct LinWork {
    V2<R> *x, *tr, *hs;        // point, trial point, gradient sums: antennas then types
    V2<R> *dl;                 // step (or, as float2, the step scaled by sc); scratch of the start point
    V2<R> *qt, *rs;            // refined relative step, residual of its equations
    R *G;                      // |g|^2, |V|^2
    V2<R> *h;                  // [K][N] conj(m) r of the pair whose first member is the antenna
    float *D, *vv;             // diagonals of the matrix: antennas, types
    float *fa, *fv;            // normalised |g|, |V|
    // both systems, amplitude then phase:
    float *Lb;                 // [nblk][q + 1][16][16]: inverted diagonal block, then the blocks below it
    float *Z;                  // eliminated border [K][npad]
    float *y, *rk;             // right-hand side, then solution: antennas, types
    float *P, *Ls, *T;         // panel, inverted diagonal block, border rows of the current column
    float *S, *part;           // Schur complement of the types, partial sums of the solves
    float *ring, *zring;       // block columns and border rows at hand
};

// One system's part of the work.
template <bool kFast>
struct LinSys {
    float *Lb, *Z, *y, *rk, *P, *Ls, *T, *S, *part, *ring, *zring;
    int npad, nblk, q, q1, K;
    // row stride and size of a block where column() points
    static constexpr int st = kFast ? kPS : kNB, bs = kNB * st;
    template <class R>
    __device__ LinSys(const LinWork<R> &w, const LinShape &s, int k, int sys)
        : npad(s.npad), nblk(s.nblk), q(s.q), q1(s.q + 1), K(k) {
        Lb = w.Lb + (size_t)sys * nblk * q1 * kNB * kNB;
        Z = w.Z + (size_t)sys * K * npad;
        y = w.y + sys * npad;
        rk = w.rk + sys * K;
        P = w.P + sys * 2 * q1 * kBS;
        Ls = w.Ls + sys * kBS;
        T = w.T + sys * kNB * K;
        S = w.S + sys * K * (K + 1);
        part = w.part + sys * 2 * 16 * kNB;
        if (kFast) {
            ring = w.ring + sys * kRing * q1 * kBS;
            zring = w.zring + sys * kRing * kNB * K;
        }
    }
    // block column b where the factorisation and the solves read it
    __device__ __forceinline__ float *column(int b) const {
        if constexpr (kFast) return ring + (b & (kRing - 1)) * q1 * kBS;
        else return Lb + (size_t)b * q1 * kNB * kNB;
    }
    // border rows of block b for type k
    __device__ __forceinline__ float *border(int b, int k) const {
        if constexpr (kFast) return zring + ((b & (kRing - 1)) * K + k) * kNB;
        else return Z + (size_t)k * npad + kNB * b;
    }
};

template <class R>
__host__ __device__ size_t lin_global(LinWork<R> &w, char *base, int N, int K, const LinShape &s) {
    Bump b(base);
    w.x = b.take<V2<R>>(N + K);
    w.tr = b.take<V2<R>>(N + K);
    w.dl = b.take<V2<R>>(N + K);
    w.qt = b.take<V2<R>>(sizeof(R) == 8 ? N + K : 0);
    w.rs = b.take<V2<R>>(sizeof(R) == 8 ? N + K : 0);
    w.G = b.take<R>(sizeof(R) == 8 ? N + K : 0);
    w.hs = b.take<V2<R>>(N + K);
    w.h = b.take<V2<R>>((size_t)K * N);
    w.D = b.take<float>(s.npad);
    w.vv = b.take<float>(K);
    w.Lb = b.take<float>((size_t)2 * s.nblk * (s.q + 1) * kNB * kNB);
    w.Z = b.take<float>((size_t)2 * K * s.npad);
    if (!s.fast) {
        w.fa = b.take<float>(s.npad);
        w.y = b.take<float>((size_t)2 * s.npad);
        w.P = b.take<float>((size_t)2 * 2 * (s.q + 1) * kBS);
    }
    return b.at;
}

template <class R, bool kFast>
__host__ __device__ size_t lin_shared(LinWork<R> &w, char *base, int K, const LinShape &s) {
    Bump b(base);
    if (kFast) {
        w.fa = b.take<float>(s.npad);
        w.y = b.take<float>((size_t)2 * s.npad);
        w.P = b.take<float>((size_t)2 * 2 * (s.q + 1) * kBS);
        w.ring = b.take<float>((size_t)2 * kRing * (s.q + 1) * kBS);
        w.zring = b.take<float>((size_t)2 * kRing * kNB * K);
    }
    w.fv = b.take<float>(K);
    w.S = b.take<float>((size_t)2 * K * (K + 1));
    w.rk = b.take<float>((size_t)2 * K);
    w.T = b.take<float>((size_t)2 * K * kNB);
    w.Ls = b.take<float>((size_t)2 * kBS);
    w.part = b.take<float>((size_t)2 * 2 * 16 * kNB);
    return b.at;
}

// Barrier of one half of the CTA (id 1 or 2).
__device__ __forceinline__ void half_sync(int sys, int n) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + sys), "r"(n) : "memory");
}

struct LinTypes {   // per type: dx, dy, antenna offset; pair base and row width; 1 / window
    int4 a[64];
    int2 b[64];
    float inv[64];
};

__device__ __forceinline__ float2 lin_obs(const CalParams &p, size_t row, int q, float inv) {
    if (p.vfmt == GC_C64) {
        const float2 v = reinterpret_cast<const float2 *>(p.vred)[row + q];
        return make_float2(v.x * inv, v.y * inv);
    }
    const int2 v = reinterpret_cast<const int2 *>(p.vred)[row + q];
    return make_float2((float)v.x * inv, (float)v.y * inv);
}

// Gradient and chi^2 at the point x.  Each pair is evaluated once, by the
// thread of its first member, h = conj(m) r; the second member's term is
// m conj(r) = conj(h), gathered after a barrier, and a type's term is h.  Sums
// hs_i = g_i^* dchi-gradient_i and hs_k = V_k^* gradient_k (a zero gain or
// visibility, whose h vanishes, gets its gradient itself).
template <class R>
__device__ R lin_resid(const CalParams &p, int c, const V2<R> *x, const LinWork<R> &w, const LinTypes &ty, R *red) {
    const int L = p.L, N = p.N, K = p.n_ubl, nt = blockDim.x;
    const size_t row = (size_t)c * p.P;
    R chi[1] = {0};
    for (int m = threadIdx.x; m < N; m += nt) {
        const int mx = m % L, my = m / L;
        const V2<R> gm = x[m];
        V2<R> s{0, 0};
        for (int k = 0; k < K; ++k) {
            const int4 a = ty.a[k];
            const int xj = mx - a.x, yj = my - a.y;
            V2<R> h{0, 0};
            if ((unsigned)xj < (unsigned)L && (unsigned)yj < (unsigned)L) {
                const int2 b = ty.b[k];
                const float2 o = lin_obs(p, row, b.x + yj * b.y + xj, ty.inv[k]);
                const V2<R> gj = x[m - a.z], V = x[N + k];
                const R ex = gj.x * V.x + gj.y * V.y, ey = gj.x * V.y - gj.y * V.x;   // conj(g_j) V
                const R px = gm.x * ex - gm.y * ey, py = gm.x * ey + gm.y * ex;       // model
                const R rx = (R)o.x - px, ry = (R)o.y - py;
                chi[0] += rx * rx + ry * ry;
                h.x = px * rx + py * ry;
                h.y = px * ry - py * rx;
                s.x += h.x;
                s.y += h.y;
            }
            w.h[(size_t)k * N + m] = h;
        }
        w.hs[m] = s;
    }
    __syncthreads();
    for (int m = threadIdx.x; m < N; m += nt) {
        const int mx = m % L, my = m / L;
        const V2<R> gm = x[m];
        const bool zero = gm.x == 0 && gm.y == 0;
        V2<R> s = w.hs[m];
        if (zero) s = V2<R>{0, 0};
        for (int k = 0; k < K; ++k) {
            const int4 a = ty.a[k];
            const bool v2 = (unsigned)(mx + a.x) < (unsigned)L && (unsigned)(my + a.y) < (unsigned)L;
            if (!zero) {
                if (v2) {
                    const V2<R> h = w.h[(size_t)k * N + m + a.z];
                    s.x += h.x;
                    s.y -= h.y;
                }
                continue;
            }
            const int2 b = ty.b[k];   // g_m = 0: sum conj(J) r with r = V_p
            const V2<R> V = x[N + k];
            if (v2) {
                const V2<R> gi = x[m + a.z];
                const float2 o = lin_obs(p, row, b.x + my * b.y + mx, ty.inv[k]);
                const R bx = gi.x * V.x - gi.y * V.y, by = gi.x * V.y + gi.y * V.x;   // g_i V
                s.x += bx * o.x + by * o.y;   // g_i V conj(r)
                s.y += by * o.x - bx * o.y;
            }
            const int xj = mx - a.x, yj = my - a.y;
            if ((unsigned)xj < (unsigned)L && (unsigned)yj < (unsigned)L) {
                const V2<R> gj = x[m - a.z];
                const float2 o = lin_obs(p, row, b.x + yj * b.y + xj, ty.inv[k]);
                const R ex = gj.x * V.x + gj.y * V.y, ey = gj.x * V.y - gj.y * V.x;
                s.x += ex * o.x + ey * o.y;   // conj(conj(g_j) V) r
                s.y += ex * o.y - ey * o.x;
            }
        }
        w.hs[m] = s;
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = nt >> 5;
    for (int k = wp; k < K; k += nw) {
        V2<R> s{0, 0};
        const V2<R> V = x[N + k];
        if (V.x == 0 && V.y == 0) {
            const int4 a = ty.a[k];
            const int2 b = ty.b[k];
            for (int m = lane; m < N; m += 32) {
                const int xj = m % L - a.x, yj = m / L - a.y;
                if ((unsigned)xj >= (unsigned)L || (unsigned)yj >= (unsigned)L) continue;
                const V2<R> gi = x[m], gj = x[m - a.z];
                const float2 o = lin_obs(p, row, b.x + yj * b.y + xj, ty.inv[k]);
                const R ex = gi.x * gj.x + gi.y * gj.y, ey = gi.y * gj.x - gi.x * gj.y;   // g_i conj(g_j)
                s.x += ex * o.x + ey * o.y;
                s.y += ex * o.y - ey * o.x;
            }
        } else {
            const V2<R> *h = w.h + (size_t)k * N;
#pragma unroll 4
            for (int m = lane; m < N; m += 32) {
                s.x += h[m].x;
                s.y += h[m].y;
            }
        }
        for (int o = 16; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (lane == 0) w.hs[N + k] = s;
    }
    block_sum<R, 1>(chi, red);
    return chi[0];
}

// |z| / unit (i2 = 1 / unit^2): 0 for z = 0 alone, else at least 1e-15, where
// its square is negligible beside the largest and still a normal number
template <class R>
__device__ __forceinline__ float lin_amp(V2<R> z, R i2) {
    if (z.x == 0 && z.y == 0) return 0.f;
    return fmaxf(sqrtf((float)((z.x * z.x + z.y * z.y) * i2)), 1e-15f);
}

// Normalised amplitudes, matrix diagonals and borders at the point x.
// Returns false when every gain or every visibility vanishes.
template <class R>
__device__ bool lin_prepare(const CalParams &p, const LinWork<R> &w, const LinShape &sh, const LinTypes &ty, R *red,
                            R &am, R &vm) {
    const int L = p.L, N = p.N, K = p.n_ubl, nt = blockDim.x;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = nt >> 5;
    R a2 = 0, v2 = 0;
    for (int m = threadIdx.x; m < N; m += nt) a2 = fmax(a2, w.x[m].x * w.x[m].x + w.x[m].y * w.x[m].y);
    for (int k = threadIdx.x; k < K; k += nt) v2 = fmax(v2, w.x[N + k].x * w.x[N + k].x + w.x[N + k].y * w.x[N + k].y);
    for (int o = 16; o > 0; o >>= 1) {
        a2 = fmax(a2, __shfl_xor_sync(0xffffffffu, a2, o));
        v2 = fmax(v2, __shfl_xor_sync(0xffffffffu, v2, o));
    }
    __syncthreads();
    if (lane == 0) {
        red[2 * wp] = a2;
        red[2 * wp + 1] = v2;
    }
    __syncthreads();
    a2 = v2 = 0;
    for (int u = 0; u < nw; ++u) {
        a2 = fmax(a2, red[2 * u]);
        v2 = fmax(v2, red[2 * u + 1]);
    }
    __syncthreads();
    if (!(a2 > 0) || !(v2 > 0) || !isfinite(a2) || !isfinite(v2)) return false;
    am = sqrt(a2);
    vm = sqrt(v2);
    const R ia2 = 1 / a2, iv2 = 1 / v2;
    for (int m = threadIdx.x; m < sh.npad; m += nt)
        w.fa[m] = m < N ? lin_amp<R>(w.x[m], ia2) : 0.f;
    for (int k = threadIdx.x; k < K; k += nt)
        w.fv[k] = lin_amp<R>(w.x[N + k], iv2);
    __syncthreads();
    for (int m = threadIdx.x; m < sh.npad; m += nt) {
        const int mx = m % L, my = m / L;
        const float fm = w.fa[m];
        float D = 0.f;
        for (int k = 0; k < K; ++k) {
            const int4 a = ty.a[k];
            const float fk = w.fv[k];
            float b1 = 0.f, b2 = 0.f;
            if (m < N && (unsigned)(mx - a.x) < (unsigned)L && (unsigned)(my - a.y) < (unsigned)L)
                b1 = w.fa[m - a.z] * w.fa[m - a.z];
            if (m < N && (unsigned)(mx + a.x) < (unsigned)L && (unsigned)(my + a.y) < (unsigned)L)
                b2 = w.fa[m + a.z] * w.fa[m + a.z];
            D = fmaf(fk * fk, b1 + b2, D);
            w.Z[(size_t)k * sh.npad + m] = fm * fk * (b1 + b2);
            w.Z[(size_t)(K + k) * sh.npad + m] = fm * fk * (b1 - b2);
        }
        w.D[m] = D;
    }
    for (int k = wp; k < K; k += nw) {
        const int4 a = ty.a[k];
        float s = 0.f;
        for (int m = lane; m < N; m += 32) {
            const int xj = m % L - a.x, yj = m / L - a.y;
            if ((unsigned)xj >= (unsigned)L || (unsigned)yj >= (unsigned)L) continue;
            const float t = w.fa[m] * w.fa[m - a.z];
            s = fmaf(t, t, s);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) w.vv[k] = s;
    }
    __syncthreads();
    return true;
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, s))));
}
__device__ __forceinline__ float4 ld4(const float *p) { return *reinterpret_cast<const float4 *>(p); }

// Block band Cholesky of one system by one half of the CTA (n threads, thread
// t), left-looking over block columns of 16; the border rides along
// (Z = L^-1 B), then the K x K Schur complement of the types is factorised.
// Diagonals carry a relative shift `reg`.  Every thread of the half returns
// the same value; false on a pivot that is not positive.
template <class R, bool kFast>
__device__ __forceinline__ bool lin_factor(const CalParams &p, const LinWork<R> &w, const LinSys<kFast> &y, const LinTypes &ty, int sys,
                           int t, int n, float reg, volatile int *fail) {
    const int L = p.L, N = p.N, K = y.K, q = y.q;
    const int lane = t & 31, wp = t >> 5, nw = n >> 5;
    float *Li = y.Ls, *T = y.T;
    const float sg = sys == 0 ? 1.f : -1.f;
    auto panel = [&](int b) { return y.P + (size_t)(b & 1) * y.q1 * kBS; };
    auto clear = [&](int b, int t0, int step) {   // block column b's panel
        float *P = panel(b);
        for (int i = t0; i < kNB * y.q1 * 4; i += step)
            *reinterpret_cast<float4 *>(P + (i >> 2) * kPS + 4 * (i & 3)) = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    auto entries = [&](int b, int t0, int step) {   // the matrix entries of block column b
        float *P = panel(b);
        for (int i = t0; i < kNB * (K + 1); i += step) {
            const int cl = i & 15, k = i >> 4, j = kNB * b + cl;
            if (k == K) {
                P[cl * kPS + cl] = j < N ? fmaf(w.D[j], 1.f + reg, 1e-12f) : 1.f;
            } else if (j < N) {
                const int4 a = ty.a[k];
                const int yj = j / L, xj = j - yj * L;
                if ((unsigned)(xj + a.x) < (unsigned)L && (unsigned)(yj + a.y) < (unsigned)L)
                    P[(cl + a.z) * kPS + cl] = sg * w.fa[j + a.z] * w.fa[j] * w.fv[k] * w.fv[k];
            }
        }
    };
    clear(0, t, n);
    half_sync(sys, n);
    entries(0, t, n);
    half_sync(sys, n);
    for (int b = 0; b < y.nblk; ++b) {
        const int smax = min(q, y.nblk - 1 - b);
        float *P = panel(b);
        // panel -= L[b+s][b-t] L[b][b-t]^T: a warp per block, a lane rows r and
        // r + 8 and columns c, c + 4, c + 8, c + 12 (32 products of 6 reads)
        {
            const int r = lane >> 2, c = lane & 3;
            for (int s = wp; s <= smax; s += nw) {
                float acc[2][4];
                float *pr = P + (kNB * s + r) * kPS + c;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[0][i] = pr[4 * i];
                    acc[1][i] = pr[8 * kPS + 4 * i];
                }
                const int tm = min(q - s, b);
                for (int tt = 1; tt <= tm; ++tt) {
                    const float *col = y.column(b - tt);
                    const float *ar = col + (s + tt) * y.bs + r * y.st, *cr = col + tt * y.bs + c * y.st;
#pragma unroll
                    for (int k = 0; k < kNB; k += 4) {
                        const float4 a0 = ld4(ar + k), a1 = ld4(ar + 8 * y.st + k);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float4 v = ld4(cr + 4 * i * y.st + k);
                            acc[0][i] -= dot4(a0, v, 0.f);
                            acc[1][i] -= dot4(a1, v, 0.f);
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    pr[4 * i] = acc[0][i];
                    pr[8 * kPS + 4 * i] = acc[1][i];
                }
            }
            if (b + 1 < y.nblk) clear(b + 1, t, n);
        }
        half_sync(sys, n);
        float *own = y.column(b), *keep = y.Lb + (size_t)b * y.q1 * 256;
        if (wp == 0) {
            // the diagonal block: lane = row; then lane = column of the inverse
            float a[kNB], rd[kNB];
            const int r = lane & 15;
#pragma unroll
            for (int j = 0; j < kNB; j += 4) {
                const float4 v = ld4(P + r * kPS + j);
                a[j] = v.x, a[j + 1] = v.y, a[j + 2] = v.z, a[j + 3] = v.w;
            }
            bool ok = true;
#pragma unroll
            for (int k = 0; k < kNB; ++k) {
                const float d = __shfl_sync(0xffffffffu, a[k], k);
                asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rd[k]) : "f"(d));
                ok = ok && d > 0.f && d < 1e30f;
                const float l = a[k] * rd[k];
                a[k] = l;
#pragma unroll
                for (int j = k + 1; j < kNB; ++j) a[j] = fmaf(-l, __shfl_sync(0xffffffffu, l, j), a[j]);
            }
            if (lane < kNB)
#pragma unroll
                for (int j = 0; j < kNB; j += 4)
                    *reinterpret_cast<float4 *>(Li + r * kPS + j) = make_float4(a[j], a[j + 1], a[j + 2], a[j + 3]);
            __syncwarp();
            float x[kNB];
#pragma unroll
            for (int i = 0; i < kNB; ++i) {
                float l[kNB];
#pragma unroll
                for (int j = 0; j < i; j += 4) {
                    const float4 v = ld4(Li + i * kPS + j);
                    l[j] = v.x, l[j + 1] = v.y, l[j + 2] = v.z, l[j + 3] = v.w;
                }
                float s = i == r ? 1.f : 0.f;
#pragma unroll
                for (int j = 0; j < i; ++j) s = fmaf(-l[j], x[j], s);
                x[i] = s * rd[i];
            }
            __syncwarp();
            if (lane < kNB) {
#pragma unroll
                for (int i = 0; i < kNB; ++i) {
                    const float v = i >= r ? x[i] : 0.f;
                    Li[i * kPS + r] = v;
                    keep[i * kNB + r] = v;
                }
            }
            if (!ok && lane == 0) *fail = 1;
        } else {
            // the border rows of this block, before the diagonal solve, and
            // the next column's entries
            for (int i = t - 32; i < kNB * K; i += n - 32) {
                const int r = i & 15, k = i >> 4;
                float acc = y.Z[(size_t)k * y.npad + kNB * b + r];
                const int tm = min(q, b);
                for (int tt = 1; tt <= tm; ++tt) {
                    const float *ar = y.column(b - tt) + tt * y.bs + r * y.st, *zr = y.border(b - tt, k);
                    float s = 0.f;
#pragma unroll
                    for (int kk = 0; kk < kNB; kk += 4) s = dot4(ld4(ar + kk), ld4(zr + kk), s);
                    acc -= s;
                }
                T[i] = acc;
            }
            if (b + 1 < y.nblk) entries(b + 1, t - 32, n - 32);
        }
        half_sync(sys, n);
        if (*fail) return false;
        // L[b+s][b] = panel Linv^T, Z_b = Linv T
        for (int i = t; i < 64 * smax; i += n) {
            const int r = kNB + (i >> 2), c = i & 3;
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int k = 0; k < kNB; k += 4) {
                const float4 a = ld4(P + r * kPS + k);
#pragma unroll
                for (int u = 0; u < 4; ++u) acc[u] = dot4(a, ld4(Li + (c + 4 * u) * kPS + k), acc[u]);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                keep[r * kNB + c + 4 * u] = acc[u];   // block r / 16 of the column
                if (kFast) own[r * kPS + c + 4 * u] = acc[u];
            }
        }
        for (int i = t; i < kNB * K; i += n) {
            const int r = i & 15, k = i >> 4;
            float s = 0.f;
#pragma unroll
            for (int kk = 0; kk < kNB; kk += 4) s = dot4(ld4(Li + r * kPS + kk), ld4(T + kNB * k + kk), s);
            y.Z[(size_t)k * y.npad + kNB * b + r] = s;
            if (kFast) y.border(b, k)[r] = s;
        }
        half_sync(sys, n);
    }
    // Schur complement of the types, S = diag(vv) - Z^T Z
    float *S = y.S;
    const int np = K * (K + 1) / 2;
    for (int e = wp; e < np; e += nw) {
        int i = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);
        while ((i + 1) * (i + 2) / 2 <= e) ++i;
        while (i * (i + 1) / 2 > e) --i;
        const int j = e - i * (i + 1) / 2;
        const float *zi = y.Z + (size_t)i * y.npad, *zj = y.Z + (size_t)j * y.npad;
        float s = 0.f;
#pragma unroll 4
        for (int m = lane; m < y.npad; m += 32) s = fmaf(zi[m], zj[m], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) S[i * (K + 1) + j] = (i == j ? fmaf(w.vv[i], 1.f + 10.f * reg, 1e-12f) : 0.f) - s;
    }
    half_sync(sys, n);
    if (wp == 0) {
        bool ok = true;
        for (int k = 0; k < K; ++k) {
            const float d = S[k * (K + 1) + k];
            ok = ok && d > 0.f && isfinite(d);
            const float rd = rsqrtf(ok ? d : 1.f);
            __syncwarp();
            for (int i = k + lane; i < K; i += 32) S[i * (K + 1) + k] *= rd;   // the diagonal: sqrt(d)
            __syncwarp();
            for (int i = k + 1 + lane; i < K; i += 32) {
                const float l = S[i * (K + 1) + k];
                for (int j = k + 1; j <= i; ++j) S[i * (K + 1) + j] -= l * S[j * (K + 1) + k];
            }
            __syncwarp();
        }
        if (!ok && lane == 0) *fail = 1;
    }
    half_sync(sys, n);
    return *fail == 0;
}

// Solve one system with its factors: the right-hand side in y (antennas) and
// rk (types) is replaced by the solution.  Each block step uses one block
// column (the inverted diagonal block and the blocks below it), which
// cp.async brings into the ring several steps ahead; one barrier a step.
// Warp 0 closes a block and carries its nearest neighbour, the other warps
// handle the farther ones a step later (forward) or earlier (backward).
template <bool kFast>
__device__ __forceinline__ void lin_solve(const LinSys<kFast> &y, int sys, int t, int n) {
    const int lane = t & 31, wp = t >> 5, nw = n >> 5, q = y.q, nb = y.nblk, K = y.K;
    const int row = lane & 15, half = 8 * (lane >> 4);
    constexpr int st = LinSys<kFast>::st, bs = LinSys<kFast>::bs;
    float *v = y.y;
    const int chunks = y.q1 * 64;   // 16-byte pieces of a block column
    // warps 1.. fetch block column b into its slot (and close a copy group)
    auto fetch = [&](int b) {
        if (wp == 0) return;
        if (b >= 0 && b < nb) {
            const float *src = y.Lb + (size_t)b * y.q1 * 256;
            float *dst = y.column(b);
            for (int i = t - 32; i < chunks; i += n - 32)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                                 gc_smem_addr(dst + (i >> 2) * kPS + 4 * (i & 3))),
                             "l"(src + 4 * i)
                             : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // the slot of a column is refilled two steps after its last reader, so a
    // ring of 8 runs five columns ahead
    constexpr int kAhead = 5;
    auto landed = [&]() { asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory"); };
    constexpr bool ring = kFast;
    // ---- forward: y_b = Linv_b r_b, then r_{b+s} -= L[b+s][b] y_b
    if (ring) {
        for (int b = 0; b < kAhead; ++b) fetch(b);
        landed();
        half_sync(sys, n);
    }
    float carry = 0.f;   // warp 0: L[b][b-1] y_{b-1}
    for (int b = 0; b < nb; ++b) {
        if (ring) fetch(b + kAhead);
        if (wp == 0) {
            const float *c = y.column(b);
            const float r = v[kNB * b + row] - carry;
            const float4 l0 = ld4(c + row * st + half), l1 = ld4(c + row * st + half + 4);
            const float li[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) s = fmaf(li[i], __shfl_sync(0xffffffffu, r, half + i), s);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            if (lane < 16) v[kNB * b + row] = s;
            if (b + 1 < nb) {
                const float4 m0 = ld4(c + bs + row * st + half), m1 = ld4(c + bs + row * st + half + 4);
                const float mi[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                float u = 0.f;
#pragma unroll
                for (int i = 0; i < 8; ++i) u = fmaf(mi[i], __shfl_sync(0xffffffffu, s, half + i), u);
                carry = u + __shfl_xor_sync(0xffffffffu, u, 16);
            }
        } else if (b >= 1) {   // the farther blocks of column b - 1
            const float *c = y.column(b - 1);
            const float *yb = v + kNB * (b - 1) + half;
            for (int s = wp + 1; s <= q && b - 1 + s < nb; s += nw - 1) {
                const float *l = c + s * bs + row * st + half;
                float u = dot4(ld4(l), ld4(yb), dot4(ld4(l + 4), ld4(yb + 4), 0.f));
                u += __shfl_xor_sync(0xffffffffu, u, 16);
                if (lane < 16) v[kNB * (b - 1 + s) + row] -= u;
            }
        }
        if (ring) landed();
        half_sync(sys, n);
    }
    // ---- types: y_V = S^-1 (r_V - Z^T y), then y -= Z y_V
    float *rk = y.rk, *S = y.S;
    const float *Z = y.Z;
    for (int k = wp; k < K; k += nw) {
        const float *zk = Z + (size_t)k * y.npad;
        float s = 0.f;
#pragma unroll 8
        for (int m = lane; m < y.npad; m += 32) s = fmaf(zk[m], v[m], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) rk[k] -= s;
    }
    half_sync(sys, n);
    if (wp == 0) {
        // K <= 64: elements lane and lane + 32
        float x0 = lane < K ? rk[lane] : 0.f, x1 = lane + 32 < K ? rk[lane + 32] : 0.f;
        for (int k = 0; k < K; ++k) {
            const float xk = __fdividef(__shfl_sync(0xffffffffu, k < 32 ? x0 : x1, k & 31), S[k * (K + 1) + k]);
            if (lane == k) x0 = xk;
            if (lane + 32 == k) x1 = xk;
            if (lane > k && lane < K) x0 -= S[lane * (K + 1) + k] * xk;
            if (lane + 32 > k && lane + 32 < K) x1 -= S[(lane + 32) * (K + 1) + k] * xk;
        }
        for (int k = K - 1; k >= 0; --k) {
            const float xk = __fdividef(__shfl_sync(0xffffffffu, k < 32 ? x0 : x1, k & 31), S[k * (K + 1) + k]);
            if (lane == k) x0 = xk;
            if (lane + 32 == k) x1 = xk;
            if (lane < k) x0 -= S[k * (K + 1) + lane] * xk;
            if (lane + 32 < k) x1 -= S[k * (K + 1) + lane + 32] * xk;
        }
        if (lane < K) rk[lane] = x0;
        if (lane + 32 < K) rk[lane + 32] = x1;
    }
    if (ring)   // the first columns of the way back, meanwhile
        for (int b = nb - 1; b > nb - 1 - kAhead; --b) fetch(b);
    half_sync(sys, n);
    for (int m = t; m < y.npad; m += n) {
        float s = v[m];
#pragma unroll 4
        for (int k = 0; k < K; ++k) s -= Z[(size_t)k * y.npad + m] * rk[k];
        v[m] = s;
    }
    // (a backward step reads two columns: one more has to have landed)
    auto landed2 = [&]() { asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 2) : "memory"); };
    if (ring) landed2();
    half_sync(sys, n);
    // ---- backward: x_b = Linv_b^T (y_b - sum_s L[b+s][b]^T x_{b+s})
    const int np = min(nw - 1, q - 1);   // warps with farther neighbours
    auto dot8 = [&](const float *l, const float *u) {
        const float4 a = ld4(u), c = ld4(u + 4);
        const float s0 = fmaf(l[0], a.x, fmaf(l[st], a.y, fmaf(l[2 * st], a.z, l[3 * st] * a.w)));
        const float s1 = fmaf(l[4 * st], c.x, fmaf(l[5 * st], c.y, fmaf(l[6 * st], c.z, l[7 * st] * c.w)));
        return s0 + s1;
    };
    for (int b = nb - 1; b >= 0; --b) {
        if (ring) fetch(b - kAhead);
        if (wp == 0) {
            const float *c = y.column(b) + half * st + row;
            float s = b + 1 < nb ? dot8(c + bs, v + kNB * (b + 1) + half) : 0.f;
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            float r = v[kNB * b + row] - s;
            if (b + 2 < nb)
                for (int o = 1; o <= np; ++o) r -= y.part[((b & 1) * 16 + o) * kNB + row];
            float x = 0.f;
#pragma unroll
            for (int i = 0; i < 8; ++i) x = fmaf(c[i * st], __shfl_sync(0xffffffffu, r, half + i), x);
            x += __shfl_xor_sync(0xffffffffu, x, 16);
            if (lane < 16) v[kNB * b + row] = x;
        } else if (wp <= np && b >= 1) {   // the farther neighbours of block b - 1
            const float *c = y.column(b - 1) + half * st + row;
            float s = 0.f;
            for (int ss = wp + 1; ss <= q && b - 1 + ss < nb; ss += nw - 1)
                s += dot8(c + ss * bs, v + kNB * (b - 1 + ss) + half);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            if (lane < 16) y.part[(((b - 1) & 1) * 16 + wp) * kNB + row] = s;
        }
        if (ring) landed2();
        half_sync(sys, n);
    }
    if (ring) asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Right-hand sides of both systems from the gradient sums h (or a residual of
// the equations), in the normalised coordinates of the factors: only h carries
// the caller's precision, the rest is FP32 like the factors.  Right-hand side
// and step go through relative changes dg / g by the amplitudes the factors
// were made with, so that factors of an earlier point differ from the present
// matrix by the pair weights alone.  (A zero amplitude has its gradient itself.)
template <class R>
__device__ void lin_rhs(const LinWork<R> &w, const LinShape &sh, int N, int K, const V2<R> *h, R am, R vm) {
    const R s2 = 1 / (am * am * vm * am * am * vm);
    for (int m = threadIdx.x; m < sh.npad; m += blockDim.x) {
        float bx = 0.f, by = 0.f;
        if (m < N) {
            const float f = w.fa[m];
            const R z = f > 0.f ? s2 : s2 * am;
            bx = __fdividef((float)(h[m].x * z), f > 0.f ? f : 1.f);
            by = __fdividef((float)(h[m].y * z), f > 0.f ? f : 1.f);
        }
        w.y[m] = bx;
        w.y[sh.npad + m] = by;
    }
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
        const float f = w.fv[k];
        const R z = f > 0.f ? s2 : s2 * vm;
        w.rk[k] = __fdividef((float)(h[N + k].x * z), f > 0.f ? f : 1.f);
        w.rk[K + k] = __fdividef((float)(h[N + k].y * z), f > 0.f ? f : 1.f);
    }
    __syncthreads();
}

// rs = hs - A qt in relative coordinates: pair p = (i, j) of weight
// W = |g_i|^2 |g_j|^2 |V|^2 adds W s to row i and to its type's row and W conj(s) to
// row j, s = q_i + conj(q_j) + w_k (the layout of lin_resid's passes).
template <class R>
__device__ void lin_residual(const CalParams &p, const LinWork<R> &w, const LinTypes &ty) {
    const int L = p.L, N = p.N, K = p.n_ubl, nt = blockDim.x;
    for (int e = threadIdx.x; e < N + K; e += nt) w.G[e] = w.x[e].x * w.x[e].x + w.x[e].y * w.x[e].y;
    __syncthreads();
    for (int m = threadIdx.x; m < N; m += nt) {
        const int mx = m % L, my = m / L;
        const V2<R> qm = w.qt[m];
        const R Gm = w.G[m];
        V2<R> s = w.hs[m];
        for (int k = 0; k < K; ++k) {
            const int4 a = ty.a[k];
            V2<R> t{0, 0};
            if ((unsigned)(mx - a.x) < (unsigned)L && (unsigned)(my - a.y) < (unsigned)L) {
                const V2<R> qj = w.qt[m - a.z], v = w.qt[N + k];
                const R W = Gm * w.G[m - a.z] * w.G[N + k];
                t.x = W * (qm.x + qj.x + v.x);
                t.y = W * (qm.y - qj.y + v.y);
                s.x -= t.x;
                s.y -= t.y;
            }
            w.h[(size_t)k * N + m] = t;
        }
        w.rs[m] = s;
    }
    __syncthreads();
    for (int m = threadIdx.x; m < N; m += nt) {
        const int mx = m % L, my = m / L;
        V2<R> s = w.rs[m];
        for (int k = 0; k < K; ++k) {
            const int4 a = ty.a[k];
            if ((unsigned)(mx + a.x) < (unsigned)L && (unsigned)(my + a.y) < (unsigned)L) {
                const V2<R> t = w.h[(size_t)k * N + m + a.z];
                s.x -= t.x;
                s.y += t.y;
            }
        }
        w.rs[m] = s;
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = nt >> 5;
    for (int k = wp; k < K; k += nw) {
        const V2<R> *t = w.h + (size_t)k * N;
        V2<R> s{0, 0};
#pragma unroll 4
        for (int m = lane; m < N; m += 32) {
            s.x += t[m].x;
            s.y += t[m].y;
        }
        for (int o = 16; o > 0; o >>= 1) {
            s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
            s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
        }
        if (lane == 0) w.rs[N + k] = V2<R>{w.hs[N + k].x - s.x, w.hs[N + k].y - s.y};
    }
    __syncthreads();
}

// Sums over the CTA (up to 16 warps; red: [16][NV + 2]), the warps' parts added by one
// thread per value: an FP64 sum by every thread would cost as much as a pass.
template <class T, int NV>
__device__ void lean_sum(T (&v)[NV], T *red) {
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q)
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
    if (lane == 0)
#pragma unroll
        for (int q = 0; q < NV; ++q) red[q * 16 + wp] = v[q];
    __syncthreads();
    if (threadIdx.x < NV) {
        T s = red[threadIdx.x * 16];
        for (int u = 1; u < nw; ++u) s += red[threadIdx.x * 16 + u];
        red[threadIdx.x * 16] = s;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = red[q * 16];
    __syncthreads();
}

struct LinNorms {
    double d2, x2;   // |step|^2, |point|^2
    float rel;       // largest |step|^2 / |element|^2
};

// The step in (g, V) from the solution of both systems (kRefined: from the
// refined relative step), with the degeneracy directions (Sec. 5.2) projected
// out: amplitude (g | -2 V), phase (i g | 0), slopes (i x g | -i dx V),
// (i y g | -i dy V); amplitude is orthogonal to the other three.  Arithmetic in T, on
// elements scaled by sc.  Writes the step and the trial point.
template <class R, class T, bool kRefined>
__device__ LinNorms lin_step(const CalParams &p, const LinWork<R> &w, const LinShape &sh, const LinTypes &ty, R am,
                             R vm, T *red) {
    const int N = p.N, K = p.n_ubl, L = p.L, ne = N + K, nt = blockDim.x;
    const R unit = fmax(am, vm), sc = 1 / unit;
    const T ua = (T)(am * sc), uv = (T)(vm * sc);
    T acc[12];
#pragma unroll
    for (int u = 0; u < 12; ++u) acc[u] = 0;
    for (int e = threadIdx.x; e < ne; e += nt) {
        const V2<R> z = w.x[e];
        const V2<T> g{(T)(z.x * sc), (T)(z.y * sc)};
        V2<T> d;
        if (kRefined) {
            const T qx = (T)w.qt[e].x, qy = (T)w.qt[e].y;
            d.x = g.x * qx - g.y * qy;
            d.y = g.x * qy + g.y * qx;
        } else {
            const float qx = e < N ? w.y[e] : w.rk[e - N], qy = e < N ? w.y[sh.npad + e] : w.rk[K + e - N];
            const float f = e < N ? w.fa[e] : w.fv[e - N];
            if (f > 0.f) {
                const T rx = (T)__fdividef(qx, f), ry = (T)__fdividef(qy, f);
                d.x = g.x * rx - g.y * ry;
                d.y = g.x * ry + g.y * rx;
            } else {
                d.x = (e < N ? ua : uv) * (T)qx;
                d.y = (e < N ? ua : uv) * (T)qy;
            }
        }
        w.dl[e] = V2<R>{(R)d.x, (R)d.y};
        const T a2 = g.x * g.x + g.y * g.y, re = g.x * d.x + g.y * d.y, im = g.x * d.y - g.y * d.x;
        acc[11] += a2;
        if (e < N) {
            const T X = (T)(e % L), Y = (T)(e / L);
            acc[0] += a2;
            acc[1] += a2;
            acc[2] += X * a2;
            acc[3] += Y * a2;
            acc[4] += X * X * a2;
            acc[5] += X * Y * a2;
            acc[6] += Y * Y * a2;
            acc[7] += re;
            acc[8] += im;
            acc[9] += X * im;
            acc[10] += Y * im;
        } else {
            const T X = (T)ty.a[e - N].x, Y = (T)ty.a[e - N].y;
            acc[0] += 4 * a2;
            acc[4] += X * X * a2;
            acc[5] += X * Y * a2;
            acc[6] += Y * Y * a2;
            acc[7] -= 2 * re;
            acc[9] -= X * im;
            acc[10] -= Y * im;
        }
    }
    lean_sum<T, 12>(acc, red);
    const T gram[14] = {acc[0], 0, acc[1], 0, acc[2], acc[4], 0, acc[3], acc[5], acc[6], acc[7], acc[8], acc[9], acc[10]};
    T cv[4];
    solve_gram4<T>(gram, cv);
    LinNorms n;
    n.x2 = (double)acc[11];
    float d2[1] = {0.f}, rel = 0.f;
    for (int e = threadIdx.x; e < ne; e += nt) {
        const V2<R> z = w.x[e];
        const V2<T> g{(T)(z.x * sc), (T)(z.y * sc)};
        T ca, cp;   // step -= (ca + i cp) g
        if (e < N) {
            ca = cv[0];
            cp = cv[1] + cv[2] * (T)(e % L) + cv[3] * (T)(e / L);
        } else {
            ca = -2 * cv[0];
            cp = -cv[2] * (T)ty.a[e - N].x - cv[3] * (T)ty.a[e - N].y;
        }
        const T dx = (T)w.dl[e].x - (ca * g.x - cp * g.y), dy = (T)w.dl[e].y - (ca * g.y + cp * g.x);
        const V2<R> st{unit * (R)dx, unit * (R)dy};
        w.dl[e] = st;
        w.tr[e] = V2<R>{z.x + st.x, z.y + st.y};
        const float fx = (float)dx, fy = (float)dy, gx = (float)g.x, gy = (float)g.y, q2 = fx * fx + fy * fy;
        d2[0] += q2;
        rel = fmaxf(rel, __fdividef(q2, gx * gx + gy * gy));
    }
    for (int o = 16; o > 0; o >>= 1) rel = fmaxf(rel, __shfl_xor_sync(0xffffffffu, rel, o));
    float *fr = reinterpret_cast<float *>(red + 16 * 12);
    if ((threadIdx.x & 31) == 0) fr[16 + (threadIdx.x >> 5)] = rel;
    lean_sum<float, 1>(d2, fr);
    for (int u = 0; u < nt / 32; ++u) rel = fmaxf(rel, fr[16 + u]);
    n.d2 = (double)d2[0];
    n.rel = rel;
    __syncthreads();
    return n;
}

template <class R, bool kFast>
__global__ void __launch_bounds__(kLThreads, 1) lincal_kernel(const CalParams p, const LinShape sh) {
    extern __shared__ __align__(128) char arena[];
    __shared__ R red[64];
    __shared__ float redf[16 * 12 + 32];
    __shared__ double redd2[16 * 12 + 32];
    __shared__ double redd[64];
    __shared__ LinTypes ty;
    __shared__ int s_fail[2], s_late;
    const int N = p.N, K = p.n_ubl, L = p.L, nt = blockDim.x, ne = N + K;
    const int hn = nt / 2, sys = threadIdx.x >= hn ? 1 : 0, ht = threadIdx.x - sys * hn;
    LinWork<R> w;
    lin_global<R>(w, p.work + (size_t)blockIdx.x * p.work_per_cta, N, K, sh);
    lin_shared<R, kFast>(w, arena, K, sh);
    const LinSys<kFast> ls(w, sh, K, sys);
    for (int k = threadIdx.x; k < K; k += nt) {
        const int dx = p.types[2 * k], dy = p.types[2 * k + 1], W = L - abs(dx);
        ty.a[k] = make_int4(dx, dy, dy * L + dx, 0);
        ty.b[k] = make_int2(p.type_ptr[k] - max(0, -dy) * W - max(0, -dx), W);
        ty.inv[k] = 1.0f / (float)(p.win_t1[k] - p.win_t0[k]);
    }
    __syncthreads();
    constexpr R kRise = sizeof(R) == 8 ? (R)1e-12 : (R)1e-6;   // rounding of chi^2 in the line search
    for (int c = blockIdx.x; c < p.C; c += gridDim.x) {
        const uint64_t t_start = gc_globaltimer();
        R *xr = reinterpret_cast<R *>(w.x);
        if (p.warm) {
            for (int i = threadIdx.x; i < N; i += nt) {
                const float2 g = p.gains[(size_t)c * N + i];
                w.x[i] = V2<R>{(R)g.x, (R)g.y};
            }
            for (int k = threadIdx.x; k < K; k += nt) {
                const float2 v = p.vmodel[(size_t)c * K + k];
                w.x[N + k] = V2<R>{(R)v.x, (R)v.y};
            }
            __syncthreads();
        } else {
            start_point<R>(p, c, xr, xr + 2 * N, red, reinterpret_cast<R *>(w.dl));
        }
        int st = GC_ENOCONV, it = 1;
        R chi2 = lin_resid<R>(p, c, w.x, w, ty, red);
        R am = 1, vm = 1;
        float moved = 0.f;   // largest relative change of an element since the factors were made
        bool factor = true, big = true;
        for (;;) {
            if (factor) {
                // FP32 factors with a relative shift of 1e-6; a matrix too
                // close to singular for it is shifted more (the step is then
                // shorter in its softest directions, the fixed point the same)
                bool ok = lin_prepare<R>(p, w, sh, ty, red, am, vm);
                if (ok) {
                    for (float reg = 1e-6f; reg < 0.1f; reg *= 100.f) {
                        if (reg > 2e-6f) lin_prepare<R>(p, w, sh, ty, red, am, vm);   // the border is overwritten
                        if (threadIdx.x < 2) s_fail[threadIdx.x] = 0;
                        __syncthreads();
                        lin_factor<R, kFast>(p, w, ls, ty, sys, ht, hn, reg, &s_fail[sys]);
                        __syncthreads();
                        ok = s_fail[0] == 0 && s_fail[1] == 0;
                        __syncthreads();
                        if (ok) break;
                    }
                }
                if (!ok) {
                    st = GC_EDEGEN;
                    break;
                }
            }
            // A step of FP32 factors errs by about 1e-6 of itself, which the next
            // steps repair but for what it moves along the degeneracies; while
            // the steps are large enough for that to show in the output's
            // binary32 digits, one pass of iterative refinement in R makes
            // them exact to R's own conditioning
            const bool refine = sizeof(R) == 8 && big;
            lin_rhs<R>(w, sh, N, K, w.hs, am, vm);
            lin_solve<kFast>(ls, sys, ht, hn);
            __syncthreads();
            LinNorms nm;
            if (refine) {
                bool zero = false;   // (relative steps need nonzero amplitudes)
                for (int e = threadIdx.x; e < ne; e += nt) {
                    const float f = e < N ? w.fa[e] : w.fv[e - N];
                    const float qx = e < N ? w.y[e] : w.rk[e - N], qy = e < N ? w.y[sh.npad + e] : w.rk[K + e - N];
                    zero = zero || f == 0.f;
                    w.qt[e] = V2<R>{(R)__fdividef(qx, f), (R)__fdividef(qy, f)};
                }
                if (!__syncthreads_or(zero)) {
                    lin_residual<R>(p, w, ty);
                    lin_rhs<R>(w, sh, N, K, w.rs, am, vm);
                    lin_solve<kFast>(ls, sys, ht, hn);
                    __syncthreads();
                    for (int e = threadIdx.x; e < ne; e += nt) {
                        const float f = e < N ? w.fa[e] : w.fv[e - N];
                        const float qx = e < N ? w.y[e] : w.rk[e - N], qy = e < N ? w.y[sh.npad + e] : w.rk[K + e - N];
                        w.qt[e].x += (R)__fdividef(qx, f);
                        w.qt[e].y += (R)__fdividef(qy, f);
                    }
                    __syncthreads();
                    nm = lin_step<R, R, true>(p, w, sh, ty, am, vm, reinterpret_cast<R *>(redd2));
                } else {
                    nm = lin_step<R, R, false>(p, w, sh, ty, am, vm, reinterpret_cast<R *>(redd2));
                }
            } else {
                nm = lin_step<R, float, false>(p, w, sh, ty, am, vm, redf);
            }
            // halving line search on chi^2; the pass that tries a point is
            // also the next iteration's gradient there
            R step = 1, c2 = 0;
            if (threadIdx.x == 0) s_late = out_of_time(p, t_start);   // (lin_resid has barriers)
            for (int ls = 0;; ++ls) {
                c2 = lin_resid<R>(p, c, w.tr, w, ty, red);
                if (c2 <= chi2 * (1 + kRise) + (R)1e-30 || ls == 7) break;
                step *= (R)0.5;
                __syncthreads();
                for (int e = threadIdx.x; e < ne; e += nt)
                    w.tr[e] = V2<R>{w.x[e].x + step * w.dl[e].x, w.x[e].y + step * w.dl[e].y};
                __syncthreads();
            }
            chi2 = c2;
            V2<R> *const old = w.x;
            w.x = w.tr;
            w.tr = old;
            if ((double)step * sqrt(nm.d2) <= p.tol * sqrt(nm.x2)) {
                st = GC_OK;
                break;
            }
            if (s_late) {
                st = GC_ETIMEOUT;
                if (threadIdx.x == 0) atomicOr(p.status, GC_DEV_TIMEOUT_CAL);
                break;
            }
            if (++it > p.max_iter) break;
            // The pair weights are products of the amplitudes, so factors made
            // before every element moved by at most a fraction e precondition
            // the present matrix within 8 e, whatever its condition: they are
            // kept while that adds at most a twelfth to a step's error (a
            // Gauss-Newton step on noisy data leaves about as much itself) and
            // the steps are small
            moved += (float)step * sqrtf(nm.rel);
            big = nm.d2 > 4e-4 * nm.x2;
            factor = step < (R)1 || nm.d2 > 1e-6 * nm.x2 || !(moved < 0.01f);
            if (factor) moved = 0.f;
        }
        __syncthreads();
        xr = reinterpret_cast<R *>(w.x);
        finish_channel<R>(p, c, xr, xr + 2 * N, min(it, p.max_iter), st, redd);
    }
}

}  // namespace

gc_status gc_lincal_run(gc_ctx *ctx, CalParams &p, bool fp64, cudaStream_t s) {
    const LinShape sh = lin_shape(p.N, p.band, p.n_ubl);
    size_t per_cta, smem;
    const void *kfn;
    auto pick = [&](auto real, auto fast) {
        using R = decltype(real);
        constexpr bool kFast = decltype(fast)::value;
        LinWork<R> w;
        per_cta = lin_global<R>(w, nullptr, p.N, p.n_ubl, sh);
        smem = lin_shared<R, kFast>(w, nullptr, p.n_ubl, sh);
        kfn = (const void *)lincal_kernel<R, kFast>;
    };
    if (fp64) sh.fast ? pick(double(), std::true_type()) : pick(double(), std::false_type());
    else sh.fast ? pick(float(), std::true_type()) : pick(float(), std::false_type());
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLSmem);
    if (e != cudaSuccess) return gc_cuda_fail(ctx, e, "cudaFuncSetAttribute(lincal)");
    // small arrays: fewer warps (a block column holds little work) and more
    // CTAs on an SM
    const int nthr = p.N > 400 ? 512 : (p.N > 128 ? 256 : 128);
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kfn, nthr, smem);
    if (e != cudaSuccess || occ < 1) return gc_cuda_fail(ctx, e, "occupancy(calibration)");
    if (ctx->tune[GC_TUNE_CAL_CTAS] > 0) occ = std::min(occ, ctx->tune[GC_TUNE_CAL_CTAS]);
    const int grid = std::min(p.C, occ * ctx->sm_count);
    const gc_status st = gc_scratch_reserve(ctx, per_cta * grid);
    if (st != GC_OK) return st;
    p.work = static_cast<char *>(ctx->scratch);
    p.work_per_cta = per_cta;
    const int rec = gc_prof_begin(ctx, s, fp64 ? "lincal_fp64" : "lincal_fp32");
    void *args[] = {&p, const_cast<LinShape *>(&sh)};
    e = cudaLaunchKernel(kfn, dim3(grid), dim3(nthr), args, smem, s);
    gc_prof_end(ctx, s, rec);
    if (e != cudaSuccess) return gc_cuda_fail(ctx, e, "launch calibration");
    return GC_OK;
}
