// ew_mg_fused.cu -- fused pieces of the multigrid V-cycle (ew_mg.cu), for the
// levels where a launch per elementary operation would cost more than its work:
//
//   k_mg_smooth2d           2D levels: one or two smoothing sweeps (damped
//                           Jacobi, or all colours of a multi-colour
//                           Gauss-Seidel sweep) per launch on overlapped tiles
//                           in shared memory, with the prolongation of the
//                           coarse correction added while the tile is staged
//   k_mg_resid_restrict2d   2D levels: residual and full weighting
//   k_mg_bottom             the rest of the cycle from a small level down to
//                           the coarsest and back, one launch of one CTA
//
// A sweep, a residual and a restriction take the operations of one elementary
// kernel a point in their order, whichever form a level takes.  Two things differ
// between the forms, by rounding: the prolongation adds the four coarse values in
// pairs in k_mg_smooth2d and one by one in k_mg_bottom, and the coarsest level is
// solved by sine transforms in k_mg_bottom (up to kMgSineMax points an axis) but by
// conjugate gradients in a launch of its own (k_mg_coarse_cg).
#include <math.h>

#include <algorithm>

#include "ew_internal.h"
#include "ew_mg.cuh"

namespace ew {

__device__ __forceinline__ float m_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float m_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float m_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double m_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double m_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double m_fma(double a, double b, double c) { return __fma_rn(a, b, c); }

// x + P e at fine point (i, j) of a 2D level: an odd index lies on coarse
// point (i - 1) / 2, an even one between two (1/2 each).  PI, PJ: the parities
// (0: even), so that a warp of one parity does no more FP64 work than it needs
template <typename T, int PI, int PJ>
__device__ __forceinline__ T corrected(T x, const T* __restrict__ e, int i, int j, int cx, int cy) {
    const int I = PI ? i >> 1 : (i >> 1) - 1, J = PJ ? j >> 1 : (j >> 1) - 1;
    const T* p = e + (int64_t)J * cx + I;
    const bool i0 = I >= 0, i1 = I + 1 < cx, j0 = J >= 0, j1 = J + 1 < cy;  // an odd index's own point always exists
    if (PI && PJ) return m_add(x, p[0]);
    if (PI) return m_fma(T(0.5), m_add(j0 ? p[0] : T(0), j1 ? p[cx] : T(0)), x);
    if (PJ) return m_fma(T(0.5), m_add(i0 ? p[0] : T(0), i1 ? p[1] : T(0)), x);
    const T a = m_add(i0 && j0 ? p[0] : T(0), i1 && j0 ? p[1] : T(0));
    const T b = m_add(i0 && j1 ? p[cx] : T(0), i1 && j1 ? p[cx + 1] : T(0));
    return m_fma(T(0.25), m_add(a, b), x);
}
template <typename T>
__device__ __forceinline__ T corrected(T x, const T* __restrict__ e, int i, int j, int cx, int cy) {
    if (i & 1) return (j & 1) ? corrected<T, 1, 1>(x, e, i, j, cx, cy) : corrected<T, 1, 0>(x, e, i, j, cx, cy);
    return (j & 1) ? corrected<T, 0, 1>(x, e, i, j, cx, cy) : corrected<T, 0, 0>(x, e, i, j, cx, cy);
}

template <typename T>
__global__ void k_mg_prolong2d(int nx, int ny, int cx, int cy, const T* __restrict__ ec, T* __restrict__ x) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= nx) return;
    const int64_t q = (int64_t)j * nx + i;
    x[q] = corrected(x[q], ec, i, j, cx, cy);
}

// Smoothing on overlapped tiles.  A CTA stages x (plus P e, when ec is given)
// and b over its TILE x TILE tile with a halo of one stencil reach per pass
// (a pass: one Jacobi sweep, or one colour), runs the passes in shared memory
// on regions that shrink by the reach, and writes its tile to xo.  A colour
// pass gives every lane a point of that colour (the elementary kernel idled
// all lanes of the other colours).  Dirichlet closure: walls hold 0; the
// fourth-order stencil's point beyond a wall is the negated mirror, which is
// the point itself at the wall's neighbour.
//
// FP64 levels are bound by the FP64 units (two operations a clock and SM): eight
// operations a point and sweep.  The update stays in the residual form all the
// same: with its constants multiplied out (k0 x + w b + sum w c_i (neighbour
// sums), four or five operations) a sweep rounds differently from the residual
// that the stopping test sees, and the lowest ||b - M x|| / ||b|| that a solve
// reaches rises by up to 2.9 times (order 4, colour sweeps, 255^2; 1.4 and 2.0 on
// 1023^2 at order 2).
// Why: at 1023^2 in FP64 a V(2,2) cycle issued 88 launches of 2-16 us; the
// halo costs 20 % more points at TILE 32 (two red-black sweeps), 42 % at 16.
template <typename T, int ORDER, bool GS, int NS, int TILE>
struct Smooth2dShape {
    static constexpr int R = ORDER == 2 ? 1 : 2;
    static constexpr int NC = GS ? (ORDER == 2 ? 2 : 3) : 1;  // passes a sweep
    static constexpr int P = NC * NS, H = R * P;
    static constexpr int SX = TILE + 2 * H, SB = TILE + 2 * (H - R);
    static constexpr size_t SMEM = sizeof(T) * ((size_t)(GS ? 1 : 2) * SX * SX + (size_t)SB * SB);
};

template <typename T, int ORDER, bool GS, int NS, int TILE>
__global__ void __launch_bounds__(256)
    k_mg_smooth2d(int nx, int ny, const T* __restrict__ x, const T* __restrict__ b, T* __restrict__ xo, Stencil<T> sa,
                  T wd, const T* __restrict__ ec, int cx, int cy) {
    using S = Smooth2dShape<T, ORDER, GS, NS, TILE>;
    constexpr int R = S::R, H = S::H, SX = S::SX, SB = S::SB, NC = S::NC, P = S::P;
    extern __shared__ __align__(16) unsigned char smem_ms[];
    T* cur = reinterpret_cast<T*>(smem_ms);
    T* nxt = GS ? cur : cur + SX * SX;
    T* sb = cur + (GS ? 1 : 2) * SX * SX;
    const int x0 = blockIdx.x * TILE, y0 = blockIdx.y * TILE, tid = threadIdx.x;
    // staged point s of parity class (s & 1): H and the tile's origin are even
    constexpr int S2 = SX / 2, CLS = S2 * S2;
    auto stage = [&](int cls, int r) {
        const int sy = 2 * (r / S2) + (cls >> 1), sx = 2 * (r % S2) + (cls & 1);
        const int gx = x0 - H + sx, gy = y0 - H + sy;
        T v = T(0);
        if (gx >= 0 && gx < nx && gy >= 0 && gy < ny) {
            v = x[(int64_t)gy * nx + gx];
            if (ec) {
                if (cls == 0)
                    v = corrected<T, H & 1, H & 1>(v, ec, gx, gy, cx, cy);
                else if (cls == 1)
                    v = corrected<T, (H + 1) & 1, H & 1>(v, ec, gx, gy, cx, cy);
                else if (cls == 2)
                    v = corrected<T, H & 1, (H + 1) & 1>(v, ec, gx, gy, cx, cy);
                else
                    v = corrected<T, (H + 1) & 1, (H + 1) & 1>(v, ec, gx, gy, cx, cy);
            }
        }
        cur[sy * SX + sx] = v;
        if (!GS) nxt[sy * SX + sx] = T(0);
    };
    if (ec) {
#pragma unroll
        for (int cls = 0; cls < 4; ++cls)
            for (int r = tid; r < CLS; r += 256) stage(cls, r);
    } else {
        for (int q = tid; q < SX * SX; q += 256) {
            const int sy = q / SX, sx = q - sy * SX;
            const int gx = x0 - H + sx, gy = y0 - H + sy;
            cur[q] = (gx >= 0 && gx < nx && gy >= 0 && gy < ny) ? x[(int64_t)gy * nx + gx] : T(0);
            if (!GS) nxt[q] = T(0);
        }
    }
    for (int q = tid; q < SB * SB; q += 256) {
        const int sy = q / SB, sx = q - sy * SB;
        const int gx = x0 - (H - R) + sx, gy = y0 - (H - R) + sy;
        sb[q] = (gx >= 0 && gx < nx && gy >= 0 && gy < ny) ? b[(int64_t)gy * nx + gx] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int e = R * (P - 1 - p);  // the pass covers the tile and e points around it
        const int W = TILE + 2 * e, WC = (W + NC - 1) / NC;
        for (int q = tid; q < WC * W; q += 256) {
            const int ry = q / WC, rc = q - ry * WC;
            const int gy = y0 - e + ry;
            int rx = rc;
            if (GS) {
                if (ORDER == 2) {
                    rx = 2 * rc + ((x0 - e + gy + p) & 1);
                } else {
                    int m = (p - (x0 - e) - gy) % 3;
                    if (m < 0) m += 3;
                    rx = 3 * rc + m;
                }
            }
            const int gx = x0 - e + rx;
            if (rx >= W || gx < 0 || gx >= nx || gy < 0 || gy >= ny) continue;
            const int c = (ry + H - e) * SX + rx + H - e;
            const T u = cur[c];
            const T bv = sb[(ry + H - R - e) * SB + rx + H - R - e];
            const T s1x = m_add(cur[c - 1], cur[c + 1]), s1y = m_add(cur[c - SX], cur[c + SX]);
            T s2x = T(0), s2y = T(0);
            if (ORDER == 4) {
                const T xl = gx == 0 ? -u : cur[c - 2], xh = gx == nx - 1 ? -u : cur[c + 2];
                const T yl = gy == 0 ? -u : cur[c - 2 * SX], yh = gy == ny - 1 ? -u : cur[c + 2 * SX];
                s2x = m_add(xl, xh);
                s2y = m_add(yl, yh);
            }
            T lap = m_mul(sa.c0, u);
            lap = m_fma(sa.c1[0], s1x, lap);
            lap = m_fma(sa.c1[1], s1y, lap);
            if (ORDER == 4) {
                lap = m_fma(sa.c2[0], s2x, lap);
                lap = m_fma(sa.c2[1], s2y, lap);
            }
            nxt[c] = m_fma(wd, m_add(m_add(bv, -u), lap), u);
        }
        __syncthreads();
        if (!GS) {
            T* t = cur;
            cur = nxt;
            nxt = t;
        }
    }
    for (int q = tid; q < TILE * TILE; q += 256) {
        const int ty = q / TILE, tx = q - ty * TILE;
        if (x0 + tx < nx && y0 + ty < ny) xo[(int64_t)(y0 + ty) * nx + x0 + tx] = cur[(ty + H) * SX + tx + H];
    }
}

// residual of a fine tile in shared memory, restricted to 32 x 8 coarse points; x_c = 0
constexpr int kRrX = 32, kRrY = 8;
template <typename T, int ORDER>
__global__ void __launch_bounds__(256)
    k_mg_resid_restrict2d(int nx, int ny, int cx, int cy, const T* __restrict__ x, const T* __restrict__ b,
                          T* __restrict__ bc, T* __restrict__ xc, Stencil<T> sa) {
    constexpr int FX = 2 * kRrX + 1, FY = 2 * kRrY + 1;
    __shared__ T sr[FY * FX];
    const int I0 = blockIdx.x * kRrX, J0 = blockIdx.y * kRrY;
    for (int q = threadIdx.x; q < FX * FY; q += 256) {
        const int sy = q / FX, sx = q - sy * FX;
        const int i = 2 * I0 + sx, j = 2 * J0 + sy;
        T r = T(0);
        if (i < nx && j < ny) {
            const int64_t p = (int64_t)j * nx + i;
            r = (b[p] - x[p]) + lap_global<T, 2, ORDER>(x, sa, p, i, j, 0, nx, ny, 1);
        }
        sr[q] = r;
    }
    __syncthreads();
    const int tx = threadIdx.x % kRrX, ty = threadIdx.x / kRrX, I = I0 + tx, J = J0 + ty;
    if (I >= cx || J >= cy) return;
    const T w[3] = {T(0.25), T(0.5), T(0.25)};
    T s = T(0);
#pragma unroll
    for (int oy = 0; oy < 3; ++oy)
#pragma unroll
        for (int ox = 0; ox < 3; ++ox) s += w[ox] * w[oy] * sr[(2 * ty + oy) * FX + 2 * tx + ox];
    bc[(int64_t)J * cx + I] = s;
    xc[(int64_t)J * cx + I] = T(0);
}

// partial sums of |b - M x|^2 (the stopping test of a solve: no residual field is
// written or read back)
template <typename T, int ORDER>
__global__ void __launch_bounds__(256)
    k_mg_resid_norm2d(int nx, int ny, const T* __restrict__ x, const T* __restrict__ b, Stencil<T> sa,
                      double* __restrict__ part) {
    __shared__ double sh[8];
    double s = 0.0;
    const int segs = (nx + 255) / 256;  // a block takes 256 points of a row at a time
    for (int64_t q = blockIdx.x; q < (int64_t)segs * ny; q += gridDim.x) {
        const int j = (int)(q / segs), i = (int)(q - (int64_t)j * segs) * 256 + threadIdx.x;
        if (i >= nx) continue;
        const int64_t p = (int64_t)j * nx + i;
        const double r = (double)((b[p] - x[p]) + lap_global<T, 2, ORDER>(x, sa, p, i, j, 0, nx, ny, 1));
        s = fma(r, r, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += sh[w];
        part[blockIdx.x] = s;
    }
}

// ---------------------------------------------------------------------------
// The bottom of the cycle in one CTA: from a small level down to the coarsest
// and back, every level's fields in shared memory, a CTA barrier between
// phases (a sweep or a colour, residual, restriction, prolongation).
// Why: a small level's launch takes 4-8 us whatever its work, a phase here a
// fraction of one; from 31^2 (FP64) a V(2,2) red-black cycle was 34 launches.
// (The same phases on a cluster of 8-16 CTAs with the fields in L2 took
// 1-3 us each: 96 us from 63^2.)
// ---------------------------------------------------------------------------
constexpr int kBotThreads = 512;

template <typename T>
__device__ __forceinline__ T bnb(const T* u, int q, int stride, int i, int n, int off) {
    const int p = i + off;
    if (p >= 0 && p < n) return u[q + off * stride];
    if (p == -1 || p == n) return T(0);
    const int m = p < 0 ? -2 - p : 2 * n - p;  // the odd mirror
    return -u[q + (m - i) * stride];
}
// sum of c_i (neighbour sums), in the order of lap_global, from r
template <typename T, int DIM, int ORDER>
__device__ __forceinline__ T bsum(const T* u, const Stencil<T>& s, T r, int q, int i, int j, int k, int nx, int ny,
                                  int nz) {
    r += s.c1[0] * (bnb(u, q, 1, i, nx, -1) + bnb(u, q, 1, i, nx, 1));
    r += s.c1[1] * (bnb(u, q, nx, j, ny, -1) + bnb(u, q, nx, j, ny, 1));
    if (DIM == 3) r += s.c1[2] * (bnb(u, q, nx * ny, k, nz, -1) + bnb(u, q, nx * ny, k, nz, 1));
    if (ORDER == 4) {
        r += s.c2[0] * (bnb(u, q, 1, i, nx, -2) + bnb(u, q, 1, i, nx, 2));
        r += s.c2[1] * (bnb(u, q, nx, j, ny, -2) + bnb(u, q, nx, j, ny, 2));
        if (DIM == 3) r += s.c2[2] * (bnb(u, q, nx * ny, k, nz, -2) + bnb(u, q, nx * ny, k, nz, 2));
    }
    return r;
}

// M x = b on the coarsest level by sine transforms (the eigenvectors of the
// stencil with its odd closure), in FP64 with the eigenvalues of the stored
// stencil, up to kMgSineMax points per axis: tmp holds 2 N doubles.
// 3 x 3 points in FP64: conjugate gradients took 10 us, this form 1 us.
template <typename T, int DIM>
__device__ void coarse_sine(int nx, int ny, int nz, const T* b, T* x, const MgSine& sn, double* tmp) {
    const int N = nx * ny * nz, tid = threadIdx.x;
    double* u = tmp;
    double* v = tmp + N;
    for (int q = tid; q < N; q += kBotThreads) u[q] = (double)b[q];
    __syncthreads();
    auto axis = [&](int a, int stride, int n) {  // v = S_a u, then exchange
        for (int q = tid; q < N; q += kBotThreads) {
            const int k = (q / stride) % n;
            double s = 0.0;
            for (int j = 0; j < n; ++j) s = fma(sn.s[a][k * n + j], u[q + (j - k) * stride], s);
            v[q] = s;
        }
        double* t = u;
        u = v;
        v = t;
        __syncthreads();
    };
    axis(0, 1, nx);
    axis(1, nx, ny);
    if (DIM == 3) axis(2, nx * ny, nz);
    for (int q = tid; q < N; q += kBotThreads) {
        const int t = q / nx, i = q - t * nx, k = DIM == 3 ? t / ny : 0, j = t - k * ny;
        u[q] /= 1.0 - (sn.c0 + sn.mu[0][i] + sn.mu[1][j] + (DIM == 3 ? sn.mu[2][k] : 0.0));
    }
    __syncthreads();
    axis(0, 1, nx);
    axis(1, nx, ny);
    if (DIM == 3) axis(2, nx * ny, nz);
    for (int q = tid; q < N; q += kBotThreads) x[q] = (T)u[q];
}

template <typename T, int DIM, int ORDER>
__global__ void __launch_bounds__(kBotThreads) k_mg_bottom(const MgBottom<T> m) {
    extern __shared__ __align__(16) unsigned char smem_bot[];
    constexpr int NC = ORDER == 2 ? 2 : 3;
    const int tid = threadIdx.x, last = m.nlev - 1;
    // level l: x, tmp, b at off[l] (+ 0, N, 2 N); `odd` bit l: x and tmp are exchanged
    int off[kMgBottomLevels];
    unsigned odd = 0;
    T* base = reinterpret_cast<T*>(smem_bot);
    {
        int o = 0;
        for (int l = 0; l < m.nlev; ++l) {
            off[l] = o;
            o += 3 * m.lv[l].n[0] * m.lv[l].n[1] * m.lv[l].n[2];
        }
        const int N = m.lv[0].n[0] * m.lv[0].n[1] * m.lv[0].n[2];
        for (int q = tid; q < N; q += kBotThreads) {
            base[q] = T(0);
            base[2 * N + q] = m.b[q];
        }
    }
    T* const cg_smem = base + m.cg_off;  // 8-byte aligned
    __syncthreads();
    auto pts = [&](int l) { return m.lv[l].n[0] * m.lv[l].n[1] * m.lv[l].n[2]; };
    auto X = [&](int l) { return base + off[l] + ((odd >> l) & 1u ? pts(l) : 0); };
    auto Y = [&](int l) { return base + off[l] + ((odd >> l) & 1u ? 0 : pts(l)); };
    auto smooth = [&](int l, int steps) {
        const MgBottomLevel<T>& L = m.lv[l];
        const int nx = L.n[0], ny = L.n[1], nz = L.n[2], N = nx * ny * nz;
        const T* b = base + off[l] + 2 * N;
        const Stencil<T> sa = L.sa;
        const T wd = L.wd;
        auto update = [&](const T* x, int q, int i, int j, int k) {
            const T u = x[q];
            return u + wd * ((b[q] - u) + bsum<T, DIM, ORDER>(x, sa, sa.c0 * u, q, i, j, k, nx, ny, nz));
        };
        for (int s = 0; s < steps; ++s) {
            T* x = X(l);
            if (m.colours) {
                const int wc = (nx + NC - 1) / NC;  // every lane a point of the colour
                for (int c = 0; c < NC; ++c) {
                    for (int p = tid; p < wc * ny * nz; p += kBotThreads) {
                        const int t = p / wc, k = DIM == 3 ? t / ny : 0, j = t - k * ny;
                        int o = (c - j - k) % NC;
                        if (o < 0) o += NC;
                        const int i = NC * (p - t * wc) + o;
                        if (i < nx) x[t * nx + i] = update(x, t * nx + i, i, j, k);
                    }
                    __syncthreads();
                }
            } else {
                T* y = Y(l);
                for (int q = tid; q < N; q += kBotThreads) {
                    const int t = q / nx, i = q - t * nx, k = DIM == 3 ? t / ny : 0, j = t - k * ny;
                    y[q] = update(x, q, i, j, k);
                }
                odd ^= 1u << l;
                __syncthreads();
            }
        }
    };
    for (int l = 0; l < last; ++l) {
        smooth(l, m.pre);
        const MgBottomLevel<T>& L = m.lv[l];
        const int nx = L.n[0], ny = L.n[1], nz = L.n[2], N = nx * ny * nz;
        const T* x = X(l);
        const T* b = base + off[l] + 2 * N;
        T* r = Y(l);  // free between the sweeps
        for (int q = tid; q < N; q += kBotThreads) {
            const int t = q / nx, i = q - t * nx, k = DIM == 3 ? t / ny : 0, j = t - k * ny;
            const T u = x[q];
            r[q] = (b[q] - u) + bsum<T, DIM, ORDER>(x, L.sa, L.sa.c0 * u, q, i, j, k, nx, ny, nz);
        }
        __syncthreads();
        const int cx = m.lv[l + 1].n[0], cy = m.lv[l + 1].n[1], Nc = pts(l + 1);
        T* xc = X(l + 1);
        T* bc = base + off[l + 1] + 2 * Nc;
        for (int q = tid; q < Nc; q += kBotThreads) {
            const int t = q / cx, I = q - t * cx, K = DIM == 3 ? t / cy : 0, J = t - K * cy;
            const T w[3] = {T(0.25), T(0.5), T(0.25)};
            T s = T(0);
#pragma unroll
            for (int oz = (DIM == 3 ? 0 : 1); oz <= (DIM == 3 ? 2 : 1); ++oz)
#pragma unroll
                for (int oy = 0; oy < 3; ++oy)
#pragma unroll
                    for (int ox = 0; ox < 3; ++ox)
                        s += w[ox] * w[oy] * (DIM == 3 ? w[oz] : T(1)) *
                             r[((DIM == 3 ? 2 * K + oz : 0) * ny + 2 * J + oy) * nx + 2 * I + ox];
            bc[q] = s;
            xc[q] = T(0);
        }
        __syncthreads();
    }
    {
        const MgBottomLevel<T>& L = m.lv[last];
        const T* b = base + off[last] + 2 * pts(last);
        if (m.sine.use)
            coarse_sine<T, DIM>(L.n[0], L.n[1], L.n[2], b, X(last), m.sine, reinterpret_cast<double*>(cg_smem));
        else
            coarse_cg<T, DIM, ORDER>(L.n[0], L.n[1], L.n[2], b, X(last), L.sa, m.cg_rtol, m.cg_maxit, cg_smem);
        __syncthreads();
    }
    for (int l = last - 1; l >= 0; --l) {
        const int nx = m.lv[l].n[0], ny = m.lv[l].n[1], N = pts(l);
        const int cx = m.lv[l + 1].n[0], cy = m.lv[l + 1].n[1], cz = m.lv[l + 1].n[2];
        const T* e = X(l + 1);
        T* x = X(l);
        for (int q = tid; q < N; q += kBotThreads) {
            const int t = q / nx, i = q - t * nx, k = DIM == 3 ? t / ny : 0, j = t - k * ny;
            const int I = (i & 1) ? i >> 1 : (i >> 1) - 1, J = (j & 1) ? j >> 1 : (j >> 1) - 1;
            const int K = DIM == 2 ? 0 : ((k & 1) ? k >> 1 : (k >> 1) - 1);
            const int nodd = (i & 1) + (j & 1) + (DIM == 3 ? (k & 1) : 1);
            const T w = nodd == 3 ? T(1) : nodd == 2 ? T(0.5) : nodd == 1 ? T(0.25) : T(0.125);
            T s = T(0);
#pragma unroll
            for (int c3 = 0; c3 < (DIM == 3 ? 2 : 1); ++c3)
#pragma unroll
                for (int c2 = 0; c2 < 2; ++c2)
#pragma unroll
                    for (int c1 = 0; c1 < 2; ++c1) {
                        const bool in = (c1 == 0 || !(i & 1)) && (c2 == 0 || !(j & 1)) && (c3 == 0 || !(k & 1)) &&
                                        I + c1 >= 0 && J + c2 >= 0 && K + c3 >= 0 && I + c1 < cx && J + c2 < cy &&
                                        K + c3 < cz;
                        if (in) s += w * e[((K + c3) * cy + J + c2) * cx + I + c1];
                    }
            x[q] += s;
        }
        __syncthreads();
        smooth(l, m.post);
    }
    const T* x = X(0);
    for (int q = tid; q < pts(0); q += kBotThreads) m.x[q] = x[q];
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T, int ORDER, bool GS, int NS, int TILE>
static ew_status smooth2d_tile(const GridGeom& g, const T* x, const T* b, T* xo, const Stencil<T>& sa, T wd, const T* ec,
                               const GridGeom* c, cudaStream_t st) {
    using S = Smooth2dShape<T, ORDER, GS, NS, TILE>;
    auto kern = k_mg_smooth2d<T, ORDER, GS, NS, TILE>;
    EW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM));
    const dim3 grid((unsigned)((g.n[0] + TILE - 1) / TILE), (unsigned)((g.n[1] + TILE - 1) / TILE));
    kern<<<grid, 256, S::SMEM, st>>>((int)g.n[0], (int)g.n[1], x, b, xo, sa, wd, ec, c ? (int)c->n[0] : 0,
                                     c ? (int)c->n[1] : 0);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}

template <typename T, int ORDER, bool GS, int NS>
static ew_status smooth2d_ns(const GridGeom& g, const T* x, const T* b, T* xo, const Stencil<T>& sa, T wd, const T* ec,
                             const GridGeom* c, cudaStream_t st) {
    // 16 x 16 tiles where 32 x 32 ones would leave SMs idle (64 x 64 tiles recompute fewer halo
    // points yet were no faster: 1023^2 25.9 against 25.3 ms a solve, 2047^2 63.8 against 57.7)
    if (((g.n[0] + 31) / 32) * ((g.n[1] + 31) / 32) >= 152)
        return smooth2d_tile<T, ORDER, GS, NS, 32>(g, x, b, xo, sa, wd, ec, c, st);
    return smooth2d_tile<T, ORDER, GS, NS, 16>(g, x, b, xo, sa, wd, ec, c, st);
}

// Two sweeps a launch but for the three colours of reach two (one sweep already has a
// halo of six) and the largest FP64 levels of order-4 Jacobi, whose halo points cost
// the FP64 units more than a launch (V(2,2), four cycles: 2047^2 5042 us with two, 4830
// with one; 1023^2 1847 and 1901)
template <typename T>
int mg_smooth2d_sweeps(const GridGeom& g, bool gs) {
    if (g.order == 4) return gs || (sizeof(T) == 8 && g.N > (int64_t)2 << 20) ? 1 : 2;
    return 2;
}
template int mg_smooth2d_sweeps<float>(const GridGeom&, bool);
template int mg_smooth2d_sweeps<double>(const GridGeom&, bool);

template <typename T>
ew_status mg_smooth2d(const GridGeom& g, const T* x, const T* b, T* xo, const Stencil<T>& sa, T wd, bool gs, int sweeps,
                      const T* ec, const GridGeom* c, cudaStream_t st) {
#define EW_S(O, GS, NS) smooth2d_ns<T, O, GS, NS>(g, x, b, xo, sa, wd, ec, c, st)
    if (g.order == 2) {
        if (gs) return sweeps == 2 ? EW_S(2, true, 2) : EW_S(2, true, 1);
        return sweeps == 2 ? EW_S(2, false, 2) : EW_S(2, false, 1);
    }
    if (gs) return EW_S(4, true, 1);
    return sweeps == 2 ? EW_S(4, false, 2) : EW_S(4, false, 1);
#undef EW_S
}
template ew_status mg_smooth2d<float>(const GridGeom&, const float*, const float*, float*, const Stencil<float>&, float,
                                      bool, int, const float*, const GridGeom*, cudaStream_t);
template ew_status mg_smooth2d<double>(const GridGeom&, const double*, const double*, double*, const Stencil<double>&,
                                       double, bool, int, const double*, const GridGeom*, cudaStream_t);

template <typename T>
ew_status mg_prolong2d(const GridGeom& f, const GridGeom& c, const T* ec, T* x, cudaStream_t st) {
    const dim3 grid((unsigned)((f.n[0] + 127) / 128), (unsigned)f.n[1]);
    k_mg_prolong2d<T><<<grid, 128, 0, st>>>((int)f.n[0], (int)f.n[1], (int)c.n[0], (int)c.n[1], ec, x);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}
template ew_status mg_prolong2d<float>(const GridGeom&, const GridGeom&, const float*, float*, cudaStream_t);
template ew_status mg_prolong2d<double>(const GridGeom&, const GridGeom&, const double*, double*, cudaStream_t);

template <typename T>
ew_status mg_resid_restrict2d(const GridGeom& f, const GridGeom& c, const T* x, const T* b, T* bc, T* xc,
                              const Stencil<T>& sa, cudaStream_t st) {
    const dim3 grid((unsigned)((c.n[0] + kRrX - 1) / kRrX), (unsigned)((c.n[1] + kRrY - 1) / kRrY));
    if (f.order == 2)
        k_mg_resid_restrict2d<T, 2><<<grid, 256, 0, st>>>((int)f.n[0], (int)f.n[1], (int)c.n[0], (int)c.n[1], x, b, bc,
                                                          xc, sa);
    else
        k_mg_resid_restrict2d<T, 4><<<grid, 256, 0, st>>>((int)f.n[0], (int)f.n[1], (int)c.n[0], (int)c.n[1], x, b, bc,
                                                          xc, sa);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}
template ew_status mg_resid_restrict2d<float>(const GridGeom&, const GridGeom&, const float*, const float*, float*,
                                              float*, const Stencil<float>&, cudaStream_t);
template ew_status mg_resid_restrict2d<double>(const GridGeom&, const GridGeom&, const double*, const double*, double*,
                                               double*, const Stencil<double>&, cudaStream_t);

template <typename T>
ew_status mg_resid_norm2d(const GridGeom& g, const T* x, const T* b, const Stencil<T>& sa, double* part, int nblocks,
                          cudaStream_t st) {
    if (g.order == 2)
        k_mg_resid_norm2d<T, 2><<<nblocks, 256, 0, st>>>((int)g.n[0], (int)g.n[1], x, b, sa, part);
    else
        k_mg_resid_norm2d<T, 4><<<nblocks, 256, 0, st>>>((int)g.n[0], (int)g.n[1], x, b, sa, part);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}
template ew_status mg_resid_norm2d<float>(const GridGeom&, const float*, const float*, const Stencil<float>&, double*,
                                          int, cudaStream_t);
template ew_status mg_resid_norm2d<double>(const GridGeom&, const double*, const double*, const Stencil<double>&,
                                           double*, int, cudaStream_t);

template <typename T>
size_t mg_bottom_smem(const int64_t* n, int nlev) {
    size_t s = 0;
    for (int l = 0; l < nlev; ++l) s += 3 * (size_t)n[l] * sizeof(T);
    return s + 8 + std::max(coarse_cg_smem<T>(n[nlev - 1]), 2 * sizeof(double) * (size_t)n[nlev - 1]);
}
template size_t mg_bottom_smem<float>(const int64_t*, int);
template size_t mg_bottom_smem<double>(const int64_t*, int);

template <typename T, int DIM, int ORDER>
static ew_status bottom(MgBottom<T> m, cudaStream_t st) {
    auto kern = k_mg_bottom<T, DIM, ORDER>;
    int64_t n[kMgBottomLevels];
    m.cg_off = 0;
    for (int l = 0; l < m.nlev; ++l) {
        n[l] = (int64_t)m.lv[l].n[0] * m.lv[l].n[1] * m.lv[l].n[2];
        m.cg_off += 3 * (int)n[l];
    }
    m.cg_off = (m.cg_off + 1) & ~1;
    // the coarsest level's sine transforms
    const MgBottomLevel<T>& lc = m.lv[m.nlev - 1];
    m.sine.use = 1;
    for (int d = 0; d < DIM; ++d)
        if (lc.n[d] > kMgSineMax) m.sine.use = 0;
    if (m.sine.use) {
        m.sine.c0 = (double)lc.sa.c0;
        for (int d = 0; d < DIM; ++d) {
            const int k1 = lc.n[d] + 1;
            for (int k = 1; k < k1; ++k) {
                const double th = M_PI * k / k1;
                m.sine.mu[d][k - 1] = 2.0 * (double)lc.sa.c1[d] * cos(th) + 2.0 * (double)lc.sa.c2[d] * cos(2.0 * th);
                for (int j = 1; j < k1; ++j)
                    m.sine.s[d][(k - 1) * (k1 - 1) + j - 1] = sqrt(2.0 / k1) * sin(th * j);
            }
        }
    }
    const size_t smem = mg_bottom_smem<T>(n, m.nlev);
    EW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<1, kBotThreads, smem, st>>>(m);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}

template <typename T>
ew_status mg_bottom(int dim, int order, const MgBottom<T>& m, cudaStream_t st) {
    if (dim == 2) return order == 2 ? bottom<T, 2, 2>(m, st) : bottom<T, 2, 4>(m, st);
    return order == 2 ? bottom<T, 3, 2>(m, st) : bottom<T, 3, 4>(m, st);
}
template ew_status mg_bottom<float>(int, int, const MgBottom<float>&, cudaStream_t);
template ew_status mg_bottom<double>(int, int, const MgBottom<double>&, cudaStream_t);

}  // namespace ew
