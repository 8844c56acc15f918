// ew_mg.cuh -- shared by the multigrid cycle (ew_mg.cu) and its fused pieces
// (ew_mg_fused.cu): the coarsest-level solver and the launchers' declarations.
#pragma once

#include "ew_internal.h"
#include "ew_stencil_dev.cuh"

namespace ew {

constexpr int kCoarseMax = 2048;  // points of the coarsest level
constexpr int kMgBottomLevels = 12;

// the cycle's levels from `lv[0]` to the coarsest, for the one-launch bottom
template <typename T>
struct MgBottomLevel {
    int n[3];
    Stencil<T> sa;  // a L_h
    T wd;           // x += wd (b - M x)
};
// sine transforms of the coarsest level: S_a[k][j] = sqrt(2 / (n + 1)) sin(pi (k + 1) (j + 1) / (n + 1)), the
// stencil's eigenvalue c0 + sum mu_a[k_a]
constexpr int kMgSineMax = 6;  // points per axis
struct MgSine {
    int use;
    double c0;
    double s[3][kMgSineMax * kMgSineMax];
    double mu[3][kMgSineMax];
};
template <typename T>
struct MgBottom {
    int nlev, pre, post;
    int colours;  // 0: damped Jacobi
    T cg_rtol;
    int cg_maxit;
    int cg_off;     // set by mg_bottom
    const T* b;     // right-hand side of lv[0]
    T* x;           // its result, from x = 0
    MgSine sine;    // set by mg_bottom
    MgBottomLevel<T> lv[kMgBottomLevels];
};
template <typename T>
ew_status mg_bottom(int dim, int order, const MgBottom<T>& m, cudaStream_t st);
// shared memory of the bottom launch from a level of n[0] points down to n[nlev - 1]
template <typename T>
size_t mg_bottom_smem(const int64_t* n, int nlev);
// sweeps one launch of mg_smooth2d can take (and must be given at most)
template <typename T>
int mg_smooth2d_sweeps(const GridGeom& g, bool gs);
// xo = `sweeps` smoothing sweeps from x (+ P ec, when ec is given, ec on grid c)
template <typename T>
ew_status mg_smooth2d(const GridGeom& g, const T* x, const T* b, T* xo, const Stencil<T>& sa, T wd, bool gs, int sweeps,
                      const T* ec, const GridGeom* c, cudaStream_t st);
template <typename T>
ew_status mg_resid_restrict2d(const GridGeom& f, const GridGeom& c, const T* x, const T* b, T* bc, T* xc,
                              const Stencil<T>& sa, cudaStream_t st);

// 3D FP32 levels (ew_mg_plane.cu).  mode 0: out = b - M x; 1: out = x + wd (b - M x); 2: one colour of the same in place
bool mg_plane3d_f2_fits(const GridGeom& g);
ew_status mg_plane3d_f2(int mode, const GridGeom& g, const float* x, const float* b, float* out,
                        const Stencil<float>& sa, float wd, int colour, int nsm, cudaStream_t st);
// part[0 .. nblocks): shares of |b - M x|^2
template <typename T>
ew_status mg_resid_norm2d(const GridGeom& g, const T* x, const T* b, const Stencil<T>& sa, double* part, int nblocks,
                          cudaStream_t st);
// x += P ec
template <typename T>
ew_status mg_prolong2d(const GridGeom& f, const GridGeom& c, const T* ec, T* x, cudaStream_t st);

// ---------------------------------------------------------------------------
// coarsest level: conjugate gradients in one CTA, all vectors in shared memory
// ---------------------------------------------------------------------------
template <typename T>
size_t coarse_cg_smem(int64_t N) {
    return sizeof(T) * (4 * (size_t)N + 32);
}

// Inner product over the CTA, or over its first warp when only that works
// (small systems): the points of each group of 32 are summed by shuffles and the groups
// added in their order, so both give the same bits.
template <typename T, bool WARP>
__device__ T coarse_dot(const T* a, const T* b, int N, T* red) {
    T t = T(0);
    if (WARP) {
        for (int g = 0; g < N; g += 32) {
            const int q = g + (int)threadIdx.x;
            T s = T(0);
            if (q < N) s += a[q] * b[q];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            t += s;
        }
        return t;
    }
    T s = T(0);
    for (int q = threadIdx.x; q < N; q += blockDim.x) s += a[q] * b[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    __syncthreads();
    return t;
}

template <typename T, int DIM, int ORDER, bool WARP>
__device__ void coarse_cg_run(int nx, int ny, int nz, const T* b, T* x, const Stencil<T>& sa, T rtol, int maxit,
                              T* smem) {
    const int N = nx * ny * nz, nt = WARP ? 32 : blockDim.x;
    T* sx = smem;
    T* sr = sx + N;
    T* sp = sr + N;
    T* sq = sp + N;
    T* red = sq + N;
    auto sync = [&]() {
        if (WARP)
            __syncwarp();
        else
            __syncthreads();
    };
    for (int q = threadIdx.x; q < N; q += nt) {
        const T v = b[q];
        sx[q] = T(0);
        sr[q] = v;
        sp[q] = v;
    }
    sync();
    T rr = coarse_dot<T, WARP>(sr, sr, N, red);
    const T stop = rtol * rtol * rr;
    for (int it = 0; it < maxit && rr > stop && rr > T(0); ++it) {
        for (int q = threadIdx.x; q < N; q += nt) {
            const int t = q / nx, i = q - t * nx, k = t / ny, j = t - k * ny;
            sq[q] = sp[q] - lap_global<T, DIM, ORDER>(sp, sa, q, i, j, k, nx, ny, nz);  // M p
        }
        sync();
        const T pq = coarse_dot<T, WARP>(sp, sq, N, red);
        if (!(pq > T(0))) break;
        const T alpha = rr / pq;
        for (int q = threadIdx.x; q < N; q += nt) {
            sx[q] += alpha * sp[q];
            sr[q] -= alpha * sq[q];
        }
        sync();
        const T rr2 = coarse_dot<T, WARP>(sr, sr, N, red);
        const T beta = rr2 / rr;
        rr = rr2;
        for (int q = threadIdx.x; q < N; q += nt) sp[q] = sr[q] + beta * sp[q];
        sync();
    }
    for (int q = threadIdx.x; q < N; q += nt) x[q] = sx[q];
}

// M x = b on the coarsest level, by the calling CTA.  Up to
// 128 points one warp works alone: its barriers and inner products cost a
// fraction of the CTA's (9 points, FP64: 50 us with 512 threads)
template <typename T, int DIM, int ORDER>
__device__ void coarse_cg(int nx, int ny, int nz, const T* b, T* x, const Stencil<T>& sa, T rtol, int maxit, T* smem) {
    if (nx * ny * nz <= 128) {
        if (threadIdx.x < 32) coarse_cg_run<T, DIM, ORDER, true>(nx, ny, nz, b, x, sa, rtol, maxit, smem);
    } else {
        coarse_cg_run<T, DIM, ORDER, false>(nx, ny, nz, b, x, sa, rtol, maxit, smem);
    }
}

}  // namespace ew
