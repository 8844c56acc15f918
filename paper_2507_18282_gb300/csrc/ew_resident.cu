// ew_resident.cu -- the whole explicit wave-solve of a small 2D grid on chip:
// the grid and its ghost layers stay in shared memory (of one CTA, or of a
// cluster of CTAs that exchange their edge rows through distributed shared
// memory), D^n and the filter sums beside them, for all N_t steps of one
// launch (eqs. explicitStep1, explicitScheme, filterQuadrature; the summed
// form of ew_stencil.cu).
#include <cooperative_groups.h>
#include <stdio.h>
#include <stdlib.h>

#include <algorithm>
#include <type_traits>

#include "ew_bc_dev.cuh"
#include "ew_dd.cuh"
#include "ew_internal.h"

namespace ew {

// ---------------------------------------------------------------------------
// whole wave-solve of a small 2D grid in one CTA
// ---------------------------------------------------------------------------
// boundary and ghost layers of a whole padded 2D grid (pitch PX, G = 2
// layers on every side) from the box closure: Dirichlet walls 0, beyond them
// the odd reflection, Neumann ghosts the even reflection.  The cross-shaped
// stencils never read the corner blocks.
template <typename T, int R>
__device__ __forceinline__ void resident_fix(T* buf, int nx, int ny, int PX, int bc, int tid, int nthr) {
    constexpr int G = 2;
    if (R != 2 && bc == 0) return;  // order 2 with Dirichlet walls reads only the zero wall layer
    const int bx = axis_bc(bc, 0), by = axis_bc(bc, 1);
    for (int q = tid; q < 2 * G * (ny + nx); q += nthr) {
        const int layer = q % G + 1, side = (q / G) & 1, r = q / (2 * G);
        int sg = 1;
        if (r < ny) {  // x-ghost of row r
            const int gx = side ? nx - 1 + layer : -layer;
            const int ix = ext_axis<int>(gx, nx, bx, sg);
            const T v = ix < 0 ? T(0) : buf[(r + G) * PX + ix + G];
            buf[(r + G) * PX + gx + G] = sg < 0 ? -v : v;
        } else {  // y-ghost of column x
            const int x = r - ny;
            const int gy = side ? ny - 1 + layer : -layer;
            const int iy = ext_axis<int>(gy, ny, by, sg);
            const T v = iy < 0 ? T(0) : buf[(iy + G) * PX + x + G];
            buf[(gy + G) * PX + x + G] = sg < 0 ? -v : v;
        }
    }
}

template <typename T, int R>
__global__ void __launch_bounds__(1024)
    k_resident2d(int nx, int ny, const T* __restrict__ vin, T* __restrict__ vout,
                 const T* __restrict__ cw, int64_t Nt, Stencil<T> st, Stencil<T> st_half) {
    constexpr int G = 2;
    const int PX = nx + 2 * G, PY = ny + 2 * G;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* sA = reinterpret_cast<T*>(smem_raw);
    T* sB = sA + PX * PY;
    T* sAcc = sB + PX * PY;
    const int64_t N = (int64_t)nx * ny;
    vin += blockIdx.x * N;
    vout += blockIdx.x * N;
    const int nthr = blockDim.x;
    const int tid = threadIdx.x;

    auto fix = [&](T* buf) { resident_fix<T, R>(buf, nx, ny, PX, st.bc, tid, nthr); };
    auto lap = [&](const T* c, int p, const Stencil<T>& s) {
        T r = s.c0 * c[p] + s.c1[0] * (c[p - 1] + c[p + 1]) + s.c1[1] * (c[p - PX] + c[p + PX]);
        if (R == 2) r += s.c2[0] * (c[p - 2] + c[p + 2]) + s.c2[1] * (c[p - 2 * PX] + c[p + 2 * PX]);
        return r;
    };

    // sA: W^n with its boundary and ghost layers; sB: D^n (same layout)
    for (int q = tid; q < PX * PY; q += nthr) {
        sA[q] = T(0);
        sB[q] = T(0);
    }
    __syncthreads();
    for (int q = tid; q < N; q += nthr) {
        int x = q % nx, y = q / nx;
        sA[(y + G) * PX + x + G] = vin[q];
    }
    __syncthreads();
    fix(sA);
    __syncthreads();
    // first step (eq. explicitStep1): D^1 = (dt^2/2) L W^0, then W^1 = W^0 + D^1
    const T c0 = cw[0], c1 = cw[1];
    for (int q = tid; q < N; q += nthr) {
        int x = q % nx, y = q / nx;
        int p = (y + G) * PX + x + G;
        sB[p] = lap(sA, p, st_half);
    }
    __syncthreads();
    for (int q = tid; q < N; q += nthr) {
        int x = q % nx, y = q / nx;
        int p = (y + G) * PX + x + G;
        T x0 = sA[p];
        T w1 = x0 + sB[p];
        sA[p] = w1;
        sAcc[q] = c0 * x0 + c1 * w1;
    }
    __syncthreads();
    fix(sA);
    __syncthreads();
    for (int64_t n = 1; n < Nt; ++n) {
        const T cn = cw[n + 1];
        // D^{n+1} = D^n + dt^2 L W^n everywhere, then W^{n+1} = W^n + D^{n+1} pointwise
        for (int q = tid; q < N; q += nthr) {
            int x = q % nx, y = q / nx;
            int p = (y + G) * PX + x + G;
            sB[p] = sB[p] + lap(sA, p, st);
        }
        __syncthreads();
        for (int q = tid; q < N; q += nthr) {
            int x = q % nx, y = q / nx;
            int p = (y + G) * PX + x + G;
            T wn = sA[p] + sB[p];
            sA[p] = wn;
            sAcc[q] += cn * wn;
        }
        __syncthreads();
        fix(sA);
        __syncthreads();
    }
    for (int q = tid; q < N; q += nthr) vout[q] = sAcc[q];
}

// one operation each, rounded once (double-FP32 pairs: ew_dd.cuh)
__device__ __forceinline__ float r_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float r_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float r_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double r_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double r_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double r_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ dd r_add(dd a, dd b) { return dd_add(a, b); }
__device__ __forceinline__ dd r_mul(dd a, dd b) { return dd_mul(a, b); }
__device__ __forceinline__ dd r_fma(dd a, dd b, dd c) { return dd_fma(a, b, c); }

// The same on a cluster of CTAs: the rows of one vector's grid are split over
// the CTAs of a cluster (each on an SM of its own), W^n is double-buffered in
// their shared memory and D^n, W^n and the filter sums of a thread's points
// stay in its registers, so a step is one pass and one cluster barrier.  A
// thread that writes W^{n+1} of a point also writes the copies others need of
// it: into the halo rows of the CTA above or below (distributed shared
// memory), and into the ghost layers beyond the box's faces.
//
// The update of a point takes the operations of the blocked 2D kernels in
// their order (BLOCKED, grids that those kernels serve in other calls: the
// same bits either way) or those of k_resident2d (the grids of one CTA).
//
// Why: one CTA is bound by the units of one SM (FP64: two operations a clock;
// 63^2 took 11 us a step), and its step was three passes over shared memory
// with two integer divisions a point; the blocked kernels' tiles are about
// 120 x 60 points and more, so up to a few 10,000 points they leave most SMs
// idle and pay a launch for a few steps.  Measured, order 2, 400 steps, one
// vector: 63^2 FP64 4290 (one CTA) -> 490 us, 127^2 FP64 4935 (blocked) ->
// 1319 us, 181^2 in pairs 2939 -> 855 us, 255^2 FP32 order 4 1340 -> 597 us.
// Bound: below about 500 points a CTA the cluster barrier (0.5 us a step),
// above it the FP64 units or the shared-memory reads of the point loop.
template <typename T, int R, int PT, bool BLOCKED>
__global__ void __launch_bounds__(1024)
    k_resident2d_cluster(int nx, int ny, const T* __restrict__ vin, T* __restrict__ vout, const T* __restrict__ cw,
                         int64_t Nt, Stencil<T> st, Stencil<T> st_half) {
    constexpr int G = 2;
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
    const int base = ny / C, rem = ny % C;
    const int rows = base + (rank < rem), y0 = rank * base + min(rank, rem);
    const int PX = nx + 2 * G, plane = (base + (rem > 0) + 2 * G) * PX;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T* own = reinterpret_cast<T*>(smem_raw);  // W^n and W^{n+1}: local row ly at row ly + G
    T* prev = rank > 0 ? cluster.map_shared_rank(own, rank - 1) : own;
    T* next = rank + 1 < C ? cluster.map_shared_rank(own, rank + 1) : own;
    const int64_t N = (int64_t)nx * ny, v = blockIdx.x / C;
    const int nthr = blockDim.x, tid = threadIdx.x, npt = rows * nx;
    vin += v * N + (int64_t)y0 * nx;
    vout += v * N + (int64_t)y0 * nx;
    for (int q = tid; q < 2 * plane; q += nthr) own[q] = T(0);  // walls stay 0

    // a thread's points: index in a buffer, and where copies of it go (-1: nowhere)
    const int bx = axis_bc(st.bc, 0), by = axis_bc(st.bc, 1);
    const bool xl_odd = !(bx & 1), xh_odd = !(bx & 2), yl_odd = !(by & 1), yh_odd = !(by & 2);
    int p[PT], cxl[PT], cxh[PT], cyl[PT], cyh[PT];
#pragma unroll
    for (int k = 0; k < PT; ++k) {
        const int q = tid + k * nthr, ly = q / nx, x = q - ly * nx;
        p[k] = q < npt ? (ly + G) * PX + x + G : -1;
        cxl[k] = cxh[k] = cyl[k] = cyh[k] = -1;
        if (q >= npt) continue;
        // distance of the ghost a point feeds beyond each face: odd reflection about the wall
        // one step outside (only point 0, two steps out), even about the wall point itself
        const int dxl = xl_odd ? (R == 2 && x == 0 ? 2 : 0) : (x <= R ? x : 0);
        const int hx = nx - 1 - x, dxh = xh_odd ? (R == 2 && hx == 0 ? 2 : 0) : (hx <= R ? hx : 0);
        if (dxl) cxl[k] = (ly + G) * PX + G - dxl;
        if (dxh) cxh[k] = (ly + G) * PX + G + nx - 1 + dxh;
        const int hy = rows - 1 - ly;
        if (rank == 0) {
            const int d = yl_odd ? (R == 2 && ly == 0 ? 2 : 0) : (ly <= R ? ly : 0);
            if (d) cyl[k] = (G - d) * PX + x + G;
        } else if (ly < R) {
            cyl[k] = (base + (rank - 1 < rem) + G + ly) * PX + x + G;
        }
        if (rank == C - 1) {
            const int d = yh_odd ? (R == 2 && hy == 0 ? 2 : 0) : (hy <= R ? hy : 0);
            if (d) cyh[k] = (G + rows - 1 + d) * PX + x + G;
        } else if (hy < R) {
            cyh[k] = (G - 1 - hy) * PX + x + G;
        }
    }
    const bool yl_neg = rank == 0 && yl_odd, yh_neg = rank == C - 1 && yh_odd;
    auto put = [&](int off, int k, T w) {  // W of point k into buffer `off` and its copies
        own[off + p[k]] = w;
        if (cxl[k] >= 0) own[off + cxl[k]] = xl_odd ? -w : w;
        if (cxh[k] >= 0) own[off + cxh[k]] = xh_odd ? -w : w;
        if (cyl[k] >= 0) prev[off + cyl[k]] = yl_neg ? -w : w;
        if (cyh[k] >= 0) next[off + cyh[k]] = yh_neg ? -w : w;
    };
    auto sync = [&]() {
        if (C > 1)
            cluster.sync();
        else
            __syncthreads();
    };
    auto lap = [&](const T* c, int q, T u, const Stencil<T>& s) {
        if constexpr (BLOCKED) {
            T r = r_mul(s.c0, u);
            r = r_fma(s.c1[0], r_add(c[q - 1], c[q + 1]), r);
            r = r_fma(s.c1[1], r_add(c[q - PX], c[q + PX]), r);
            if (R == 2) {
                r = r_fma(s.c2[0], r_add(c[q - 2], c[q + 2]), r);
                r = r_fma(s.c2[1], r_add(c[q - 2 * PX], c[q + 2 * PX]), r);
            }
            return r;
        }
        T r = s.c0 * c[q] + s.c1[0] * (c[q - 1] + c[q + 1]) + s.c1[1] * (c[q - PX] + c[q + PX]);
        if (R == 2) r += s.c2[0] * (c[q - 2] + c[q + 2]) + s.c2[1] * (c[q - 2 * PX] + c[q + 2 * PX]);
        return r;
    };
    sync();
    T w[PT], d[PT], acc[PT];
#pragma unroll
    for (int k = 0; k < PT; ++k) {
        w[k] = d[k] = acc[k] = T(0);
        if (p[k] >= 0) {
            w[k] = vin[tid + k * nthr];
            put(0, k, w[k]);
        }
    }
    sync();
    const T c0 = cw[0], c1 = cw[1];
#pragma unroll
    for (int k = 0; k < PT; ++k)
        if (p[k] >= 0) {
            if constexpr (BLOCKED) {  // the sum of k_first_step2d
                T r = st_half.c0 * w[k];
                r += st_half.c1[0] * (own[p[k] - 1] + own[p[k] + 1]);
                r += st_half.c1[1] * (own[p[k] - PX] + own[p[k] + PX]);
                if (R == 2) {
                    r += st_half.c2[0] * (own[p[k] - 2] + own[p[k] + 2]);
                    r += st_half.c2[1] * (own[p[k] - 2 * PX] + own[p[k] + 2 * PX]);
                }
                d[k] = r;
            } else {
                d[k] = lap(own, p[k], w[k], st_half);
            }
            const T w1 = w[k] + d[k];
            acc[k] = c0 * w[k] + c1 * w1;
            w[k] = w1;
            put(plane, k, w1);
        }
    int cur = plane;
    T cn = Nt > 1 ? cw[2] : T(0);
    for (int64_t n = 1; n < Nt; ++n) {
        sync();
        const T cs = cn;
        if (n + 1 < Nt) cn = cw[n + 2];
        const int nxt = plane - cur;
#pragma unroll
        for (int k = 0; k < PT; ++k)
            if (p[k] >= 0) {
                T wn;
                if constexpr (BLOCKED) {
                    d[k] = r_add(d[k], lap(own + cur, p[k], w[k], st));
                    wn = r_add(w[k], d[k]);
                    acc[k] = r_fma(cs, wn, acc[k]);
                } else {
                    d[k] = d[k] + lap(own + cur, p[k], w[k], st);
                    wn = w[k] + d[k];
                    acc[k] += cs * wn;
                }
                w[k] = wn;
                put(nxt, k, wn);
            }
        cur = nxt;
    }
    sync();  // no CTA leaves while another may still write into its shared memory
#pragma unroll
    for (int k = 0; k < PT; ++k)
        if (p[k] >= 0) vout[tid + k * nthr] = acc[k];
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T>
static size_t resident_smem(const GridGeom& g) {
    return sizeof(T) * ((size_t)2 * (g.n[0] + 4) * (g.n[1] + 4) + (size_t)g.n[0] * g.n[1]);
}

// one CTA a vector: every grid of up to 16384 points whose three fields fit its shared memory
template <typename T>
static bool fits_cta(const GridGeom& g, int nvec) {
    return resident_smem<T>(g) <= 200 * 1024 && g.N <= 16384 && nvec <= 4 * 152;
}

constexpr int kResMaxPts = 4096;  // points a CTA of the cluster form (four a thread)

// CTAs a cluster for nvec vectors of this grid; 0: not the cluster form.
// Sixteen CTAs a vector are the fastest up to 16 vectors (63^2 and 127^2, all
// types: e.g. 127^2 in FP64, 16 vectors, 3.55 ms against 4.79 ms with 8); with
// more vectors the SMs fill anyway, so fewer CTAs a vector pay fewer barriers
// (63^2 in FP32, 64 vectors: 194 us with 2, 309 us with 4).  Small grids take
// one CTA where the barrier would cost more than it spreads: below about 2000
// points in FP32 (31^2, 200 steps: 76 us against 128 us with 4), 900 in pairs,
// 400 in FP64.
template <typename T>
static int cluster_ctas(const GridGeom& g, int nvec) {
    if (g.n[0] < 4 || g.n[1] < 4) return 0;  // ghosts mirror points of the edge CTAs only
    const int small = sizeof(T) == 4 ? 2048 : std::is_same<T, dd>::value ? 900 : 400;
    int C = nvec <= 16 ? 16 : nvec <= 36 ? 4 : nvec <= 76 ? 2 : 1;
    if (g.N < small) C = 1;
    while (C > 1 && g.n[1] < 3 * C) C /= 2;
    while (C < 16 && (g.n[1] + C - 1) / C * g.n[0] > kResMaxPts) C *= 2;
    if (g.n[1] < 3 * C || (g.n[1] + C - 1) / C * g.n[0] > kResMaxPts) return 0;
    // FP64 with one CTA a vector: the one-CTA form's passes are 8-20 % faster (31^2, 63^2, 256 vectors)
    if (std::is_same<T, double>::value && C == 1) return 0;
    return C;
}

// The cluster form also takes larger grids with few vectors, which the blocked
// kernels would run on a fraction of the SMs.  The line is where the next form
// takes the same time (400 steps): FP32 up to 181^2 points a vector (beyond, the
// tiles of ew_persist2d.cu: 255^2, order 4, 455 against 597 us here); pairs 16 x
// 255^2 (3838 against 5781 us blocked); FP64 4 x 255^2 (4830 against 4938 us
// blocked), and 16 x 127^2 (3554 against 8124 us).  FP64 at order 4 crosses at
// 61,000 points (40 steps: 200^2 468 against 684 us blocked, 62,664 points 703
// against 688, 256^2 709 against 688).
template <typename T>
static bool fits_cluster(const GridGeom& g, int nvec) {
    if (g.N > (sizeof(T) == 4 ? 32768 : 65536)) return false;
    if (std::is_same<T, double>::value && g.order == 4 && g.N > 60000) return false;
    if (std::is_same<T, dd>::value) return nvec <= 16;
    if (g.N * nvec > 262144 + 2048) return false;
    return sizeof(T) == 4 || g.N <= 16384 || nvec <= 4;
}

template <typename T, int R, bool BLOCKED>
static void* cluster_kernel(int PT) {
    if (PT == 1) return (void*)k_resident2d_cluster<T, R, 1, BLOCKED>;
    return PT == 2 ? (void*)k_resident2d_cluster<T, R, 2, BLOCKED> : (void*)k_resident2d_cluster<T, R, 4, BLOCKED>;
}

// the launch of the cluster form with C CTAs a vector
template <typename T>
static ResidentPlan cluster_plan(const GridGeom& g, bool blocked, int C) {
    ResidentPlan p;
    // points a thread: 512 threads beat 1024 once each has two points (a barrier of fewer warps;
    // 127^2 FP32 order 4, 16 CTAs, 8 vectors, 400 steps: 565 us with one point, 365 with two, 408 with four)
    p.pts = (int)((g.n[1] + C - 1) / C * g.n[0]);  // points of the fullest CTA
    p.PT = p.pts <= 512 ? 1 : p.pts <= 1024 ? 2 : 4;
    p.C = C;
    p.blocked = blocked;
    p.threads = ((p.pts + p.PT - 1) / p.PT + 31) / 32 * 32;
    p.smem = 2 * sizeof(T) * (size_t)((g.n[1] + C - 1) / C + 4) * (size_t)(g.n[0] + 4);
    if (g.order == 2)
        p.kern = blocked ? cluster_kernel<T, 1, true>(p.PT) : cluster_kernel<T, 1, false>(p.PT);
    else
        p.kern = blocked ? cluster_kernel<T, 2, true>(p.PT) : cluster_kernel<T, 2, false>(p.PT);
    return p;
}

static cudaLaunchConfig_t cluster_config(const ResidentPlan& p, int nvec, cudaLaunchAttribute* at, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(nvec * p.C));
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)p.C;
    at->val.clusterDim.y = at->val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cfg;
}

// Clusters of this plan that the device holds at a time.  16 CTAs are beyond the portable size, and where
// fewer SMs of a GPC are visible (a partitioned GPU) less than that may be too many: 0.  The query takes 0.2 us.
static int clusters_at_a_time(const ResidentPlan& p) {
    if (const char* e = getenv("EW_TEST_MAX_CLUSTER"))  // test hook: no larger clusters on this device
        if (p.C > atoi(e)) return 0;
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = cluster_config(p, 1, &at, nullptr);
    int n = 0;
    if (cudaFuncSetAttribute(p.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.smem) == cudaSuccess &&
        cudaFuncSetAttribute(p.kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, p.kern, &cfg) == cudaSuccess)
        return n;
    cudaGetLastError();
    return 0;
}

// Many vectors of a grid too large for one CTA of the cluster form: its clusters
// and the one-CTA form (152 vectors a wave) then differ by how full their last
// waves are.  One CTA takes 2.6 + 1.35e-4 N times as long for a vector as a CTA of
// four in FP32 (N = 8200: 262 against 282 us for 152 vectors of 55 x 149, order 2, 60
// steps; 1026 against 1144 us for 608 of 57 x 144, order 4), which loses where the
// waves come out no longer: (24 x 500, 176 vectors: 472 against 252 us); at order 4
// narrow grids (28 columns and fewer) and more than 9500 points stay with the
// clusters (18 x 508, 140 vectors: 306 against 258 us).  Pairs in clusters of two:
// only a second wave of a few CTAs loses (264 x 17, 77 vectors, order 2: 269 against
// 282 us).  FP64 is bound by the SMs' FP64 units, so two CTAs a vector gain only
// where one CTA leaves most of a second wave empty (75 x 74, order 4, 40 steps: 228
// vectors 1602 in clusters against 1803 us; 120 vectors of 47 x 88 839 against 699
// us; 304 of 407 x 12, order 2, 1234 against 1049 us).
template <typename T>
static bool one_cta_wins(const GridGeom& g, int nvec, int C) {
    if (nvec <= 76) return false;
    if (std::is_same<T, double>::value) return (nvec * C + 151) / 152 > (nvec + 151) / 152 * 1.6;
    if (std::is_same<T, dd>::value) return C == 2 && nvec * C > 152 && nvec * C <= 172;
    if (sizeof(T) != 4 || C != 4 || (g.order == 4 && (g.n[0] < 32 || g.N > 9500))) return false;
    return (nvec * C + 151) / 152 > (nvec + 151) / 152 * (2.6 + 1.35e-4 * (double)g.N);
}

// Pairs at order 4 where the clusters take several waves: a wave takes 1.4 + 0.8e-3
// pts us a step (pts: points a CTA), the blocked kernels 9.2 us up to about 720,000
// points of all vectors where their tiles fill (444 x 91, 40 steps: 14 vectors, two
// waves, 297 against 367 us; 15 vectors, three waves, 425 against 374 us; but 59 x
// 593, 16 vectors, 282 against 569 us)
static bool pairs_blocked_wins(const GridGeom& g, int nvec, const ResidentPlan& p, int at_a_time) {
    const int waves = (nvec + at_a_time - 1) / at_a_time;
    return g.order == 4 && waves > 1 && g.N * nvec <= 720000 && p.pts >= 2550 && g.n[0] >= 100 &&
           waves * (1.4 + 0.8e-3 * p.pts) > 9.2;
}

template <typename T>
ResidentPlan resident_plan(const GridGeom& g, int nvec) {
    if (g.dim != 2 || g.map) return ResidentPlan();
    const bool cta = fits_cta<T>(g, nvec);
    if (cta || fits_cluster<T>(g, nvec))
        // smaller clusters where the wanted ones do not fit the device, as far as their CTAs' points allow
        for (int C = cluster_ctas<T>(g, nvec); C > 0; C /= 2) {
            const ResidentPlan p = cluster_plan<T>(g, !cta, C);
            if (p.pts > kResMaxPts || (std::is_same<T, double>::value && C == 1)) break;
            if (cta && one_cta_wins<T>(g, nvec, C)) break;
            const int n = clusters_at_a_time(p);
            if (n == 0) continue;
            if (!cta && std::is_same<T, dd>::value && pairs_blocked_wins(g, nvec, p, n)) break;
            return p;
        }
    ResidentPlan one;
    if (cta) one.C = 1, one.pts = (int)g.N;
    return one;
}
template ResidentPlan resident_plan<float>(const GridGeom&, int);
template ResidentPlan resident_plan<double>(const GridGeom&, int);
template ResidentPlan resident_plan<dd>(const GridGeom&, int);

// one-CTA form
template <typename T, int R>
static ew_status resident_cta(const GridGeom& g, const T* vin, T* vout, const T* cw, const FilterPlan& plan, int nvec,
                              const Stencil<T>& s, const Stencil<T>& sh, cudaStream_t st) {
    const size_t smem = resident_smem<T>(g);
    const int threads = (int)std::min<int64_t>(1024, ((g.N + 31) / 32) * 32);
    EW_CUDA_TRY(cudaFuncSetAttribute(k_resident2d<T, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_resident2d<T, R><<<nvec, threads, smem, st>>>((int)g.n[0], (int)g.n[1], vin, vout, cw, plan.Nt, s, sh);
    EW_CUDA_TRY(cudaGetLastError());
    return EW_OK;
}

template <typename T>
OnChipForm resident_form(const GridGeom& g, const ResidentPlan& p) {
    char buf[96];
    snprintf(buf, sizeof buf, "k_resident2d_cluster<%s, %d, %d, %s>",
             sizeof(T) == 4 ? "float" : std::is_same<T, dd>::value ? "dd" : "double", g.order == 2 ? 1 : 2, p.PT,
             p.blocked ? "true" : "false");
    return OnChipForm{buf, 1, (int)g.n[0], (int)((g.n[1] + p.C - 1) / p.C)};
}
template OnChipForm resident_form<float>(const GridGeom&, const ResidentPlan&);
template OnChipForm resident_form<double>(const GridGeom&, const ResidentPlan&);
template OnChipForm resident_form<dd>(const GridGeom&, const ResidentPlan&);

template <typename T>
ew_status resident_wave_solve(const GridGeom& g, const ResidentPlan& p, const T* vin, T* vout, const T* cw,
                              const FilterPlan& plan, int nvec, cudaStream_t st) {
    Stencil<T> s = make_stencil<T>(g, plan.dt * plan.dt);
    Stencil<T> sh = make_stencil<T>(g, 0.5 * plan.dt * plan.dt);
    cudaEvent_t ev = fused_begin(st);
    if (p.kern) {
        int nx = (int)g.n[0], ny = (int)g.n[1];
        int64_t Nt = plan.Nt;
        void* args[] = {(void*)&nx, (void*)&ny, (void*)&vin, (void*)&vout, (void*)&cw, (void*)&Nt, (void*)&s, (void*)&sh};
        cudaLaunchAttribute at;
        const cudaLaunchConfig_t cfg = cluster_config(p, nvec, &at, st);
        EW_CUDA_TRY(cudaLaunchKernelExC(&cfg, p.kern, args));
    } else if (g.order == 2) {
        EW_TRY((resident_cta<T, 1>(g, vin, vout, cw, plan, nvec, s, sh, st)));
    } else {
        EW_TRY((resident_cta<T, 2>(g, vin, vout, cw, plan, nvec, s, sh, st)));
    }
    fused_end(ev, st, g.N * nvec, g.N * nvec * plan.Nt);
    return EW_OK;
}
template ew_status resident_wave_solve<float>(const GridGeom&, const ResidentPlan&, const float*, float*, const float*,
                                              const FilterPlan&, int, cudaStream_t);
template ew_status resident_wave_solve<double>(const GridGeom&, const ResidentPlan&, const double*, double*,
                                               const double*, const FilterPlan&, int, cudaStream_t);
template ew_status resident_wave_solve<dd>(const GridGeom&, const ResidentPlan&, const dd*, dd*, const dd*,
                                           const FilterPlan&, int, cudaStream_t);

}  // namespace ew
