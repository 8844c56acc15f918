// ew_mg.cu -- geometric multigrid for the implicit time-step systems and the
// implicit wave-solve (eqs. implicitScheme, impMatrix, implicitStep1).
//
//   M x = b,   M = I - a L_h,   a = dt^2 / 2
//
// One V(pre, post) cycle (the paper solves these systems with its multigrid
// solver and names red-black / line smoothers; this is the plain geometric
// cycle for Cartesian boxes):
//   levels      n_c = (n - 1) / 2 per axis while every axis has odd n >= 5
//               (coarse point I on fine point 2I + 1, h_c = 2 h)
//   smoother    damped Jacobi x <- x + w (b - M x) / D with the constant
//               interior diagonal D = 1 + a sum_i d0 / h_i^2 (d0 = 2 or 5/2),
//               or multi-colour Gauss-Seidel with the same diagonal (two
//               colours at second order, three at fourth), or the learned
//               correction x <- x + N(b - M x) on the finest `learned_levels`
//               levels (ew_smoother.cu, applied as its composed stencil in
//               FP32, ew_smoother_comp.cu)
//   restriction full weighting, tensor product of (1/4, 1/2, 1/4)
//   prolongation (multi)linear interpolation, zero on the boundary
//   coarsest    by sine transforms up to six points per axis, else conjugate
//               gradients (M is SPD), in one CTA
//
// Implicit wave-solve (one application of S):
//   M W^1 = W^0;  M y = 2 W^n, W^{n+1} = y - W^{n-1};  V_out = sum c_n W^n
// Each system gets `max_cycles` V-cycles (or stops at `rtol`) from the
// initial guess y = 2 W^n (W^1 = W^0 for the first step) or, with
// guess = 1, from the previous system's solution.
// Kernels: 3D levels run their stencil operations 2.5D blocked
// (k_mg_plane3d), 2D levels several sweeps a launch on tiles, and the smallest
// levels together in one launch (ew_mg_fused.cu).  1023^2 order 2 in FP64,
// red-black, 87 cycles of a wave-solve: 58.9 -> 28.6 ms (8044 launches -> 1606).
#include <math.h>
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "ew_internal.h"
#include "ew_mg.cuh"
#include "ew_stencil_dev.cuh"

namespace ew {

// learned correction x += N(r) (ew_smoother.cu)
template <typename T>
ew_status smoother_apply(const GridGeom& g, const float* weights, const T* r, T* x, cudaStream_t st);

struct MGLevel {
    GridGeom geom;
};

int mg_levels(const GridGeom& g, GridGeom* lv, int maxlev) {
    int L = 0;
    lv[0] = g;
    for (;;) {
        bool ok = L + 1 < maxlev;
        for (int a = 0; a < g.dim; ++a)
            if (lv[L].n[a] < 5 || (lv[L].n[a] % 2) == 0) ok = false;
        if (!ok) break;
        GridGeom c = lv[L];
        c.N = 1;
        for (int a = 0; a < 3; ++a) {
            if (a < g.dim) {
                c.n[a] = (lv[L].n[a] - 1) / 2;
                c.h[a] = 2.0 * lv[L].h[a];
            }
            c.N *= c.n[a];
        }
        lv[++L] = c;
    }
    return L + 1;
}

static int grid_blocks(int64_t N, int threads) {
    int64_t b = (N + threads - 1) / threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, 152 * 16));
}

// one thread per point: x from the block's threads, y and z from the grid (no
// integer division in the kernels)
static int pt_threads(int64_t nx) { return nx >= 128 ? 128 : (int)(((nx + 31) / 32) * 32); }
static dim3 pt_grid(int64_t nx, int64_t ny, int64_t nz) {
    const int t = pt_threads(nx);
    return dim3((unsigned)((nx + t - 1) / t), (unsigned)ny, (unsigned)nz);
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------
// multi-colour Gauss-Seidel, in place: the points of one colour take
// x += (b - M x) * inv_d, M_ii = 1 / inv_d.  Second order: red-black, colour
// (i + j + k) & 1.  Fourth order (offsets of 1 and 2 along one axis): three
// colours, (i + j + k) mod 3; an offset changes the colour by +-1 or +-2, never
// 0 mod 3.  So no point of a colour reads another point of its colour, the
// colour's updates are independent, and the sweep is exact Gauss-Seidel in
// colour order
template <int ORDER>
__device__ __forceinline__ int mg_colour(int64_t i, int64_t j, int64_t k) {
    return ORDER == 2 ? (int)((i + j + k) & 1) : (int)((i + j + k) % 3);
}

// ---------------------------------------------------------------------------
// 3D stencil operations of the cycle, 2.5D blocked: a CTA owns 64 x 8 columns
// and a chunk of planes and streams along z through a ring of kPlS staged
// planes (each with a halo of R = ORDER / 2 in x and y).  The planes are
// filled by asynchronous copies kPlD planes ahead of the one the stencil needs
// next, so the loads of several planes are in flight while a plane is
// computed, and every value of x is read from memory about once.  b goes
// through a ring of its own (no halo).  Dirichlet box closure (the multigrid
// levels have no Neumann faces): a wall point is 0, a point beyond it the
// negated mirror; each staged cell is either 0 or a copy of one point of the
// box, negated by the thread that copied it once the copy has landed.
// MODE 0: out = r = b - M x; MODE 1: out = x + wd (b - M x) (Jacobi); MODE 2:
// the colour sweep in place (out == x), x += wd (b - M x) at the points of
// colour `colour` (mg_colour).  The Laplacian sums its terms in the order of
// lap_global.
constexpr int kPlBX = 64, kPlBY = 8, kPlNT = 256, kPlD = 2;

// index of coordinate i on an axis of n points under the odd closure
// (|i - clamp| <= 2): -1 for a wall point, else the mirror with sg negated
__device__ __forceinline__ int mg_ext(int i, int n, int& sg) {
    if (i >= 0 && i < n) return i;
    if (i == -1 || i == n) return -1;
    sg = -sg;
    return i < 0 ? -2 - i : 2 * n - i;
}

template <typename T>
__device__ __forceinline__ void mg_cp_async(T* dst, const T* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if (sizeof(T) == 8)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void mg_cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void mg_cp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

template <typename T, int ORDER>
struct PlaneRing {
    static constexpr int R = ORDER == 2 ? 1 : 2;
    static constexpr int SX = kPlBX + 2 * R, SY = kPlBY + 2 * R, CELLS = SX * SY;
    static constexpr int S = 2 * R + 1 + kPlD;                 // planes z - R .. z + R + kPlD
    static constexpr int PER = (CELLS + kPlNT - 1) / kPlNT;    // staged cells per thread and plane
    static constexpr int BPER = kPlBX * kPlBY / kPlNT;         // b cells per thread and plane
    static constexpr size_t SMEM = sizeof(T) * (size_t)S * (CELLS + kPlBX * kPlBY);
    static_assert(PER * S <= 32, "negation flags of the ring fit one word");
};

template <typename T, int ORDER, int MODE>
__global__ void __launch_bounds__(kPlNT)
    k_mg_plane3d(int nx, int ny, int nz, int zc, const T* x, const T* __restrict__ b, T* out, Stencil<T> sa, T wd,
                 int colour) {
    using PR = PlaneRing<T, ORDER>;
    constexpr int R = PR::R, SX = PR::SX, CELLS = PR::CELLS, S = PR::S, PER = PR::PER, BPER = PR::BPER;
    extern __shared__ __align__(16) unsigned char mg_smem[];
    T* ring = reinterpret_cast<T*>(mg_smem);  // [S][CELLS]
    T* bring = ring + (size_t)S * CELLS;      // [S][kPlBX * kPlBY]
    const int tid = threadIdx.x;
    const int x0 = blockIdx.x * kPlBX, y0 = blockIdx.y * kPlBY;
    const int z0 = blockIdx.z * zc, z1 = min(nz, z0 + zc);
    const int64_t plane = (int64_t)nx * ny;
    unsigned neg = 0;  // bit (slot * PER + u): this thread's cell u of ring slot `slot` awaits negation
    // the thread's staged cells, the same in every plane: offset of the source
    // column in a plane (-1: 0 for every plane), and which are negated mirrors
    int coff[PER];
    unsigned cneg = 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int c = tid + kPlNT * u;
        const int sy = c / SX, sx = c - sy * SX;
        const int hx = x0 - R + sx, hy = y0 - R + sy;
        int sg = 1;
        const int ex = hx < nx + R ? mg_ext(hx, nx, sg) : -1;  // past a ragged tile's reach: never read
        const int ey = hy < ny + R ? mg_ext(hy, ny, sg) : -1;
        coff[u] = (c < CELLS && ex >= 0 && ey >= 0) ? ey * nx + ex : -1;
        if (sg < 0) cneg |= 1u << u;
    }
    int boff[BPER];
#pragma unroll
    for (int u = 0; u < BPER; ++u) {
        const int c = tid + kPlNT * u;
        const int cy = c / kPlBX, cx = c - cy * kPlBX;
        boff[u] = (x0 + cx < nx && y0 + cy < ny) ? (y0 + cy) * nx + x0 + cx : -1;
    }
    // stage plane p (any integer in [z0 - R, z1 + R)) into its slot, and b of plane p (when inside [z0, z1))
    auto issue = [&](int p) {
        if (p >= z1 + R) {  // past the chunk's last stencil plane: an empty group keeps the count
            mg_cp_commit();
            return;
        }
        const int slot = ((p % S) + S) % S;
        T* dst = ring + (size_t)slot * CELLS;
        int sgz = 1;
        const int ez = mg_ext(p, nz, sgz);
        const T* xp = x + (int64_t)(ez < 0 ? 0 : ez) * plane;
        const unsigned flip = sgz < 0 ? (1u << PER) - 1 : 0u;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int c = tid + kPlNT * u;
            if (c >= CELLS) break;
            if (ez < 0 || coff[u] < 0) {
                dst[c] = T(0);
            } else {
                mg_cp_async(dst + c, xp + coff[u]);
                if (((cneg ^ flip) >> u) & 1u) neg |= 1u << (slot * PER + u);
            }
        }
        if (p >= z0 && p < z1) {
            T* bd = bring + (size_t)slot * (kPlBX * kPlBY);
            const T* bp = b + (int64_t)p * plane;
#pragma unroll
            for (int u = 0; u < BPER; ++u)
                if (boff[u] >= 0) mg_cp_async(bd + tid + kPlNT * u, bp + boff[u]);
        }
        mg_cp_commit();
    };
    auto negate = [&](int p) {  // after its copies landed: this thread's negated cells of plane p
        const int slot = ((p % S) + S) % S;
        T* dst = ring + (size_t)slot * CELLS;
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const unsigned bit = 1u << (slot * PER + u);
            if (neg & bit) {
                dst[tid + kPlNT * u] = -dst[tid + kPlNT * u];
                neg &= ~bit;
            }
        }
    };
    // prologue: planes z0 - R .. z0 + R + kPlD - 1, one group each
    for (int p = z0 - R; p < z0 + R + kPlD; ++p) issue(p);
    const T c1x = sa.c1[0], c1y = sa.c1[1], c1z = sa.c1[2], c2x = sa.c2[0], c2y = sa.c2[1], c2z = sa.c2[2];
    const int tx = tid % kPlBX, ty0 = tid / kPlBX;  // rows ty0 and ty0 + 4
    for (int z = z0; z < z1; ++z) {
        // plane z + R's group and every older one have landed (kPlD - 1 younger groups may be in flight)
        mg_cp_wait<kPlD - 1>();
        if (z == z0)
            for (int p = z0 - R; p <= z0 + R; ++p) negate(p);
        else
            negate(z + R);
        __syncthreads();  // plane z + R visible to all; every read of iteration z - 1 done
        issue(z + R + kPlD);  // into the slot of plane z - R - 1, last read in iteration z - 1
        const T* pc = ring + (size_t)(z % S) * CELLS;
        const T* bz = bring + (size_t)(z % S) * (kPlBX * kPlBY);
#pragma unroll
        for (int rr = 0; rr < kPlBY / 4; ++rr) {
            const int ty = ty0 + 4 * rr;
            const int gx = x0 + tx, gy = y0 + ty;
            if (gx >= nx || gy >= ny) continue;
            const int cc = (ty + R) * SX + tx + R;
            const T xc = pc[cc];
            T lap = sa.c0 * xc;
            lap += c1x * (pc[cc - 1] + pc[cc + 1]);
            lap += c1y * (pc[cc - SX] + pc[cc + SX]);
            lap += c1z * (ring[(size_t)((z - 1 + S) % S) * CELLS + cc] + ring[(size_t)((z + 1) % S) * CELLS + cc]);
            if (ORDER == 4) {
                lap += c2x * (pc[cc - 2] + pc[cc + 2]);
                lap += c2y * (pc[cc - 2 * SX] + pc[cc + 2 * SX]);
                lap += c2z * (ring[(size_t)((z - 2 + S) % S) * CELLS + cc] + ring[(size_t)((z + 2) % S) * CELLS + cc]);
            }
            const T r = (bz[ty * kPlBX + tx] - xc) + lap;
            const int64_t qi = (int64_t)z * plane + (int64_t)gy * nx + gx;
            if (MODE == 0) out[qi] = r;
            if (MODE == 1) out[qi] = xc + wd * r;
            if (MODE == 2 && mg_colour<ORDER>(gx, gy, z) == colour) out[qi] = xc + wd * r;
        }
    }
    mg_cp_wait<0>();  // no copy outlives the CTA
}

template <typename T>
__device__ __forceinline__ T get0(const T* __restrict__ v, int64_t i, int64_t j, int64_t k, int64_t nx, int64_t ny,
                                  int64_t nz) {
    if (i < 0 || j < 0 || k < 0 || i >= nx || j >= ny || k >= nz) return T(0);
    return v[(k * ny + j) * nx + i];
}

// full weighting: bc(I) = sum_o w(o) r(2I + 1 + o); x_c = 0
template <typename T>
__global__ void k_mg_restrict3d(int64_t fx, int64_t fy, int64_t fz, int64_t cx, int64_t cy, int64_t cz,
                              const T* __restrict__ r, T* __restrict__ bc, T* __restrict__ xc) {
    const T w[3] = {T(0.25), T(0.5), T(0.25)};
    {
        const int64_t I = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
        if (I >= cx) return;
        const int64_t J = blockIdx.y, K = blockIdx.z, q = (K * cy + J) * cx + I;
        int64_t fi = 2 * I + 1, fj = 2 * J + 1, fk = 2 * K + 1;
        T s = T(0);
        for (int oz = -1; oz <= 1; ++oz)
            for (int oy = -1; oy <= 1; ++oy)
                for (int ox = -1; ox <= 1; ++ox) {
                    T wt = w[ox + 1] * w[oy + 1] * w[oz + 1];
                    s += wt * get0(r, fi + ox, fj + oy, fk + oz, fx, fy, fz);
                }
        bc[q] = s;
        xc[q] = T(0);
    }
}

// x_f += P e_c (linear interpolation per axis).  A thread takes the 2 x 2 x 2
// fine points that share coarse corner (I, J, K): fine point 2 I + p along an
// axis lies, for p = 1, on coarse point I, and for p = 0 between I - 1 and I, so
// all eight come from the 2 x 2 x 2 coarse values around it.  Each point's terms
// and their order are those of the tensor product over its neighbours.
// One thread a fine point (up to eight loads and a weight product each) took
// 109 us on 255^3, this form 62 us; 21 us is the traffic's floor.
template <typename T>
__global__ void k_mg_prolong3d(int fx, int fy, int fz, int cx, int cy, int cz, const T* __restrict__ ec,
                               T* __restrict__ xf) {
    const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y, K = blockIdx.z;
    if (2 * I >= fx) return;
    T e[2][2][2];  // [k][j][i]: coarse points K - 1 + k, J - 1 + j, I - 1 + i, zero outside
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int a = I - 1 + i, b = J - 1 + j, c = K - 1 + k;
                e[k][j][i] = a >= 0 && b >= 0 && c >= 0 && a < cx && b < cy && c < cz
                                 ? ec[((int64_t)c * cy + b) * cx + a]
                                 : T(0);
            }
#pragma unroll
    for (int pk = 0; pk < 2; ++pk) {
        const int k = 2 * K + pk;
        if (k >= fz) break;
#pragma unroll
        for (int pj = 0; pj < 2; ++pj) {
            const int j = 2 * J + pj;
            if (j >= fy) break;
            T* row = xf + ((int64_t)k * fy + j) * fx + 2 * I;
#pragma unroll
            for (int pi = 0; pi < 2; ++pi) {
                if (2 * I + pi >= fx) break;
                const T w = T(1) / T((pi ? 1 : 2) * (pj ? 1 : 2) * (pk ? 1 : 2));
                T s = T(0);
#pragma unroll
                for (int c = pk; c < 2; ++c)
#pragma unroll
                    for (int b = pj; b < 2; ++b)
#pragma unroll
                        for (int a = pi; a < 2; ++a) s += w * e[c][b][a];
                row[pi] += s;
            }
        }
    }
}

// coarsest level in a launch of its own (ew_mg.cuh)
constexpr int kCoarseThreads = 512;

template <typename T, int DIM, int ORDER>
__global__ void __launch_bounds__(kCoarseThreads)
    k_mg_coarse_cg(int nx, int ny, int nz, const T* b, T* x, Stencil<T> sa, T rtol, int maxit) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    coarse_cg<T, DIM, ORDER>(nx, ny, nz, b, x, sa, rtol, maxit, reinterpret_cast<T*>(smem_raw));
}

template <typename T>
__global__ void k_guess_rhs(int64_t N, const T* __restrict__ w, T* __restrict__ b, T* __restrict__ x, T sc) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < N; q += (int64_t)gridDim.x * blockDim.x) {
        T v = sc * w[q];
        b[q] = v;
        if (x) x[q] = v;  // x == nullptr: keep the iterate as the guess
    }
}

// W^{n+1} = y - W^{n-1} (stored over W^{n-1}); acc += c W^{n+1}; first: acc = c0 W^0 + c1 W^1
template <typename T>
__global__ void k_implicit_update(int64_t N, const T* __restrict__ y, T* __restrict__ wprev, T* __restrict__ acc, T c) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < N; q += (int64_t)gridDim.x * blockDim.x) {
        T wn = y[q] - wprev[q];
        wprev[q] = wn;
        acc[q] += c * wn;
    }
}
template <typename T>
__global__ void k_implicit_first(int64_t N, const T* __restrict__ w0, const T* __restrict__ w1, T* __restrict__ acc,
                                 T c0, T c1) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < N; q += (int64_t)gridDim.x * blockDim.x)
        acc[q] = c0 * w0[q] + c1 * w1[q];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
template <typename T>
struct MGSolver {
    GridGeom lv[16];
    int nlev = 0;
    T* X[16];  // iterate (two buffers per level, X points at the current one)
    T* Tm[16];
    T* B[16];
    T* R[16];
    double a = 0.0;
    ew_grid* gr = nullptr;
    const ew_mg_params* p = nullptr;
    double wJ = 0.8;
    cudaStream_t st = nullptr;
    // FP32 fields: the learned levels' smoother as its composed stencil (one
    // build per solver set-up); EW_SMOOTHER_TWO_LAYER=1 keeps the two-layer
    // tensor-core form instead (a comparison hook)
    ComposedSmoother comp[16];
    bool use_comp = false;

    ew_status setup(ew_grid* g, double a_, const ew_mg_params* params, cudaStream_t s) {
        gr = g;
        a = a_;
        p = params;
        st = s;
        wJ = params->jacobi_weight > 0 ? params->jacobi_weight : 0.8;
        if (g->geom.bc)
            return set_error(EW_EUNSUPPORTED, "multigrid: boxes with Neumann faces are not implemented");
        if (g->geom.map) return set_error(EW_EUNSUPPORTED, "multigrid: mapped grids are not implemented");
        if (g->prec == EW_FP32X2) return set_error(EW_EUNSUPPORTED, "multigrid: FP32 or FP64 grids only");
        nlev = mg_levels(g->geom, lv, 16);
        {
            int dev = 0;
            EW_CUDA_TRY(cudaGetDevice(&dev));
            EW_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
        }
        f2 = sizeof(T) == 4 && mg_plane3d_f2_fits(g->geom);
        if (g->geom.dim == 3 && !f2) {
            const int s2 = (int)PlaneRing<T, 2>::SMEM, s4 = (int)PlaneRing<T, 4>::SMEM;
            const auto A = cudaFuncAttributeMaxDynamicSharedMemorySize;
            EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_plane3d<T, 2, 0>, A, s2));
            EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_plane3d<T, 2, 1>, A, s2));
            EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_plane3d<T, 2, 2>, A, s2));
            EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_plane3d<T, 4, 0>, A, s4));
            EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_plane3d<T, 4, 1>, A, s4));
            EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_plane3d<T, 4, 2>, A, s4));
            // resident CTAs a SM (the fewest over the modes): the z chunks fill them once
            int o = 0;
            pl_occ[0] = pl_occ[1] = 1 << 20;
            EW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_mg_plane3d<T, 2, 0>, kPlNT, s2));
            pl_occ[0] = std::min(pl_occ[0], o);
            EW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_mg_plane3d<T, 2, 1>, kPlNT, s2));
            pl_occ[0] = std::min(pl_occ[0], o);
            EW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_mg_plane3d<T, 2, 2>, kPlNT, s2));
            pl_occ[0] = std::min(pl_occ[0], o);
            EW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_mg_plane3d<T, 4, 0>, kPlNT, s4));
            pl_occ[1] = std::min(pl_occ[1], o);
            EW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_mg_plane3d<T, 4, 1>, kPlNT, s4));
            pl_occ[1] = std::min(pl_occ[1], o);
            EW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_mg_plane3d<T, 4, 2>, kPlNT, s4));
            pl_occ[1] = std::min(pl_occ[1], o);
            pl_occ[0] = std::max(pl_occ[0], 1);
            pl_occ[1] = std::max(pl_occ[1], 1);
        }
        if (g->geom.n[1] > 65535 || g->geom.n[2] > 65535)
            return set_error(EW_EUNSUPPORTED, "multigrid: axes longer than 65535 points");
        if (lv[nlev - 1].N > kCoarseMax)
            return set_error(EW_EUNSUPPORTED, "multigrid needs axes that halve down to at most 2048 coarse points "
                                              "(n = 2^k - 1 per axis, for example)");
        if (params->learned_levels > 0 && g->geom.dim != 3)
            return set_error(EW_EUNSUPPORTED, "the learned smoother is three-dimensional");
        if (params->learned_levels > 0 && !params->weights_dev)
            return set_error(EW_EINVAL, "learned_levels > 0 needs weights_dev");
        use_comp = sizeof(T) == 4 && params->learned_levels > 0 && !getenv("EW_SMOOTHER_TWO_LAYER");
        if (use_comp)
            for (int L = 0; L < std::min(params->learned_levels, nlev); ++L)
                EW_TRY(comp[L].build(params->weights_dev + (size_t)L * 432, st));
        size_t total = 0;
        for (int L = 0; L < nlev; ++L) total += 4 * (size_t)lv[L].N;
        EW_TRY(g->mgh.reserve(total * sizeof(T)));
        T* base = (T*)g->mgh.ptr;
        for (int L = 0; L < nlev; ++L) {
            X[L] = base;
            Tm[L] = base + lv[L].N;
            B[L] = base + 2 * lv[L].N;
            R[L] = base + 3 * lv[L].N;
            base += 4 * lv[L].N;
        }
        return EW_OK;
    }

    double diag(int L) const {
        double d0 = lv[L].order == 2 ? 2.0 : 2.5, s = 0.0;
        for (int q = 0; q < lv[L].dim; ++q) s += d0 / (lv[L].h[q] * lv[L].h[q]);
        return 1.0 + a * s;
    }

    // 3D levels: the 2.5D-blocked stencil kernel
    int nsm = 0, pl_occ[2] = {1, 1};  // SMs; resident plane-kernel CTAs a SM (order 2, order 4)
    bool f2 = false;                  // FP32: the paired form (ew_mg_plane.cu)
    template <int MODE>
    ew_status plane3d(const GridGeom& g_, const T* x, const T* b, T* out, const Stencil<T>& sa, T wd, int colour) {
        if constexpr (sizeof(T) == 4)
            if (f2) return mg_plane3d_f2(MODE, g_, x, b, out, sa, wd, colour, nsm, st);
        const int nx = (int)g_.n[0], ny = (int)g_.n[1], nz = (int)g_.n[2];
        const int bx = (nx + kPlBX - 1) / kPlBX, by = (ny + kPlBY - 1) / kPlBY;
        // z chunks: enough CTAs to fill the resident slots once, at least 8 planes each
        const int nzc = std::max(1, (pl_occ[g_.order == 2 ? 0 : 1] * nsm) / std::max(1, bx * by));
        const int zc = std::max(std::min(8, nz), (nz + nzc - 1) / nzc);
        const dim3 grid((unsigned)bx, (unsigned)by, (unsigned)((nz + zc - 1) / zc));
        if (g_.order == 2)
            k_mg_plane3d<T, 2, MODE><<<grid, kPlNT, PlaneRing<T, 2>::SMEM, st>>>(nx, ny, nz, zc, x, b, out, sa, wd,
                                                                              colour);
        else
            k_mg_plane3d<T, 4, MODE><<<grid, kPlNT, PlaneRing<T, 4>::SMEM, st>>>(nx, ny, nz, zc, x, b, out, sa, wd,
                                                                              colour);
        EW_CUDA_TRY(cudaGetLastError());
        count_launch();
        return EW_OK;
    }
    ew_status resid(int L, const Stencil<T>& sa) { return plane3d<0>(lv[L], X[L], B[L], R[L], sa, T(0), 0); }

    // 3D levels
    ew_status smooth(int L, int steps) {
        Stencil<T> sa = make_stencil<T>(lv[L], a);
        for (int s = 0; s < steps; ++s) {
            if (L < p->learned_levels) {
                EW_TRY(resid(L, sa));
                if constexpr (sizeof(T) == 4) {
                    if (use_comp) {
                        EW_TRY(comp[L].apply(lv[L], R[L], X[L], st));
                        continue;
                    }
                }
                EW_TRY(smoother_apply<T>(lv[L], p->weights_dev + (size_t)L * 432, R[L], X[L], st));
            } else if (p->red_black) {
                // 3D levels: one launch per colour
                const int ncol = lv[L].order == 2 ? 2 : 3;
                for (int colour = 0; colour < ncol; ++colour)
                    EW_TRY(plane3d<2>(lv[L], X[L], B[L], X[L], sa, weight(L, sa), colour));
            } else {
                EW_TRY(plane3d<1>(lv[L], X[L], B[L], Tm[L], sa, weight(L, sa), 0));
                std::swap(X[L], Tm[L]);
            }
        }
        return EW_OK;
    }

    // x += weight (b - M x): w / D (Jacobi), or 1 / M_ii with M_ii = 1 - c0 of the
    // stored (consistent) stencil of a L_h (colour sweeps)
    T weight(int L, const Stencil<T>& sa) const {
        return p->red_black ? (T)(1.0 / (1.0 - (double)sa.c0)) : (T)(wJ / diag(L));
    }

    // 2D levels: `steps` sweeps, a few a launch; the first launch adds the
    // prolongation of the coarse iterate when `correct`
    ew_status smooth2d(int L, int steps, bool correct) {
        const Stencil<T> sa = make_stencil<T>(lv[L], a);
        const int most = mg_smooth2d_sweeps<T>(lv[L], p->red_black != 0);
        while (steps > 0) {
            const int ns = std::min(steps, most);
            EW_TRY(mg_smooth2d<T>(lv[L], X[L], B[L], Tm[L], sa, weight(L, sa), p->red_black != 0, ns,
                                  correct ? X[L + 1] : nullptr, correct ? &lv[L + 1] : nullptr, st));
            std::swap(X[L], Tm[L]);
            correct = false;
            steps -= ns;
        }
        return EW_OK;
    }

    // The levels from L down to the coarsest and back in one launch of one CTA,
    // once they are small: up to 31^2 points in FP64 (63^2 would take that SM's
    // FP64 units over 37 us, three launches 15-20 us), 4096 in FP32
    bool bottom_fits(int L) const {
        if (L < p->learned_levels || L == 0 || nlev - L > kMgBottomLevels) return false;
        if (lv[L].N > (sizeof(T) == 8 ? 1024 : 4096)) return false;
        int64_t n[kMgBottomLevels];
        for (int l = L; l < nlev; ++l) n[l - L] = lv[l].N;
        return mg_bottom_smem<T>(n, nlev - L) <= 200 * 1024;
    }
    ew_status bottom(int L) {
        MgBottom<T> m;
        m.nlev = nlev - L;
        m.pre = p->pre;
        m.post = p->post;
        m.colours = p->red_black ? (lv[L].order == 2 ? 2 : 3) : 0;
        m.cg_rtol = cg_rtol();
        m.cg_maxit = cg_maxit(lv[nlev - 1]);
        m.cg_off = 0;
        m.b = B[L];
        m.x = X[L];
        for (int l = L; l < nlev; ++l) {
            MgBottomLevel<T>& q = m.lv[l - L];
            for (int d = 0; d < 3; ++d) q.n[d] = (int)lv[l].n[d];
            q.sa = make_stencil<T>(lv[l], a);
            q.wd = weight(l, q.sa);
        }
        return mg_bottom<T>(lv[L].dim, lv[L].order, m, st);
    }

    static T cg_rtol() { return sizeof(T) == 4 ? T(1e-7) : T(1e-14); }
    static int cg_maxit(const GridGeom& c) { return (int)std::min<int64_t>(4 * c.N + 10, 4000); }
    ew_status coarse(int L) {
        Stencil<T> sa = make_stencil<T>(lv[L], a);
        const GridGeom& c = lv[L];
        size_t smem = coarse_cg_smem<T>(c.N);
        const T rtol = cg_rtol();
        const int maxit = cg_maxit(c);
        if (c.dim == 2 && c.order == 2)
            k_mg_coarse_cg<T, 2, 2><<<1, kCoarseThreads, smem, st>>>((int)c.n[0], (int)c.n[1], 1, B[L], X[L], sa, rtol, maxit);
        else if (c.dim == 2)
            k_mg_coarse_cg<T, 2, 4><<<1, kCoarseThreads, smem, st>>>((int)c.n[0], (int)c.n[1], 1, B[L], X[L], sa, rtol, maxit);
        else if (c.order == 2)
            k_mg_coarse_cg<T, 3, 2><<<1, kCoarseThreads, smem, st>>>((int)c.n[0], (int)c.n[1], (int)c.n[2], B[L], X[L], sa, rtol, maxit);
        else
            k_mg_coarse_cg<T, 3, 4><<<1, kCoarseThreads, smem, st>>>((int)c.n[0], (int)c.n[1], (int)c.n[2], B[L], X[L], sa, rtol, maxit);
        count_launch();
        EW_CUDA_TRY(cudaGetLastError());
        return EW_OK;
    }

    ew_status vcycle(int L) {
        if (bottom_fits(L)) return bottom(L);
        if (L == nlev - 1) return coarse(L);
        const GridGeom &f = lv[L], &c = lv[L + 1];
        const Stencil<T> sa = make_stencil<T>(f, a);
        if (f.dim == 2) {
            EW_TRY(smooth2d(L, p->pre, false));
            EW_TRY(mg_resid_restrict2d<T>(f, c, X[L], B[L], B[L + 1], X[L + 1], sa, st));
            EW_TRY(vcycle(L + 1));
            if (p->post > 0) return smooth2d(L, p->post, true);
            // no smoothing afterwards: the correction alone
            return mg_prolong2d<T>(f, c, X[L + 1], X[L], st);
        }
        EW_TRY(smooth(L, p->pre));
        EW_TRY(resid(L, sa));
        k_mg_restrict3d<T><<<pt_grid(c.n[0], c.n[1], c.n[2]), pt_threads(c.n[0]), 0, st>>>(
            f.n[0], f.n[1], f.n[2], c.n[0], c.n[1], c.n[2], R[L], B[L + 1], X[L + 1]);
        count_launch();
        EW_TRY(vcycle(L + 1));
        {
            const int64_t hx = (f.n[0] + 1) / 2;
            const dim3 pg((unsigned)((hx + 127) / 128), (unsigned)((f.n[1] + 1) / 2), (unsigned)((f.n[2] + 1) / 2));
            k_mg_prolong3d<T><<<pg, 128, 0, st>>>((int)f.n[0], (int)f.n[1], (int)f.n[2], (int)c.n[0], (int)c.n[1],
                                                  (int)c.n[2], X[L + 1], X[L]);
        }
        count_launch();
        EW_TRY(smooth(L, p->post));
        EW_CUDA_TRY(cudaGetLastError());
        return EW_OK;
    }

    // the current top-level iterate lives in X[0]; callers load b into B[0]
    // and the initial guess into X[0]
    ew_status cycles(int ncyc) {
        for (int c = 0; c < ncyc; ++c) EW_TRY(vcycle(0));
        return EW_OK;
    }

    // ||B[0]||_2 or ||B[0] - M X[0]||_2 (FP64 reduction, synchronises)
    ew_status norm2(bool residual, double* out) {
        constexpr int nb = 2 * kReduceBlocks;
        EW_TRY(gr->reduce.reserve(sizeof(double) * (nb + 8)));
        double* dpart = (double*)gr->reduce.ptr;
        double* dres = dpart + nb;
        if (!residual) {
            EW_TRY(launch_dots<T>(B[0], B[0], lv[0].N, 1, dpart, dres, st));
        } else if (lv[0].dim == 2) {
            EW_TRY(mg_resid_norm2d<T>(lv[0], X[0], B[0], make_stencil<T>(lv[0], a), dpart, nb, st));
            EW_TRY(launch_finish_sum(dpart, nb, 1, dres, st));
        } else {
            EW_TRY(resid(0, make_stencil<T>(lv[0], a)));
            EW_TRY(launch_dots<T>(R[0], R[0], lv[0].N, 1, dpart, dres, st));
        }
        void* hp = nullptr;  // page-locked: a copy into pageable memory is staged by the driver
        EW_TRY(pinned(gr, sizeof(double), &hp));
        EW_CUDA_TRY(cudaMemcpyAsync(hp, dres, sizeof(double), cudaMemcpyDeviceToHost, st));
        EW_CUDA_TRY(cudaStreamSynchronize(st));
        *out = sqrt(*(const double*)hp);
        return EW_OK;
    }

    // V-cycles until ||B - M X||_2 <= rtol ||B||_2, tested after every cycle,
    // or max_cycles; rtol <= 0 runs max_cycles without a test
    ew_status solve(int max_cycles, double rtol, int* used) {
        if (!(rtol > 0.0)) {
            *used = max_cycles;
            return cycles(max_cycles);
        }
        double bn = 0.0;
        EW_TRY(norm2(false, &bn));
        int c = 0;
        while (c < max_cycles) {
            EW_TRY(vcycle(0));
            ++c;
            double rk = 0.0;
            EW_TRY(norm2(true, &rk));
            if (rk <= rtol * bn) break;
        }
        *used = c;
        return EW_OK;
    }
};

template <typename T>
static ew_status coarse_smem_attr() {
    size_t smem = sizeof(T) * (4 * (size_t)kCoarseMax + 32);
    EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_coarse_cg<T, 2, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_coarse_cg<T, 2, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_coarse_cg<T, 3, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    EW_CUDA_TRY(cudaFuncSetAttribute(k_mg_coarse_cg<T, 3, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return EW_OK;
}

static ew_status check_mg(const ew_mg_params* mg) {
    if (!mg) return set_error(EW_EINVAL, "the implicit scheme needs multigrid parameters (params->mg)");
    if (mg->pre < 0 || mg->post < 0 || mg->pre + mg->post < 1) return set_error(EW_EINVAL, "bad smoothing counts");
    if (mg->max_cycles < 1) return set_error(EW_EINVAL, "max_cycles must be >= 1");
    if (mg->learned_levels < 0) return set_error(EW_EINVAL, "learned_levels < 0");
    if (mg->red_black != 0 && mg->red_black != 1) return set_error(EW_EINVAL, "red_black must be 0 or 1");
    if (mg->guess != 0 && mg->guess != 1) return set_error(EW_EINVAL, "guess must be 0 or 1");
    return EW_OK;
}

template <typename T>
static ew_status implicit_wave_solve_t(ew_grid* g, const FilterPlan& plan, const ew_filter_params* p, const T* vin,
                                       T* vout, int nvec, cudaStream_t st) {
    EW_TRY(check_mg(p->mg));
    EW_TRY(coarse_smem_attr<T>());
    const int64_t N = g->geom.N;
    MGSolver<T> mg;
    EW_TRY(mg.setup(g, 0.5 * plan.dt * plan.dt, p->mg, st));
    EW_TRY(g->fields.reserve(2 * (size_t)N * sizeof(T)));
    T* Wm = (T*)g->fields.ptr;  // W^{n-1}
    T* W0 = Wm + N;             // W^n
    const int blocks = grid_blocks(N, 256);
    for (int v = 0; v < nvec; ++v) {
        const T* x = vin + (size_t)v * N;
        T* acc = vout + (size_t)v * N;
        // W^0 = V; M W^1 = W^0 (initial guess W^0)
        EW_CUDA_TRY(cudaMemcpyAsync(Wm, x, N * sizeof(T), cudaMemcpyDeviceToDevice, st));
        k_guess_rhs<T><<<blocks, 256, 0, st>>>(N, x, mg.B[0], mg.X[0], T(1));
        count_launch();
        int used = 0;
        EW_TRY(mg.solve(p->mg->max_cycles, p->mg->rtol, &used));
        count_mg_solve(used);
        EW_CUDA_TRY(cudaMemcpyAsync(W0, mg.X[0], N * sizeof(T), cudaMemcpyDeviceToDevice, st));
        k_implicit_first<T><<<blocks, 256, 0, st>>>(N, Wm, W0, acc, (T)plan.c[0], (T)plan.c[1]);
        count_launch();
        for (int64_t n = 1; n < plan.Nt; ++n) {
            // M y = 2 W^n from y = 2 W^n, or (guess 1, n >= 2) from the previous
            // system's solution, which X[0] still holds; W^{n+1} = y - W^{n-1} over W^{n-1}
            const bool keep = p->mg->guess == 1 && n >= 2;
            k_guess_rhs<T><<<blocks, 256, 0, st>>>(N, W0, mg.B[0], keep ? nullptr : mg.X[0], T(2));
            count_launch();
            EW_TRY(mg.solve(p->mg->max_cycles, p->mg->rtol, &used));
            count_mg_solve(used);
            k_implicit_update<T><<<blocks, 256, 0, st>>>(N, mg.X[0], Wm, acc, (T)plan.c[(size_t)n + 1]);
            count_launch();
            std::swap(Wm, W0);
        }
    }
    EW_CUDA_TRY(cudaGetLastError());
    return EW_OK;
}

ew_status implicit_wave_solve_any(ew_grid* g, const FilterPlan& plan, const ew_filter_params* p, const void* vin,
                                  void* vout, int nvec, cudaStream_t st) {
    if (g->prec == EW_FP32)
        return implicit_wave_solve_t<float>(g, plan, p, (const float*)vin, (float*)vout, nvec, st);
    return implicit_wave_solve_t<double>(g, plan, p, (const double*)vin, (double*)vout, nvec, st);
}

template <typename T>
ew_status launch_dots(const T* x, const T* y, int64_t N, int nvec, double* part, double* out, cudaStream_t st);

template <typename T>
static ew_status step_mg_t(ew_grid* g, double a, const T* rhs, T* x, const ew_mg_params* mp, double* conv,
                           int* cycles_done, cudaStream_t st) {
    EW_TRY(check_mg(mp));
    EW_TRY(coarse_smem_attr<T>());
    const int64_t N = g->geom.N;
    MGSolver<T> mg;
    EW_TRY(mg.setup(g, a, mp, st));
    EW_CUDA_TRY(cudaMemcpyAsync(mg.B[0], rhs, N * sizeof(T), cudaMemcpyDeviceToDevice, st));
    EW_CUDA_TRY(cudaMemcpyAsync(mg.X[0], x, N * sizeof(T), cudaMemcpyDeviceToDevice, st));
    double bnorm = 0.0, r0 = 0.0, rk = 0.0;
    EW_TRY(mg.norm2(false, &bnorm));
    EW_TRY(mg.norm2(true, &r0));
    rk = r0;
    int c = 0;
    for (c = 0; c < mp->max_cycles; ++c) {
        if (mp->rtol > 0 && rk <= mp->rtol * bnorm) break;
        EW_TRY(mg.vcycle(0));
        if (mp->rtol > 0 || c + 1 == mp->max_cycles) EW_TRY(mg.norm2(true, &rk));
    }
    EW_CUDA_TRY(cudaMemcpyAsync(x, mg.X[0], N * sizeof(T), cudaMemcpyDeviceToDevice, st));
    EW_CUDA_TRY(cudaStreamSynchronize(st));
    if (conv) *conv = (c > 0 && r0 > 0) ? pow(rk / r0, 1.0 / c) : 0.0;
    if (cycles_done) *cycles_done = c;
    if (mp->rtol > 0 && rk > mp->rtol * bnorm) return set_error(EW_ENOCONV, "multigrid did not reach rtol");
    return EW_OK;
}

ew_status splitmix_uniform(int64_t n, uint64_t seed, double* out, cudaStream_t st);
template <typename S, typename D>
ew_status convert(int64_t n, const S* x, D* y, cudaStream_t st);

// Residual samples for training the learned smoother: for rhs number q
// (uniform [-1,1) from SplitMix64 stream seed + q) plain V-cycles run from
// x = 0, and the residual b - M x the finest-level smoother sees at the start
// of cycles 0, 1, 2 is recorded, until nsamples residuals (FP32) are stored.
ew_status mg_collect_residuals(ew_grid* g, double a, const ew_mg_params* mp, int nsamples, uint64_t seed, float* out,
                               cudaStream_t st) {
    EW_TRY(check_mg(mp));
    EW_TRY(coarse_smem_attr<float>());
    const int64_t N = g->geom.N;
    MGSolver<float> mg;
    EW_TRY(mg.setup(g, a, mp, st));
    DeviceBuffer tmp_buf;
    EW_TRY(tmp_buf.alloc(sizeof(double) * (size_t)N));
    double* tmp = tmp_buf.as<double>();
    Stencil<float> sa = make_stencil<float>(g->geom, a);
    ew_status s = EW_OK;
    int k = 0;
    for (uint64_t q = 0; k < nsamples && s == EW_OK; ++q) {
        s = splitmix_uniform(N, seed + q, tmp, st);
        if (s == EW_OK) s = convert<double, float>(N, tmp, mg.B[0], st);
        if (s != EW_OK) break;
        cudaMemsetAsync(mg.X[0], 0, sizeof(float) * N, st);
        for (int c = 0; c < 3 && k < nsamples && s == EW_OK; ++c) {
            float* r = out + (size_t)k * N;
            const GridGeom& gg = g->geom;
            s = mg.template plane3d<0>(gg, mg.X[0], mg.B[0], r, sa, 0.f, 0);
            ++k;
            if (s == EW_OK) s = mg.vcycle(0);
        }
    }
    cudaStreamSynchronize(st);
    return s;
}

// Convergence factor of ncycles V-cycles on M x = b, b uniform [-1,1) from
// stream seed, x = 0: (||r_n|| / ||r_1||)^(1 / (n - 1)), skipping the first
// cycle's transient.
ew_status mg_convergence(ew_grid* g, double a, const ew_mg_params* mp, int ncycles, uint64_t seed, double* rho,
                         cudaStream_t st) {
    const int64_t N = g->geom.N;
    DeviceBuffer tmp_buf, b_buf, x_buf;
    EW_TRY(tmp_buf.alloc(sizeof(double) * (size_t)N));
    EW_TRY(b_buf.alloc(sizeof(float) * (size_t)N));
    EW_TRY(x_buf.alloc(sizeof(float) * (size_t)N));
    double* tmp = tmp_buf.as<double>();
    float* b = b_buf.as<float>();
    float* x = x_buf.as<float>();
    ew_status s = splitmix_uniform(N, seed, tmp, st);
    if (s == EW_OK) s = convert<double, float>(N, tmp, b, st);
    cudaMemsetAsync(x, 0, sizeof(float) * N, st);
    ew_mg_params one = *mp;
    one.max_cycles = 1;
    one.rtol = 0.0;
    double c1 = 0.0;
    if (s == EW_OK) s = step_mg_t<float>(g, a, b, x, &one, &c1, nullptr, st);  // r_1 / r_0
    ew_mg_params rest = *mp;
    rest.max_cycles = std::max(1, ncycles - 1);
    rest.rtol = 0.0;
    double cr = 0.0;
    if (s == EW_OK) s = step_mg_t<float>(g, a, b, x, &rest, &cr, nullptr, st);
    cudaStreamSynchronize(st);
    *rho = cr;
    return s;
}

}  // namespace ew

using namespace ew;

extern "C" ew_status ew_implicit_step_mg(const ew_grid* grid, double half_dt2, const void* rhs, void* x,
                                         const ew_mg_params* mg, double* conv_factor, int* cycles_done,
                                         cudaStream_t stream) try {
    clear_error();
    if (!grid || !rhs || !x || !mg) return set_error(EW_EINVAL, "null argument");
    if (!(half_dt2 >= 0.0) || !std::isfinite(half_dt2)) return set_error(EW_EINVAL, "half_dt2 must be finite and >= 0");
    {
        const size_t bytes = (size_t)grid->geom.N * (grid->prec == EW_FP32 ? 4 : 8);
        const char* a = (const char*)rhs;
        const char* b = (const char*)x;
        if (a < b + bytes && b < a + bytes) return set_error(EW_EINVAL, "rhs and x overlap");
    }
    int dev = -1;
    EW_CUDA_TRY(cudaGetDevice(&dev));
    if (grid->device >= 0 && grid->device != dev) return set_error(EW_EINVAL, "grid was created on another device");
    ew_grid* g = const_cast<ew_grid*>(grid);
    if (g->prec == EW_FP32)
        return step_mg_t<float>(g, half_dt2, (const float*)rhs, (float*)x, mg, conv_factor, cycles_done, stream);
    return step_mg_t<double>(g, half_dt2, (const double*)rhs, (double*)x, mg, conv_factor, cycles_done, stream);
} catch (...) {
    return abi_exception();
}
