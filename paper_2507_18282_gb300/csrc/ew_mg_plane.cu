// ew_mg_plane.cu -- stencil operations of the multigrid cycle on 3D FP32 levels
// (residual, damped Jacobi, one colour of a multi-colour sweep), streamed along
// z.
//
// A CTA covers 64 x 32 points of the box (16 warps, two columns and two rows a
// thread, paired FP32 instructions), of which all but a rim of R = order / 2
// are outputs, and a chunk of planes.  The planes of x arrive by asynchronous
// copies kMpAhead planes ahead in a ring in shared memory; the z-neighbours of
// a thread's points stay in its registers, b is loaded one plane ahead.  One
// barrier a plane; two CTAs share an SM.  Dirichlet closure: walls hold 0, a
// point beyond a wall the negated mirror (negated in place by the thread that
// copied it).  The operations of a point and their order are those of
// k_mg_plane3d (ew_mg.cu), which keeps the FP64 levels.
//
// Bound: instruction issue (260 instructions a warp and plane, issued on 67 %
// of the cycles).  Measured, 255^3 order 4, one residual: 90 us (64 x 8 columns a
// CTA, scalar instructions, every stencil point from shared memory) -> 79 us;
// Jacobi sweep on 31^3 10.0 -> 6.6 us.
#include <stdlib.h>

#include <algorithm>

#include "ew_internal.h"
#include "ew_mg.cuh"
#include "ew_tb2d_dev.cuh"  // cp_async4, p_add, p_mul, p_fma, s_add

namespace ew {

constexpr int kMpX = 64, kMpY = 32, kMpPlane = kMpX * kMpY, kMpThreads = 512, kMpAhead = 2;

template <int N>
__device__ __forceinline__ void mp_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

// index of coordinate i under the odd closure: -1 for a wall (or farther than
// the stencil reaches), else the mirror, with sg negated beyond a wall
__device__ __forceinline__ int mp_ext(int i, int n, int& sg) {
    if (i >= 0 && i < n) return i;
    if (i == -1 || i == n || i < -2 || i > n + 1) return -1;
    sg = -sg;
    const int m = i < 0 ? -2 - i : 2 * n - i;
    return m >= 0 && m < n ? m : -1;
}

// MODE 0: out = b - M x; 1: out = x + wd (b - M x); 2: the same in place at the
// points of colour `colour`
template <int ORDER, int MODE>
__global__ void __launch_bounds__(kMpThreads, 2)
    k_mg_plane3d_f2(int nx, int ny, int nz, int zc, const float* x, const float* __restrict__ b, float* out,
                    Stencil<float> sa, float wd, int colour) {
    constexpr int R = ORDER == 2 ? 1 : 2, Q = 2 * R + 1, NW = R + 1 + kMpAhead;
    constexpr int TX = kMpX - 4, TY = kMpY - 2 * R;  // rim of two columns either side: pairs are outputs or not
    extern __shared__ __align__(16) unsigned char smem_mp[];
    float* sX = reinterpret_cast<float*>(smem_mp);  // [NW][plane]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = 2 * lane, r0 = 2 * warp;
    const int gx = blockIdx.x * TX - 2 + c, gy0 = blockIdx.y * TY - R + r0;
    const int zs = blockIdx.z * zc, ze = min(nz, zs + zc);
    const int64_t plane = (int64_t)nx * ny;
    int sxa = 1, sxb = 1;
    const int ixa = mp_ext(gx, nx, sxa), ixb = mp_ext(gx + 1, nx, sxb);
    const bool own_x = c >= 2 && c < 2 + TX && gx < nx, own_xb = own_x && gx + 1 < nx;
    unsigned srca[2], srcb[2];
    int sga[2], sgb[2];
    bool own[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        int sy = 1;
        const int iy = mp_ext(gy0 + j, ny, sy);
        sga[j] = (ixa < 0 || iy < 0) ? 0 : sxa * sy;
        sgb[j] = (ixb < 0 || iy < 0) ? 0 : sxb * sy;
        srca[j] = sga[j] ? (unsigned)iy * (unsigned)nx + (unsigned)ixa : 0u;
        srcb[j] = sgb[j] ? (unsigned)iy * (unsigned)nx + (unsigned)ixb : 0u;
        own[j] = own_x && r0 + j >= R && r0 + j < R + TY && gy0 + j < ny;
    }
    const bool flips = sga[0] < 0 || sga[1] < 0 || sgb[0] < 0 || sgb[1] < 0;
    const unsigned o = (unsigned)gy0 * (unsigned)nx + (unsigned)gx;  // modulo 2^32: a rim row's is unused
    const unsigned b00 = own[0] ? o : 0u, b01 = own[0] && own_xb ? o + 1u : 0u;
    const unsigned b10 = own[1] ? o + (unsigned)nx : 0u, b11 = own[1] && own_xb ? o + (unsigned)nx + 1u : 0u;
    const int me = r0 * kMpX + c;
    const int xm = max(c - 2, 0) - c, xp = min(c + 2, kMpX - 2) - c;
    int up[R], dw[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        up[q] = max(r0 - 1 - q, 0) * kMpX + c;
        dw[q] = min(r0 + 2 + q, kMpY - 1) * kMpX + c;
    }
    for (int q = 0; q < NW; ++q)  // walls: 0 for good
#pragma unroll
        for (int j = 0; j < 2; ++j) *reinterpret_cast<float2*>(sX + q * kMpPlane + me + j * kMpX) = make_float2(0.f, 0.f);

    const int zlo = zs - R, zhi = ze + R;
    auto copy_x = [&](int z, int slot) {
        if (z < zhi) {
            int sg = 1;
            const int iz = mp_ext(z, nz, sg);
            float* w = sX + slot * kMpPlane + me;
            const float* p = x + (int64_t)iz * plane;
            if (iz < 0) {
                *reinterpret_cast<float2*>(w) = *reinterpret_cast<float2*>(w + kMpX) = make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (sga[j]) cp_async4(w + j * kMpX, p + srca[j]);
                    if (sgb[j]) cp_async4(w + j * kMpX + 1, p + srcb[j]);
                }
            }
        }
        mp_commit();
    };
    auto load_b = [&](int z, float2 (&v)[2]) {  // only owned points are used
        if (z < zs || z >= ze) return;
        const float* p = b + (int64_t)z * plane;
        v[0] = make_float2(p[b00], p[b01]);
        v[1] = make_float2(p[b10], p[b11]);
    };
    float2 wq[Q][2];
#pragma unroll
    for (int q = 0; q < Q; ++q) wq[q][0] = wq[q][1] = make_float2(0.f, 0.f);
    const float2 C0{sa.c0, sa.c0}, C1X{sa.c1[0], sa.c1[0]}, C1Y{sa.c1[1], sa.c1[1]}, C1Z{sa.c1[2], sa.c1[2]};
    const float2 C2X{sa.c2[0], sa.c2[0]}, C2Y{sa.c2[1], sa.c2[1]}, C2Z{sa.c2[2], sa.c2[2]}, WD{wd, wd};
    const float2 M1{-1.f, -1.f};
#pragma unroll
    for (int q = 0; q < kMpAhead; ++q) copy_x(zlo + q, q);
    float2 bn[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    load_b(zlo - R, bn);
    int ws = 0;
    for (int zb = zlo; zb < zhi; zb += Q) {
#pragma unroll
        for (int t = 0; t < Q; ++t) {  // queue entry q of step zb + t is register (q + t + 1) mod Q
            const int z = zb + t;
            if (z >= zhi) break;
            mp_wait<kMpAhead - 1>();
            float2 bv[2] = {bn[0], bn[1]};
            {
                float* p = sX + ws * kMpPlane + me;
                float2 v[2] = {*reinterpret_cast<const float2*>(p), *reinterpret_cast<const float2*>(p + kMpX)};
                if (flips || z < 0 || z >= nz) {
                    int sz = 1;
                    mp_ext(z, nz, sz);
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        if (sga[j] * sz < 0) v[j].x = -v[j].x;
                        if (sgb[j] * sz < 0) v[j].y = -v[j].y;
                    }
                    *reinterpret_cast<float2*>(p) = v[0];
                    *reinterpret_cast<float2*>(p + kMpX) = v[1];
                }
                wq[t][0] = v[0];
                wq[t][1] = v[1];
            }
            {   // into a slot last read in the previous step
                int w2 = ws + kMpAhead;
                if (w2 >= NW) w2 -= NW;
                copy_x(z + kMpAhead, w2);
            }
            load_b(z + 1 - R, bn);
            int wr = ws - R;
            if (wr < 0) wr += NW;
            const float* sq = sX + wr * kMpPlane;
#define EW_Q(q) wq[((q) + t + 1) % Q]
            const float2 u[2] = {EW_Q(R)[0], EW_Q(R)[1]};
            float2 ru[R], rd[R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                ru[q] = *reinterpret_cast<const float2*>(sq + up[q]);
                rd[q] = *reinterpret_cast<const float2*>(sq + dw[q]);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float2 L = *reinterpret_cast<const float2*>(sq + me + j * kMpX + xm);
                const float2 P = *reinterpret_cast<const float2*>(sq + me + j * kMpX + xp);
                float2 sx1;
                sx1.x = s_add(L.y, u[j].y);
                sx1.y = s_add(u[j].x, P.x);
                float2 lap = p_mul(C0, u[j]);
                lap = p_fma(C1X, sx1, lap);
                lap = p_fma(C1Y, j == 0 ? p_add(ru[0], u[1]) : p_add(u[0], rd[0]), lap);
                lap = p_fma(C1Z, p_add(EW_Q(R - 1)[j], EW_Q(R + 1)[j]), lap);
                if constexpr (R == 2) {
                    lap = p_fma(C2X, p_add(L, P), lap);
                    lap = p_fma(C2Y, j == 0 ? p_add(ru[R - 1], rd[0]) : p_add(ru[0], rd[R - 1]), lap);
                    lap = p_fma(C2Z, p_add(EW_Q(0)[j], EW_Q(Q - 1)[j]), lap);
                }
                const float2 r = p_add(p_fma(M1, u[j], bv[j]), lap);  // (b - x) + a L x
                const float2 v = MODE == 0 ? r : p_fma(WD, r, u[j]);
                const int pz = z - R;
                if (own[j] && pz >= zs) {
                    const int64_t at = pz * plane + (o + (unsigned)(j * nx));
                    if (MODE < 2) {
                        out[at] = v.x;
                        if (own_xb) out[at + 1] = v.y;
                    } else {
                        const int s = gx + gy0 + j + pz;
                        if ((ORDER == 2 ? (s & 1) : s % 3) == colour) out[at] = v.x;
                        if (own_xb && (ORDER == 2 ? ((s + 1) & 1) : (s + 1) % 3) == colour) out[at + 1] = v.y;
                    }
                }
            }
#undef EW_Q
            ws = ws + 1 == NW ? 0 : ws + 1;
            __syncthreads();
        }
    }
    mp_wait<0>();
}

bool mg_plane3d_f2_fits(const GridGeom& g) { return g.n[0] * g.n[1] < INT32_MAX && g.n[1] <= 65535 * 28; }

template <int MODE>
static ew_status plane(const GridGeom& g, const float* x, const float* b, float* out, const Stencil<float>& sa, float wd,
                       int colour, int nsm, cudaStream_t st) {
    const int nx = (int)g.n[0], ny = (int)g.n[1], nz = (int)g.n[2], R = g.order == 2 ? 1 : 2;
    const int64_t tx = (nx + kMpX - 5) / (kMpX - 4), ty = (ny + kMpY - 2 * R - 1) / (kMpY - 2 * R);
    // z chunks: waves of CTAs (two an SM) times the planes of a chunk with its lead-in, at its least
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int c = 1; c <= std::min(nz, 128); ++c) {
        const int64_t zc = (nz + c - 1) / c, waves = (tx * ty * c + 2 * nsm - 1) / (2 * nsm);
        if (waves * (zc + 2 * R + 4) < cost) {
            cost = waves * (zc + 2 * R + 4);
            best = c;
        }
    }
    const int zc = (nz + best - 1) / best;
    const dim3 grid((unsigned)tx, (unsigned)ty, (unsigned)((nz + zc - 1) / zc));
    const size_t smem = sizeof(float) * (size_t)(R + 1 + kMpAhead) * kMpPlane;
    auto kern = g.order == 2 ? k_mg_plane3d_f2<2, MODE> : k_mg_plane3d_f2<4, MODE>;
    EW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    kern<<<grid, kMpThreads, smem, st>>>(nx, ny, nz, zc, x, b, out, sa, wd, colour);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}

ew_status mg_plane3d_f2(int mode, const GridGeom& g, const float* x, const float* b, float* out,
                        const Stencil<float>& sa, float wd, int colour, int nsm, cudaStream_t st) {
    if (const char* e = getenv("EW_TEST_MG_PLANE_FAIL"))  // test hook: launches of this mode fail
        if (atoi(e) == mode) return cuda_error(cudaErrorLaunchOutOfResources, "multigrid plane kernel (test hook)");
    if (mode == 0) return plane<0>(g, x, b, out, sa, wd, colour, nsm, st);
    if (mode == 1) return plane<1>(g, x, b, out, sa, wd, colour, nsm, st);
    return plane<2>(g, x, b, out, sa, wd, colour, nsm, st);
}

}  // namespace ew
