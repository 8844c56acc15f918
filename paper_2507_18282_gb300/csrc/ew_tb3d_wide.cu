// ew_tb3d_wide.cu -- temporally blocked fused leapfrog + filter steps on 3D
// grids, FP32, second and fourth order (eqs. explicitScheme,
// filterQuadrature), in the summed form of the recurrence (ew_stencil.cu).
//
// 2.5D blocking as in ew_tb3d.cu: a CTA owns a column of the box and streams it
// along z; the B time levels of one launch are pipelined R planes apart (R =
// order / 2), so at step z level 0 brings in plane z of W^n and level k
// computes plane z - R k from level k-1's planes around it.  One barrier a
// plane serves all levels.  Here a CTA covers 64 x 32 points (16 warps, two
// columns and two rows a thread, paired FP32 instructions), the box's z extent
// is cut into chunks where the columns alone would not fill the SMs evenly,
// and the inputs arrive ahead of their use: W^n by asynchronous copies three
// planes ahead, straight into the ring that level 1 reads its
// x/y neighbours from; D^n and the filter sums are loaded one plane ahead into
// registers.  Each thread keeps the 2R+1 planes of its own points per level, and
// the D of the last R planes of each level but the last, in registers; the x/y
// neighbours come from shared memory (a ring of R+1 planes a level; order 2:
// the columns beside a pair from the neighbouring lanes).
//
// Points outside the box are the box closure's extension (ew_bc_dev.cuh): the
// copying thread negates odd mirrors in place once they have arrived, walls
// stay 0, and the update keeps the extension exact.  Wrong x/y neighbours at
// the region's edge spread R points a level and stay inside the rim.
//
// Order of operations.  Second order: that of k_step_tb3d.  Fourth order:
// that of k_step3d (the first terms of each Laplacian part contracted into one
// multiply-add), so a solve at one step a launch gives the same bits.
//
// Why this shape.  Owned points are 1344 of 2048 at depth 2 of order 4 and 1456
// at depth 3 of order 2, against 576 and 676 of 1024 for a 32 x 32 region; four
// points a thread share their row neighbours and every per-plane cost.  All
// inputs and results move as single elements: the same kernel with 8-byte
// copies, pair loads and pair stores on padded rows took 4.33 ms where this
// one takes 3.55 ms (255^3, order 4, 43 steps).  Bound: instruction latency at
// 16 warps an SM (330 instructions a warp and plane at order 4, issued on 44 % of the
// cycles).  Measured: 511^3 order 2, 117 steps 44.7 (32 x 32 region, one row a
// thread) -> 39.2 ms; 191 x 161 x 143 order 4, 2 vectors, 151 steps 14.5 (one
// step a launch) -> 8.0 ms; 255^3 order 4 100 -> 200 Gcell-steps/s.
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "ew_bc_dev.cuh"
#include "ew_internal.h"
#include "ew_tb2d_dev.cuh"  // cp_async4/8, p_add, p_mul, p_fma, s_add

namespace ew {

constexpr int kWX = 64, kWY = 32, kWPlane = kWX * kWY, kWThreads = 512;

template <int R, int B>
struct Tb3wShape {
    static constexpr int H = R * B;                   // planes of lead-in and run-out, rim rows
    static constexpr int HX = (H + 1) & ~1;           // rim columns: even, so column pairs stay aligned
    static constexpr int TX = kWX - 2 * HX, TY = kWY - 2 * H;
    static constexpr int PF = 3;                      // planes of W^n in flight
    static constexpr int NW = R + 1 + PF;             // W^n ring
    static constexpr int NL = R + 1;                  // ring of each level but the last
    static constexpr size_t SMEM = sizeof(float) * (size_t)kWPlane * (NW + (B - 1) * NL);
    static_assert(TX > 0 && TY > 0, "rim larger than the region");
};

template <int N>
__device__ __forceinline__ void cp_async_wait_group() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }

template <int R, int B>
__global__ void __launch_bounds__(kWThreads, 1)
    k_step_tb3d_wide(int nx, int ny, int nz, const float* __restrict__ Din, const float* __restrict__ Win,
                     float* __restrict__ Dout, float* __restrict__ Wout, float* __restrict__ acc,
                     const float* __restrict__ cw, Stencil<float> st, int64_t fstride, int nzc, int zc) {
    using S = Tb3wShape<R, B>;
    constexpr int H = S::H, HX = S::HX, TX = S::TX, TY = S::TY, PF = S::PF, NW = S::NW, NL = S::NL;
    extern __shared__ __align__(16) unsigned char smem_w[];
    float* sW = reinterpret_cast<float*>(smem_w);  // [NW][plane]
    float* sL = sW + NW * kWPlane;                 // [B - 1][NL][plane]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = 2 * lane, r0 = 2 * warp;
    const int gx = blockIdx.x * TX - HX + c, gy0 = blockIdx.y * TY - H + r0;
    const int v = blockIdx.z / nzc;
    const int zs = (blockIdx.z - v * nzc) * zc, ze = min(nz, zs + zc);
    const int64_t plane = (int64_t)nx * ny;
    Din += v * fstride;
    Win += v * fstride;
    Dout += v * fstride;
    Wout += v * fstride;
    acc += v * plane * nz;

    // sources of the thread's 2 x 2 points: offsets within a plane and signs (0: a wall)
    const int bcx = axis_bc(st.bc, 0), bcy = axis_bc(st.bc, 1), bcz = axis_bc(st.bc, 2);
    int sxa = 1, sxb = 1;
    const int ixa = ext_axis<int>(gx, nx, bcx, sxa), ixb = ext_axis<int>(gx + 1, nx, bcx, sxb);
    const bool own_x = c >= HX && c < HX + TX && gx < nx, own_xb = own_x && gx + 1 < nx;
    unsigned srca[2], srcb[2];
    int sga[2], sgb[2];
    bool own[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        int sy = 1;
        const int iy = ext_axis<int>(gy0 + j, ny, bcy, sy);
        sga[j] = (ixa < 0 || iy < 0) ? 0 : sxa * sy;
        sgb[j] = (ixb < 0 || iy < 0) ? 0 : sxb * sy;
        srca[j] = sga[j] ? (unsigned)iy * (unsigned)nx + (unsigned)ixa : 0u;
        srcb[j] = sgb[j] ? (unsigned)iy * (unsigned)nx + (unsigned)ixb : 0u;
        own[j] = own_x && r0 + j >= H && r0 + j < H + TY && gy0 + j < ny;
    }
    // the filter sums' offsets (offset 0 for points that are not owned: loaded and not used)
    const unsigned o = (unsigned)gy0 * (unsigned)nx + (unsigned)gx;  // modulo 2^32: a rim row's is unused
    const unsigned a00 = own[0] ? o : 0u, a01 = own[0] && own_xb ? o + 1u : 0u;
    const unsigned a10 = own[1] ? o + (unsigned)nx : 0u, a11 = own[1] && own_xb ? o + (unsigned)nx + 1u : 0u;
    const bool flips = sga[0] < 0 || sga[1] < 0 || sgb[0] < 0 || sgb[1] < 0;
    const int me = r0 * kWX + c;  // this thread's first cell of a plane (row j: + j kWX)
    // neighbour pairs and rows, clamped at the region's edge (those values are wrong but stay in the rim)
    const int xm = max(c - 2, 0) - c, xp = min(c + 2, kWX - 2) - c;
    int up[R], dw[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
        up[q] = max(r0 - 1 - q, 0) * kWX + c;
        dw[q] = min(r0 + 2 + q, kWY - 1) * kWX + c;
    }

    // walls: 0 for good (no copy writes them)
    for (int q = 0; q < NW; ++q)
#pragma unroll
        for (int j = 0; j < 2; ++j) *reinterpret_cast<float2*>(sW + q * kWPlane + me + j * kWX) = make_float2(0.f, 0.f);

    const int zlo = zs - H, zhi = ze + H;
    // the plane of the box that holds plane z's values and its sign (-1: a wall plane)
    auto zsrc = [&](int z, int& sg) { return z >= 0 && z < nz ? z : ext_axis<int>(z, nz, bcz, sg); };
    // `fast`: a step whose planes all lie inside the box and the chunk (no z test)
    auto copy_w = [&](bool fast, int z, int slot) {  // plane z of W^n into a ring slot
        float* w = sW + slot * kWPlane + me;
        if (fast || z < zhi) {
            int sg = 1;
            const int iz = fast ? z : zsrc(z, sg);
            const float* p = Win + (int64_t)iz * plane;
            if (!fast && iz < 0) {
                *reinterpret_cast<float2*>(w) = *reinterpret_cast<float2*>(w + kWX) = make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    if (sga[j]) cp_async4(w + j * kWX, p + srca[j]);
                    if (sgb[j]) cp_async4(w + j * kWX + 1, p + srcb[j]);
                }
            }
        }
        cp_async_commit();
    };
    auto load_d = [&](bool fast, int z, float2 (&d)[2]) {  // plane z of D^n (a mirror's values unsigned)
        int iz = z;
        if (!fast) {
            d[0] = d[1] = make_float2(0.f, 0.f);
            if (z < zlo || z >= ze + H - R) return;
            int sg = 1;
            iz = zsrc(z, sg);
            if (iz < 0) return;
        }
        const float* p = Din + (int64_t)iz * plane;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            d[j].x = sga[j] ? p[srca[j]] : 0.f;
            d[j].y = sgb[j] ? p[srcb[j]] : 0.f;
        }
    };
    auto load_a = [&](bool fast, int z, float2 (&a)[2]) {  // the filter sums of plane z (only owned ones are used)
        if (!fast && (z < zs || z >= ze)) return;
        const float* p = acc + (int64_t)z * plane;
        a[0] = make_float2(p[a00], p[a01]);
        a[1] = make_float2(p[a10], p[a11]);
    };
    auto signs = [&](float2 (&x)[2], int sz) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (sga[j] * sz < 0) x[j].x = -x[j].x;
            if (sgb[j] * sz < 0) x[j].y = -x[j].y;
        }
    };

    constexpr int Q = 2 * R + 1;
    float2 Wq[B][Q][2];                  // Wq[k]: level k's planes around the one level k + 1 computes (a rotating queue)
    float2 Dq[B > 1 ? B - 1 : 1][R][2];  // Dq[k]: D of level k + 1, oldest first
    constexpr int NA = B == 2 ? 1 : R * (B - 1) + 1;
    float2 Aq[NA][2];                    // filter sums between level 1 and the last (B != 2)
    float2 CW[B];
#pragma unroll
    for (int k = 0; k < B; ++k) {
        CW[k] = make_float2(cw[k], cw[k]);
#pragma unroll
        for (int q = 0; q < Q; ++q) Wq[k][q][0] = Wq[k][q][1] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < (B > 1 ? B - 1 : 1); ++k)
#pragma unroll
        for (int q = 0; q < R; ++q) Dq[k][q][0] = Dq[k][q][1] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < NA; ++q) Aq[q][0] = Aq[q][1] = make_float2(0.f, 0.f);
    const float2 C0{st.c0, st.c0}, C1X{st.c1[0], st.c1[0]}, C1Y{st.c1[1], st.c1[1]}, C1Z{st.c1[2], st.c1[2]};
    const float2 C2X{st.c2[0], st.c2[0]}, C2Y{st.c2[1], st.c2[1]}, C2Z{st.c2[2], st.c2[2]};
    // the filter sum of plane z - LA is needed at step z
    constexpr int LA = B == 2 ? R * B : R;

#pragma unroll
    for (int q = 0; q < PF; ++q) copy_w(false, zlo + q, q);
    float2 dnx[2], anx[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};  // D^n and filter sums of the next step
    load_d(false, zlo - R, dnx);
    load_a(false, zlo - LA, anx);
    int ws = 0, ls = 0;  // ring slots of step z: W^n, levels
    // the queues of W rotate with the step (the loop is unrolled by their length) where the
    // filter-sum queue can rotate with them or is absent; else they are shifted
    constexpr bool turn = R == 2 || NA == Q;
    constexpr int U = turn ? Q : 1;
    constexpr bool rot = turn && NA == Q;
    // one plane; t = (z - zlo) mod Q: queue entry q is register (q + t + 1) mod Q
    auto step = [&](bool fast, int t, int z) {
        cp_async_wait_group<PF - 1>();  // this thread's copies of plane z have landed
        float2 wn[2], dn[2] = {dnx[0], dnx[1]}, an[2] = {anx[0], anx[1]};
        {
            float* p = sW + ws * kWPlane + me;
            wn[0] = *reinterpret_cast<const float2*>(p);
            wn[1] = *reinterpret_cast<const float2*>(p + kWX);
            if (fast ? flips : (flips || z < R || z >= nz)) {  // mirrors take their signs
                int sz = 1, szd = 1;
                if (!fast) {
                    zsrc(z, sz);
                    zsrc(z - R, szd);
                }
                signs(wn, sz);
                signs(dn, szd);
                *reinterpret_cast<float2*>(p) = wn[0];
                *reinterpret_cast<float2*>(p + kWX) = wn[1];
            }
        }
        {   // the copies of plane z + PF, into a slot last read in the previous step
            int w2 = ws + PF;
            if (w2 >= NW) w2 -= NW;
            copy_w(fast, z + PF, w2);
        }
        load_d(fast, z + 1 - R, dnx);
        load_a(fast, z + 1 - LA, anx);
        // level rings: slot ls is written in this step, slot ls + 1 (R steps old) is read
        const int lr = ls + 1 == NL ? 0 : ls + 1;
        int wr = ws - R;
        if (wr < 0) wr += NW;
        if (B != 2) {
            if constexpr (!rot) {
#pragma unroll
                for (int q = NA - 1; q > 0; --q) {
                    Aq[q][0] = Aq[q - 1][0];
                    Aq[q][1] = Aq[q - 1][1];
                }
            }
            const int e = rot ? (NA - 1 - t) % NA : 0;
            Aq[e][0] = an[0];
            Aq[e][1] = an[1];
        }
#pragma unroll
        for (int k = 1; k <= B; ++k) {
            const float* sq = k == 1 ? sW + wr * kWPlane : sL + ((k - 2) * NL + lr) * kWPlane;
            float2(&wq)[Q][2] = Wq[k - 1];
#define EW_Q(q) wq[turn ? ((q) + t + 1) % Q : (q)]
            if constexpr (!turn) {
#pragma unroll
                for (int q = 0; q < Q - 1; ++q) {
                    wq[q][0] = wq[q + 1][0];
                    wq[q][1] = wq[q + 1][1];
                }
            }
            EW_Q(Q - 1)[0] = wn[0];
            EW_Q(Q - 1)[1] = wn[1];
            const float2 u[2] = {EW_Q(R)[0], EW_Q(R)[1]};
            float2 ru[R], rd[R];
#pragma unroll
            for (int q = 0; q < R; ++q) {
                ru[q] = *reinterpret_cast<const float2*>(sq + up[q]);
                rd[q] = *reinterpret_cast<const float2*>(sq + dw[q]);
            }
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float2 sx1, lap;
                const float2 sy1 = j == 0 ? p_add(ru[0], u[1]) : p_add(u[0], rd[0]);
                const float2 sz1 = p_add(EW_Q(R - 1)[j], EW_Q(R + 1)[j]);
                if constexpr (R == 1) {  // the columns beside the pair come from the neighbouring lanes
                    sx1.x = s_add(__shfl_up_sync(0xffffffffu, u[j].y, 1), u[j].y);
                    sx1.y = s_add(u[j].x, __shfl_down_sync(0xffffffffu, u[j].x, 1));
                    lap = p_mul(C0, u[j]);
                    lap = p_fma(C1X, sx1, lap);
                    lap = p_fma(C1Y, sy1, lap);
                    lap = p_fma(C1Z, sz1, lap);
                } else {
                    const float2 L = *reinterpret_cast<const float2*>(sq + me + j * kWX + xm);
                    const float2 P = *reinterpret_cast<const float2*>(sq + me + j * kWX + xp);
                    sx1.x = s_add(L.y, u[j].y);
                    sx1.y = s_add(u[j].x, P.x);
                    lap = p_fma(C0, u[j], p_mul(C1X, sx1));
                    lap = p_fma(C1Y, sy1, lap);
                    lap = p_fma(C1Z, sz1, lap);
                    const float2 sy2 = j == 0 ? p_add(ru[R - 1], rd[0]) : p_add(ru[0], rd[R - 1]);
                    float2 l2 = p_fma(C2X, p_add(L, P), p_mul(C2Y, sy2));
                    l2 = p_fma(C2Z, p_add(EW_Q(0)[j], EW_Q(Q - 1)[j]), l2);
                    lap = p_add(lap, l2);
                }
                const float2 d = p_add(dn[j], lap);
                const float2 w = p_add(u[j], d);
                const int ae = rot ? (R * (k - 1) + 2 * NA - 1 - t) % NA : R * (k - 1);
                if (B != 2) Aq[ae][j] = p_fma(CW[k - 1], w, Aq[ae][j]);
                if (k < B) {
                    dn[j] = Dq[k - 1][0][j];
#pragma unroll
                    for (int q = 0; q < R - 1; ++q) Dq[k - 1][q][j] = Dq[k - 1][q + 1][j];
                    Dq[k - 1][R - 1][j] = d;
                    wn[j] = w;
                    *reinterpret_cast<float2*>(sL + ((k - 1) * NL + ls) * kWPlane + me + j * kWX) = w;
                } else {
                    float2 a;
                    if constexpr (B == 2)  // level 1's W of this plane is the centre of its queue
                        a = p_fma(CW[1], w, p_fma(CW[0], u[j], an[j]));
                    else
                        a = Aq[ae][j];
                    if (own[j] && (fast || z >= zs + H)) {
                        const int64_t at = (z - H) * plane + (o + (unsigned)(j * nx));
                        Wout[at] = w.x;
                        Dout[at] = d.x;
                        acc[at] = a.x;
                        if (own_xb) {
                            Wout[at + 1] = w.y;
                            Dout[at + 1] = d.y;
                            acc[at + 1] = a.y;
                        }
                    }
                }
            }
#undef EW_Q
        }
        ws = ws + 1 == NW ? 0 : ws + 1;
        ls = lr;
        __syncthreads();
    };
    // fast steps: stores valid, and planes z + PF (W^n), z + 1 - R (D^n), z + 1 - LA (sums) inside box and chunk
    const int f0 = zs + H, f1 = min(min(nz, zhi) - PF, ze + LA - 1);
    for (int zb = zlo; zb < zhi; zb += U) {
        if (zb >= f0 && zb + U <= f1) {
#pragma unroll
            for (int t = 0; t < U; ++t) step(true, t, zb + t);
        } else {
#pragma unroll
            for (int t = 0; t < U; ++t) {
                if (zb + t >= zhi) break;
                step(false, t, zb + t);
            }
        }
    }
    cp_async_wait_group<0>();
}

template <int R, int B>
static ew_status launch_wide(const GridGeom& g, const float* Din, const float* Win, float* Dout, float* Wout, float* acc,
                             const float* cw, const Stencil<float>& s, int nvec, int64_t fstride, cudaStream_t st) {
    using S = Tb3wShape<R, B>;
    auto kern = k_step_tb3d_wide<R, B>;
    EW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM));
    int dev = 0, nsm = 0;
    EW_CUDA_TRY(cudaGetDevice(&dev));
    EW_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int nx = (int)g.n[0], ny = (int)g.n[1], nz = (int)g.n[2];
    const int64_t tx = (nx + S::TX - 1) / S::TX, ty = (ny + S::TY - 1) / S::TY;
    // z chunks: the number of waves of CTAs (one an SM) times the planes of a chunk with its
    // lead-in and run-out (and about four planes of start-up), at its least
    int best = 1;
    int64_t best_cost = INT64_MAX;
    for (int c = 1; c <= std::min(nz, 64) && c * (int64_t)nvec <= 65535; ++c) {
        const int64_t zc = (nz + c - 1) / c, waves = (tx * ty * nvec * c + nsm - 1) / nsm;
        const int64_t cost = waves * (zc + 2 * S::H + 4);
        if (cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    const int zc = (nz + best - 1) / best, nzc = (nz + zc - 1) / zc;
    const dim3 grid((unsigned)tx, (unsigned)ty, (unsigned)(nvec * nzc));
    cudaEvent_t ev = fused_begin(st);
    kern<<<grid, kWThreads, S::SMEM, st>>>(nx, ny, nz, Din, Win, Dout, Wout, acc, cw, s, fstride, nzc, zc);
    EW_CUDA_TRY(cudaGetLastError());
    fused_end(ev, st, g.N * nvec, g.N * nvec * B);
    return EW_OK;
}

// Planes are addressed with 32-bit offsets.  Fourth order: a launch of two steps leads
// in over four planes, so one vector of a few planes goes to the one-step kernel
// (40 steps: 5^3 259 against 345 us here, 200 x 200 x 6 341 against 390, 800 x 600 x 6
// 1009 against 1472; from eight planes on this form wins, 200 x 200 x 8 390 against 422,
// and with several vectors, which it takes in one launch, 200 x 200 x 6, 4 vectors 560
// against 1393).
bool tb3d_wide_fits(const GridGeom& g, int nvec) {
    if (g.order == 4 && nvec == 1 && g.n[2] < 8) return false;
    return g.dim == 3 && g.n[0] * g.n[1] < INT32_MAX && g.n[1] <= 65535 * 20 && nvec <= 65535;
}

// b levels in one launch: a kernel of that depth
static ew_status launch_depth(int b, const GridGeom& g, const float* Din, const float* Win, float* Dout, float* Wout,
                              float* acc, const float* cw, const Stencil<float>& s, int nvec, int64_t fstride,
                              cudaStream_t st) {
#define EW_W(R, B) launch_wide<R, B>(g, Din, Win, Dout, Wout, acc, cw, s, nvec, fstride, st)
    if (g.order == 4) return b >= 2 ? EW_W(2, 2) : EW_W(2, 1);
    if (b >= 4) return EW_W(1, 4);
    if (b == 3) return EW_W(1, 3);
    return b == 2 ? EW_W(1, 2) : EW_W(1, 1);
#undef EW_W
}

// Second order, kNarrow + depth: the 32 x 32 regions of ew_tb3d.cu.  They can win
// where the 64 x 32 regions overhang the box by a fifth or more (27 x 463 x 132, 6
// vectors, 46 steps: 2.06 ms at depth 2 against 2.49 ms at the best depth of the wide
// ones) or the planes are few (not always: 374 x 122 x 30 455 against 366 us), so
// there the tuner times them too; without the tuner (a depth asked for) they take
// the boxes up to 32 points wide.
constexpr int kNarrow = 16;
static bool narrow_may_win(const GridGeom& g) {
    const double over = (double)((g.n[0] + 59) / 60 * 60) / g.n[0] * ((g.n[1] + 27) / 28 * 28) / g.n[1];
    return g.order == 2 && (over > 1.2 || g.n[2] < 64);
}
static ew_status launch_variant(int v, int b, const GridGeom& g, const float* Din, const float* Win, float* Dout,
                                float* Wout, float* acc, const float* cw, const Stencil<float>& s, int nvec,
                                int64_t fstride, cudaStream_t st) {
    if (v >= kNarrow) return tb3d_f2_step(v - kNarrow, g, Din, Win, Dout, Wout, acc, cw, b, s, nvec, fstride, st);
    return launch_depth(b, g, Din, Win, Dout, Wout, acc, cw, s, nvec, fstride, st);
}

// EW_TB3D_VARIANT=wide:d or narrow:d (d = 2, 3, 4) fixes the second-order variant
// instead of timing them, the 64 x 32 or the 32 x 32 regions at depth d: a tuning
// and testing override.  0: not set; EW_EINVAL for any other text
static ew_status forced_variant(int* v) {
    *v = 0;
    const char* e = getenv("EW_TB3D_VARIANT");
    if (!e) return EW_OK;
    const bool narrow = !strncmp(e, "narrow:", 7);
    const char* d = narrow ? e + 7 : !strncmp(e, "wide:", 5) ? e + 5 : "";
    if (d[0] < '2' || d[0] > '4' || d[1]) return set_error(EW_EINVAL, "EW_TB3D_VARIANT: wide:d or narrow:d, d = 2, 3, 4");
    *v = (narrow ? kNarrow : 0) + d[0] - '0';
    return EW_OK;
}

// depth autotuner (second order): times depths 2..4 on the caller's buffers
// (before the real wave-solve overwrites them) and caches the fastest per grid
// shape.  Fourth order: depth 2 (a rim of 4; depth 3 would leave 20 of 32 rows)
using Tb3dKey = std::tuple<int64_t, int64_t, int64_t, int, int>;  // nx, ny, nz, nvec, device
static std::map<Tb3dKey, int> g_tb3w_cache;
static std::mutex g_tb3w_mu;

ew_status tb3d_wide_tune(const GridGeom& g, const FilterPlan& plan, const float* cdev, float* const* F, float* acc,
                         int nvec, int64_t fstride, cudaStream_t st) {
    if (g.order != 2) return EW_OK;
    int dev = 0, forced = 0;
    EW_TRY(forced_variant(&forced));
    if (forced) return EW_OK;
    EW_CUDA_TRY(cudaGetDevice(&dev));
    Tb3dKey key{g.n[0], g.n[1], g.n[2], nvec, dev};
    {
        std::lock_guard<std::mutex> lk(g_tb3w_mu);
        if (g_tb3w_cache.count(key)) return EW_OK;
    }
    Stencil<float> s = make_stencil<float>(g, plan.dt * plan.dt);
    ProfilePause pause;  // tuning launches are not counted
    EventPair ev;
    EW_TRY(ev.create());
    int best = 3;
    double best_rate = -1.0;
    for (int v : {2, 3, 4, kNarrow + 2, kNarrow + 3, kNarrow + 4}) {
        const int B = v % kNarrow;
        if (v >= kNarrow && !narrow_may_win(g)) continue;
        for (int rep = 0; rep < 3; ++rep) {  // one warm launch, two timed
            if (rep == 1) EW_CUDA_TRY(cudaEventRecord(ev.a, st));
            EW_TRY(launch_variant(v, B, g, F[0], F[1], F[2], F[3], acc, cdev, s, nvec, fstride, st));
        }
        EW_CUDA_TRY(cudaEventRecord(ev.b, st));
        EW_CUDA_TRY(cudaEventSynchronize(ev.b));
        float ms = 0.f;
        EW_CUDA_TRY(cudaEventElapsedTime(&ms, ev.a, ev.b));
        const double rate = 2.0 * B / std::max(ms, 1e-6f);  // time steps per ms
        if (getenv("EW_TUNE_LOG"))
            fprintf(stderr, "[ew tune] %lldx%lldx%lld 3D order 2 fp32: depth %d%s: %.4f ms/step\n", (long long)g.n[0],
                    (long long)g.n[1], (long long)g.n[2], B, v >= kNarrow ? ", 32 x 32" : "", 1.0 / rate);
        if (rate > best_rate) {
            best_rate = rate;
            best = v;
        }
    }
    std::lock_guard<std::mutex> lk(g_tb3w_mu);
    g_tb3w_cache[key] = best;
    return EW_OK;
}

// Advance from level L (W = F[cur], D = F[prv]) to level Nt in launches of up
// to B levels (the tuned depth, or `tb` when tb > 1).
ew_status tb3d_wide_advance(const GridGeom& g, const FilterPlan& plan, const float* cdev, float* const* F, int* prv,
                            int* cur, int64_t L, float* acc, int nvec, int64_t fstride, int tb, cudaStream_t st) {
    if (nvec > 65535) return set_error(EW_EUNSUPPORTED, "too many vectors in one call");
    Stencil<float> s = make_stencil<float>(g, plan.dt * plan.dt);
    int B = g.order == 4 ? 2 : 4;
    if (tb > 1) {
        B = std::min(tb, B);
    } else if (g.order == 2) {
        int dev = 0, forced = 0;
        EW_CUDA_TRY(cudaGetDevice(&dev));
        EW_TRY(forced_variant(&forced));
        std::lock_guard<std::mutex> lk(g_tb3w_mu);
        auto it = g_tb3w_cache.find(Tb3dKey{g.n[0], g.n[1], g.n[2], nvec, dev});
        if (forced)
            B = forced;
        else if (it != g_tb3w_cache.end())
            B = it->second;
    }
    int v = 0;  // variant: below kNarrow the 64 x 32 regions
    if (B >= kNarrow) {
        v = B;
        B -= kNarrow;
    } else if (tb > 1 && g.order == 2 && g.n[0] <= 32) {
        v = kNarrow + B;
    }
    int p = *prv, c = *cur, a = -1, d = -1;
    for (int q = 0; q < 4; ++q)
        if (q != p && q != c) (a < 0 ? a : d) = q;
    while (L < plan.Nt) {
        const int b = (int)std::min<int64_t>(B, plan.Nt - L);
        EW_TRY(launch_variant(v, b, g, F[p], F[c], F[a], F[d], acc, cdev + L + 1, s, nvec, fstride, st));
        L += b;
        std::swap(p, a);
        std::swap(c, d);
    }
    *prv = p;
    *cur = c;
    return EW_OK;
}

}  // namespace ew
