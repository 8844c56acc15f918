// ew_mapped_tb.cu -- temporally blocked fused leapfrog + filter steps on a
// curvilinear grid, FP32 (eqs. explicitScheme, filterQuadrature with the
// conservative 9-point operator of ew_mapped.cu):
//
//   D^{n+1} = D^n + dt^2 / J (J L W^n),  W^{n+1} = W^n + D^{n+1},  acc += c W^{n+1}
//
// One launch advances every point by b <= B steps.  A CTA owns a TX x TY tile
// and stages the tile plus a halo of H = B points: D^n, W^n and the four
// coupling planes E, N, NE, SE, one TMA tensor load each, zeros outside the
// grid.  With zero couplings, centre and 1/J there, a point outside stays 0
// (the boundary vertices), so the step loop has no branch.  Each thread keeps
// D, the filter sum, the centre coupling and dt^2 / J of its column pair's KY
// rows in registers and slides windows of W, N, NE and SE along y; W^n and
// W^{n+1} alternate between two shared buffers (the second is the one D^n
// arrived in), one barrier a step.  The couplings stay staged for all vectors
// of a CTA.  The operations of a point and their order are those of
// k_mapped_step, so both give the same bits.
//
// Why: one step a launch moved 48 B a point and step (the couplings are half
// of it) and ran at 0.8 of the measured HBM bandwidth; b steps a launch move
// 48 / b.  Two CTAs of
// 64 x 64 points share an SM, so one's copies overlap the other's steps.
// Bound: shared-memory wavefronts (19 a warp and row of 64 points: about four
// points a clock and SM) and the copies.  128 registers a thread, 40 bytes spilled
// at depth 7, 20 at depth 5.  Measured, 2047^2, 415 steps: 17.0 ms
// (k_mapped_step, 102 Gcell-steps/s) -> 5.7 ms.
#include <algorithm>

#include "ew_internal.h"
#include "ew_tb2d_dev.cuh"
#include "ew_tma_dev.cuh"

namespace ew {

template <int NWX, int NTY, int KY, int B>
struct MappedTbShape {
    static constexpr int CWX = 64 * NWX, CWY = NTY * KY;  // compute region (two columns a lane)
    static constexpr int RX = CWX + 2, RY = CWY + 2;      // staged region
    static constexpr int H = B, TX = RX - 2 * H, TY = RY - 2 * H;
    static constexpr int O = (4 - H % 4) % 4;             // x0 mod 4 (x0 = TX t - H): the loads start at x0 - O
    static constexpr int BOXW = (RX + O + 3) & ~3;
    static constexpr int BUF = BOXW * RY, BUFP = (BUF + 31) & ~31;  // copy destinations 128-byte aligned
    static constexpr int NT = 32 * NWX * NTY;
    static constexpr size_t SMEM = sizeof(float) * 6 * (size_t)BUFP + 16;
    static_assert(H % 2 == 1 && TX % 4 == 0 && TX > 0 && TY > 0, "column pairs and loads stay aligned");
    static_assert(BOXW <= 256 && RY <= 256, "tensor-map box dimensions are at most 256");
};

template <int NWX, int NTY, int KY, int B>
__global__ void __launch_bounds__(32 * NWX * NTY, 512 / (32 * NWX * NTY))
    k_step_mapped_tb(const __grid_constant__ CUtensorMap mapD, const __grid_constant__ CUtensorMap mapW,
                     const __grid_constant__ CUtensorMap mapC, int nx, int ny, int pitch,
                     const float* __restrict__ coef, float* __restrict__ Dout, float* __restrict__ Wout,
                     float* __restrict__ acc, const float* __restrict__ cw, int b, float dt2, int nvec, int vpc,
                     int64_t fstride, int* gave_up) {
    using S = MappedTbShape<NWX, NTY, KY, B>;
    constexpr int H = S::H, TX = S::TX, TY = S::TY, O = S::O, P = S::BOXW, BUFP = S::BUFP;
    extern __shared__ __align__(128) unsigned char smem_mt[];
    float* sD = reinterpret_cast<float*>(smem_mt);
    float* sW = sD + BUFP;
    const float *sE = sW + BUFP, *sN = sE + BUFP, *sNE = sN + BUFP, *sSE = sNE + BUFP;
    uint64_t* bar = reinterpret_cast<uint64_t*>(sD + 6 * BUFP);  // [0]: couplings, [1]: fields
    const int tid = threadIdx.x, lane = tid & 31;
    const int wx = (tid >> 5) % NWX, ty = (tid >> 5) / NWX;
    const int x0 = blockIdx.x * TX - H, y0 = blockIdx.y * TY - H;
    const int v0 = blockIdx.z * vpc, v1 = min(nvec, v0 + vpc);
    const int64_t N = (int64_t)nx * ny, plane = (int64_t)pitch * ny;
    if (tid == 0) {
        tma_mbar_init(&bar[0], 1);
        tma_mbar_init(&bar[1], 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        tma_mbar_arrive_expect(&bar[0], 4u * S::BUF * 4u);
        for (int q = 0; q < 4; ++q) tma_load_3d(sD + (2 + q) * BUFP, &mapC, x0 - O, y0, q, &bar[0]);
    }
    __syncthreads();
    const int sx = 1 + 2 * (32 * wx + lane), sy0 = 1 + ty * KY;  // staged column of the pair, first staged row
    const int cx = sx + O;                                       // its shared-memory column (even)
    const int gx = x0 + sx, gy0 = y0 + sy0;
    const bool in_x = gx >= 0 && gx < nx;  // gx is even: the pair's second column is inside or a pad column
    const bool own_x = in_x && sx >= H && sx < H + TX, own_b = own_x && gx + 1 < nx;
    const int klo = max(0, H - sy0), khi = min(min(KY, H + TY - sy0), ny - gy0);
    // centre coupling and dt^2 / J of the thread's points (0 outside: those points stay 0)
    float2 cc[KY], tj[KY];
#pragma unroll
    for (int k = 0; k < KY; ++k) {
        cc[k] = tj[k] = make_float2(0.f, 0.f);
        const int gy = gy0 + k;
        if (in_x && gy >= 0 && gy < ny) {
            const float* c = coef + 4 * plane + (int64_t)gy * pitch + gx;
            cc[k] = *reinterpret_cast<const float2*>(c);
            const float2 rj = *reinterpret_cast<const float2*>(c + plane);
            tj[k] = p_mul(make_float2(dt2, dt2), rj);
        }
    }
    bool ok = true;
    for (int v = v0; v < v1; ++v) {
        if (tid == 0) {
            tma_mbar_arrive_expect(&bar[1], 2u * S::BUF * 4u);
            tma_load_3d(sD, &mapD, x0 - O, y0, v, &bar[1]);
            tma_load_3d(sW, &mapW, x0 - O, y0, v, &bar[1]);
        }
        // the filter sums load while the copies arrive
        float2 accp[KY];
        const int64_t ab = (int64_t)v * N + (int64_t)gy0 * nx + gx;
#pragma unroll
        for (int k = 0; k < KY; ++k) {
            const bool oy = k >= klo && k < khi;
            accp[k].x = (own_x && oy) ? acc[ab + (int64_t)k * nx] : 0.f;
            accp[k].y = (own_b && oy) ? acc[ab + (int64_t)k * nx + 1] : 0.f;
        }
        if (v == v0) ok = tma_mbar_wait_bounded(&bar[0], 0u);
        ok = tma_mbar_wait_bounded(&bar[1], (unsigned)(v - v0) & 1u) && ok;
        if (__syncthreads_or(!ok)) {
            if (tid == 0) *(volatile int*)gave_up = 1;
            // no copy may outlive the CTA: give those in flight another bounded chance
            tma_mbar_wait_bounded(&bar[0], 0u);
            tma_mbar_wait_bounded(&bar[1], (unsigned)(v - v0) & 1u);
            return;
        }
        float2 dd[KY];
#pragma unroll
        for (int k = 0; k < KY; ++k) dd[k] = *reinterpret_cast<const float2*>(sD + (sy0 + k) * P + cx);
        float* cur = sW;
        float* nxt = sD;  // each entry of D^n is read above only by the thread that overwrites it
        for (int s = 0; s < b; ++s) {
            const bool last = s == b - 1;
            const float cs = cw[s];
            const float2 CS{cs, cs};
            // rows y - 1, y of W as columns (x - 1, x), (x, x + 1), (x + 1, x + 2)
            auto row = [&](const float* p, float2& l, float2& c, float2& r) {
                const float2 a = *reinterpret_cast<const float2*>(p - 2), q = *reinterpret_cast<const float2*>(p + 2);
                c = *reinterpret_cast<const float2*>(p);
                l = make_float2(a.y, c.x);
                r = make_float2(c.y, q.x);
            };
            float2 ml, mc, mr, ul, uc, ur;
            const int q0 = sy0 * P + cx;
            row(cur + q0 - P, ml, mc, mr);
            row(cur + q0, ul, uc, ur);
            float2 ns = *reinterpret_cast<const float2*>(sN + q0 - P);              // N of row y - 1
            const float2 ne0 = *reinterpret_cast<const float2*>(sNE + q0 - P);
            float2 nesw = make_float2(sNE[q0 - P - 1], ne0.x);                      // NE at (x - 1, y - 1)
            float2 se = *reinterpret_cast<const float2*>(sSE + q0);                 // SE of row y
#pragma unroll
            for (int k = 0; k < KY; ++k) {
                const int q = q0 + k * P;
                float2 nl, nc, nr;
                row(cur + q + P, nl, nc, nr);
                const float2 e = *reinterpret_cast<const float2*>(sE + q);
                const float2 ew = make_float2(sE[q - 1], e.x);
                const float2 n = *reinterpret_cast<const float2*>(sN + q);
                const float2 ne = *reinterpret_cast<const float2*>(sNE + q);
                const float nel = sNE[q - 1];
                const float2 sep = *reinterpret_cast<const float2*>(sSE + q + P);
                const float2 senw = make_float2(sSE[q + P - 1], sep.x);             // SE at (x - 1, y + 1)
                float2 r = p_mul(cc[k], uc);
                r = p_fma(e, ur, r);
                r = p_fma(ew, ul, r);
                r = p_fma(n, nc, r);
                r = p_fma(ns, mc, r);
                r = p_fma(ne, nr, r);
                r = p_fma(nesw, ml, r);
                r = p_fma(se, mr, r);
                r = p_fma(senw, nl, r);
                const float2 d = p_fma(tj[k], r, dd[k]);
                const float2 nv = p_add(uc, d);
                dd[k] = d;
                accp[k] = p_fma(CS, nv, accp[k]);
                if (!last) {
                    *reinterpret_cast<float2*>(nxt + q) = nv;
                } else if (own_x && k >= klo && k < khi) {
                    const int64_t f = (int64_t)v * fstride + (int64_t)(gy0 + k) * pitch + gx;
                    *reinterpret_cast<float2*>(Wout + f) = nv;
                }
                ml = ul, mc = uc, mr = ur;
                ul = nl, uc = nc, ur = nr;
                ns = n;
                nesw = make_float2(nel, ne.x);
                se = sep;
            }
            __syncthreads();
            float* t = cur;
            cur = nxt;
            nxt = t;
        }
        // the next vector's copies overwrite what the last step read
        if (v + 1 < v1) fence_async_smem();
#pragma unroll
        for (int k = 0; k < KY; ++k)
            if (own_x && k >= klo && k < khi) {
                const int64_t f = (int64_t)v * fstride + (int64_t)(gy0 + k) * pitch + gx;
                *reinterpret_cast<float2*>(Dout + f) = dd[k];
                acc[ab + (int64_t)k * nx] = accp[k].x;
                if (own_b) acc[ab + (int64_t)k * nx + 1] = accp[k].y;
            }
        if (v + 1 < v1) __syncthreads();  // every thread's fence precedes the next copies
    }
}

// vectors a CTA: as many as leave four waves of CTAs (two an SM), so that the
// couplings are staged once for them
static int vectors_per_cta(int nvec, int64_t tiles, int nsm) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(nvec, nvec * tiles / (4 * 2 * (int64_t)nsm)));
}

template <int B>
static ew_status advance(const GridGeom& g, const FilterPlan& plan, const float* c, const float* cdev, float* const* F,
                         float* acc, int nvec, int64_t fstride, float dt2, int nsm, cudaStream_t st) {
    using S = MappedTbShape<1, 8, 8, B>;
    auto kern = k_step_mapped_tb<1, 8, 8, B>;
    EW_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM));
    const int nx = (int)g.n[0], ny = (int)g.n[1], pitch = (int)pitch2d(g.n[0]);
    const int64_t tx = (nx + S::TX - 1) / S::TX, ty = (ny + S::TY - 1) / S::TY;
    if (ty > 65535) return set_error(EW_EUNSUPPORTED, "mapped grid: too many rows of tiles");
    const int vpc = vectors_per_cta(nvec, tx * ty, nsm);
    const dim3 grid((unsigned)tx, (unsigned)ty, (unsigned)((nvec + vpc - 1) / vpc));
    CUtensorMap mC, mF[4];
    EW_TRY(field_map(c, nx, ny, pitch, 4, (int64_t)pitch * ny, S::BOXW, S::RY, &mC));
    for (int q = 0; q < 4; ++q) EW_TRY(field_map(F[q], nx, ny, pitch, nvec, fstride, S::BOXW, S::RY, &mF[q]));
    int p = 0, w = 1, a = 2, d = 3;
    for (int64_t L = 1; L < plan.Nt;) {
        const int b = (int)std::min<int64_t>(B, plan.Nt - L);
        cudaEvent_t ev = fused_begin(st);
        kern<<<grid, S::NT, S::SMEM, st>>>(mF[p], mF[w], mC, nx, ny, pitch, c, F[a], F[d], acc, cdev + L + 1, b, dt2,
                                           nvec, vpc, fstride, g.gave_up);
        EW_CUDA_TRY(cudaGetLastError());
        fused_end(ev, st, g.N * nvec, g.N * nvec * b);
        L += b;
        std::swap(p, a);
        std::swap(w, d);
    }
    return EW_OK;
}

ew_status mapped_advance(const GridGeom& g, const FilterPlan& plan, const float* c, const float* cdev, float* const* F,
                         float* acc, int nvec, int64_t fstride, float dt2, cudaStream_t st) {
    // Depth 7 (tile 52 x 52) moves the fewest bytes a step and is the faster one wherever a CTA
    // stages the couplings for one vector; where it keeps them for several, the fields' share is
    // smaller and the depth-5 tile's (56 x 56) fewer halo points win (2047^2, 4 vectors, 1000 steps:
    // 42.8 against 46.1 ms; 1 vector: 14.3 against 13.7 ms).  Depth 3 and a 128 x 64 region a CTA of
    // 16 warps (one CTA an SM, nothing to overlap its copies with) were slower at every size.
    if (!g.gave_up) return set_error(EW_EINVAL, "blocked curvilinear step: the grid has no word for waits that give up");
    using S5 = MappedTbShape<1, 8, 8, 5>;
    int dev = 0, nsm = 0;
    EW_CUDA_TRY(cudaGetDevice(&dev));
    EW_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int64_t t5 = ((g.n[0] + S5::TX - 1) / S5::TX) * ((g.n[1] + S5::TY - 1) / S5::TY);
    if (vectors_per_cta(nvec, t5, nsm) > 1) return advance<5>(g, plan, c, cdev, F, acc, nvec, fstride, dt2, nsm, st);
    return advance<7>(g, plan, c, cdev, F, acc, nvec, fstride, dt2, nsm, st);
}

}  // namespace ew
