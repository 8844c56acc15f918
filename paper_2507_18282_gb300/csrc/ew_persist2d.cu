// ew_persist2d.cu -- steps 2 .. N_t of an explicit FP32 wave-solve on 2D boxes
// whose vectors fit on the chip, in one cooperative launch (eqs.
// explicitScheme, filterQuadrature; the summed form of ew_stencil.cu).
//
// Every CTA owns one tile of one vector for the whole solve: W^n alternates
// between two shared-memory buffers, D^n = W^n - W^{n-1} and the filter sums of
// a thread's column pair and KY rows stay in its registers.  The tile carries
// a halo of H = R B points, as in the blocked kernels (ew_tb2d_dev.cuh): after
// B steps without communication the owned points are still exact, and the CTA
// exchanges: it publishes the points of its tile that its neighbours' halos
// need (H + 1 deep), then reads its own halo, with the box closure's extension
// for points outside the box.
//
// A published value is one 8-byte record of its bits and the number of the
// exchange, written and read as a single 64-bit access, so a reader that finds
// the number has the value: no fence, no flag and no barrier between CTAs, one
// trip through L2.  (Fields, a fence and a flag a tile took 3.0-3.7 us an
// exchange.)  The records of consecutive exchanges go to two
// buffers in turn: a CTA overwrites a buffer only after it has read, from every
// tile around it, records of the exchange in between, which those tiles
// published after they had read this buffer.  The buffers are cleared before
// the launch (exchanges count from 1).
//
// The CTAs of a launch wait for one another, so the launch is cooperative (all
// are resident, or it fails).  Every wait is bounded (about two seconds of SM
// clock); a CTA that gives up records it in the grid's flag (EW_ETIMEOUT at the
// next synchronising call) and leaves; the others' waits run out too.
//
// The operations of a point and their order are those of tb2d_tile: the same
// bits as the blocked kernels.
//
// Registers: 64 a thread at 1024 threads an SM; the shapes spill 20 to 64 bytes a
// thread, those of six rows (128 x 96 regions) 128, mostly values of the exchange.
//
// Why: up to about 800,000 points of all vectors the blocked kernels' tiles do
// not fill the SMs, and each launch stages its tiles anew for eight steps at
// most: 26 us a launch of eight steps, whatever the grid.  Bound: latency of a
// step (shared-memory reads, then arithmetic, then a barrier) and of the
// exchanges (2 us each at 64 x 64 points).  Measured, 400 steps, order 4: 300 x
// 250 1300 -> 455 us, 383 x 319 with 4 vectors 1358 -> 865 us, 517 x 389 with 4
// vectors and a Neumann face 1661 -> 1015 us.
#include <stdlib.h>

#include <algorithm>
#include <vector>

#include "ew_bc_dev.cuh"
#include "ew_internal.h"
#include "ew_tb2d_dev.cuh"

namespace ew {

template <int R, int NWX, int NTY, int KY, int B>
struct PersistShape {
    static constexpr int CWX = 64 * NWX, CWY = NTY * KY;      // compute region
    static constexpr int RX = CWX + 2 * R, RY = CWY + 2 * R;  // staged region
    static constexpr int OFF = R & 1, PX = RX + 2 * OFF;      // column pairs start on an even index
    static constexpr int H = R * B, TX = RX - 2 * H, TY = RY - 2 * H;
    static constexpr int NT = 32 * NWX * NTY;
    static constexpr size_t SMEM = sizeof(float) * 2 * (size_t)PX * RY;
    static_assert(TX > 0 && TY > 0, "halo too large for the tile");
};

// a record: a value's bits below, the exchange's number above
__device__ __forceinline__ void publish(unsigned long long* r, float v, int e) {
    const unsigned long long x = ((unsigned long long)(unsigned)e << 32) | __float_as_uint(v);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;\n" ::"l"(r), "l"(x) : "memory");
}
__device__ __forceinline__ unsigned long long peek(const unsigned long long* r) {
    unsigned long long x;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(x) : "l"(r) : "memory");
    return x;
}

// MINB: CTAs an SM the register budget is sized for
template <int R, int NWX, int NTY, int KY, int B, int MINB>
__global__ void __launch_bounds__(32 * NWX * NTY, MINB)
    k_persist2d(int nx, int ny, const float* __restrict__ Din, const float* __restrict__ Win, float* __restrict__ acc,
                const float* __restrict__ cw, int64_t Nt, Stencil<float> st, int ntx, int nty, int64_t fstride,
                unsigned long long* rec, int stall, int* gave_up) {
    using S = PersistShape<R, NWX, NTY, KY, B>;
    constexpr int RX = S::RX, RY = S::RY, PX = S::PX, OFF = S::OFF, H = S::H, NT = S::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float* nxt = reinterpret_cast<float*>(smem_raw);  // D^n at staging, then the level being written
    float* cur = nxt + PX * RY;                       // W^n
    const int tid = threadIdx.x;
    const int per = ntx * nty, tv = blockIdx.x % per, v = blockIdx.x / per;
    const int tx = tv % ntx, ty_ = tv / ntx;
    // owned tile [xs, xs + w) x [ys, ys + h): the axes cut into even shares
    const int xs = (int)((int64_t)nx * tx / ntx), w = (int)((int64_t)nx * (tx + 1) / ntx) - xs;
    const int ys = (int)((int64_t)ny * ty_ / nty), h = (int)((int64_t)ny * (ty_ + 1) / nty) - ys;
    const int x0 = xs - H, y0 = ys - H;
    const int64_t N = (int64_t)nx * ny;
    acc += v * N;
    Din += v * fstride;
    Win += v * fstride;
    rec += 4 * N * v;  // [buffer][point][W, D]
    const int bcx = axis_bc(st.bc, 0), bcy = axis_bc(st.bc, 1);
    const int wr = w + 2 * H, hr = h + 2 * H;  // the part of the staged region that matters

    // the active point holding cell (sx, sy) of the staged region (-1: a wall) and its sign
    auto source = [&](int sx, int sy, int& sg) -> int64_t {
        int sgx = 1, sgy = 1;
        const int gx = x0 + sx, gy = y0 + sy;
        const int ix = gx >= 0 && gx < nx ? gx : ext_axis<int>(gx, nx, bcx, sgx);
        const int iy = gy >= 0 && gy < ny ? gy : ext_axis<int>(gy, ny, bcy, sgy);
        sg = sgx * sgy;
        return ix < 0 || iy < 0 ? -1 : (int64_t)iy * nx + ix;
    };
    for (int q = tid; q < RX * RY; q += NT) {
        const int sy = q / RX, sx = q - sy * RX;
        float d = 0.f, u = 0.f;
        if (sx < wr && sy < hr) {
            int sg = 1;
            const int64_t g = source(sx, sy, sg);
            if (g >= 0) {
                d = sg < 0 ? -Din[g] : Din[g];
                u = sg < 0 ? -Win[g] : Win[g];
            }
        }
        nxt[sy * PX + sx + OFF] = d;
        cur[sy * PX + sx + OFF] = u;
    }

    const int lane = tid & 31;
    const int wx = (tid >> 5) % NWX, ty = (tid >> 5) / NWX;
    const int sx = R + 2 * (32 * wx + lane);  // first of the thread's two staged columns
    const int cx = sx + OFF;                  // its shared-memory column (even)
    const int sy0 = R + ty * KY;              // first staged row of its segment
    const bool own_a = sx >= H && sx < H + w, own_b = sx + 1 >= H && sx + 1 < H + w;
    const int klo = max(0, H - sy0), khi = min(KY, H + h - sy0);
    const int64_t gbase = (int64_t)(y0 + sy0) * nx + x0 + sx;
    float2 accp[KY];
#pragma unroll
    for (int k = 0; k < KY; ++k) {
        const bool oy = k >= klo && k < khi;
        accp[k].x = (own_a && oy) ? acc[gbase + (int64_t)k * nx] : 0.f;
        accp[k].y = (own_b && oy) ? acc[gbase + (int64_t)k * nx + 1] : 0.f;
    }
    __syncthreads();
    float2 dd[KY];
#pragma unroll
    for (int k = 0; k < KY; ++k) dd[k] = *reinterpret_cast<const float2*>(nxt + (sy0 + k) * PX + cx);

    const float2 C0{st.c0, st.c0}, C1X{st.c1[0], st.c1[0]}, C1Y{st.c1[1], st.c1[1]};
    const float2 C2X{st.c2[0], st.c2[0]}, C2Y{st.c2[1], st.c2[1]};
    // the thread's columns lie in the ring that neighbours read (or in any ring row)
    const bool ring_xa = sx - H < H + 1 || sx - H >= w - (H + 1), ring_xb = sx + 1 - H < H + 1 || sx + 1 - H >= w - (H + 1);
    int e = 0;
    for (int64_t L = 1;;) {
        const int b = (int)min((int64_t)B, Nt - L);
        for (int s = 0; s < b; ++s) {
            const float* col = cur + cx;
            float2 w0 = R == 2 ? *reinterpret_cast<const float2*>(col + (sy0 - 2) * PX) : float2{0.f, 0.f};
            float2 w1 = *reinterpret_cast<const float2*>(col + (sy0 - 1) * PX);
            float2 w2 = *reinterpret_cast<const float2*>(col + sy0 * PX);
            float2 w3 = *reinterpret_cast<const float2*>(col + (sy0 + 1) * PX);
            const float cs = cw[L + 1 + s];
            const float2 CS{cs, cs};
#pragma unroll
            for (int k = 0; k < KY; ++k) {
                const int row = (sy0 + k) * PX + cx;
                const float2 w4 = (R == 2 || k + 1 < KY) ? *reinterpret_cast<const float2*>(col + (sy0 + k + 2) * PX)
                                                         : float2{0.f, 0.f};
                const float2 Lf = *reinterpret_cast<const float2*>(cur + row - 2);  // columns x-2, x-1
                const float2 Rt = *reinterpret_cast<const float2*>(cur + row + 2);  // columns x+2, x+3
                float2 sx1;
                sx1.x = s_add(Lf.y, w2.y);
                sx1.y = s_add(w2.x, Rt.x);
                float2 lap = p_mul(C0, w2);
                lap = p_fma(C1X, sx1, lap);
                lap = p_fma(C1Y, p_add(w1, w3), lap);
                if (R == 2) {
                    lap = p_fma(C2X, p_add(Lf, Rt), lap);
                    lap = p_fma(C2Y, p_add(w0, w4), lap);
                }
                const float2 d = p_add(dd[k], lap);
                const float2 nv = p_add(w2, d);
                *reinterpret_cast<float2*>(nxt + row) = nv;
                dd[k] = d;
                accp[k] = p_fma(CS, nv, accp[k]);
                w0 = w1;
                w1 = w2;
                w2 = w3;
                w3 = w4;
            }
            __syncthreads();
            float* t = cur;
            cur = nxt;
            nxt = t;
        }
        L += b;
        if (L >= Nt) break;

        // ---- exchange e: my ring out, my halo in ----------------------------------
        ++e;
        unsigned long long* const buf = rec + (e & 1) * 2 * N;
#pragma unroll
        for (int k = 0; k < KY; ++k) {
            if (k < klo || k >= khi || (stall && blockIdx.x == 0)) continue;
            const int oy = sy0 + k - H;
            const bool ry = oy < H + 1 || oy >= h - (H + 1);
            const bool pa = own_a && (ry || ring_xa), pb = own_b && (ry || ring_xb);
            if (!pa && !pb) continue;
            const float2 u = *reinterpret_cast<const float2*>(cur + (sy0 + k) * PX + cx);
            unsigned long long* r = buf + 2 * (gbase + (int64_t)k * nx);
            if (pa) {
                publish(r, u.x, e);
                publish(r + 1, dd[k].x, e);
            }
            if (pb) {
                publish(r + 2, u.y, e);
                publish(r + 3, dd[k].y, e);
            }
        }
        // halo cells: the rows above and below the tile, then the columns beside it, a few a
        // thread at a time so that their reads overlap
        const int top = H * wr, ncell = 2 * top + 2 * H * h;
        bool ok = true;
        constexpr int M = 4;
        for (int q0 = tid; q0 < ncell; q0 += M * NT) {
            const unsigned long long* r[M];
            int cell[M];
            bool neg[M];
            unsigned long long a[M], d[M];
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const int q = q0 + m * NT;
                cell[m] = -1;
                r[m] = buf;
                neg[m] = false;
                if (q < ncell) {
                    int sxx, syy, sg = 1;
                    if (q < 2 * top) {
                        const int rr = q / wr;
                        sxx = q - rr * wr;
                        syy = rr < H ? rr : rr + h;
                    } else {
                        const int p = q - 2 * top, rr = p / (2 * H), cc = p - rr * 2 * H;
                        sxx = cc < H ? cc : cc + w;
                        syy = H + rr;
                    }
                    const int64_t g = source(sxx, syy, sg);
                    const int c = syy * PX + sxx + OFF;
                    if (g >= 0) {
                        cell[m] = c;
                        r[m] = buf + 2 * g;
                        neg[m] = sg < 0;
                    } else {
                        cur[c] = nxt[c] = 0.f;  // a wall
                    }
                }
            }
#pragma unroll
            for (int m = 0; m < M; ++m)
                if (cell[m] >= 0) {
                    a[m] = peek(r[m]);
                    d[m] = peek(r[m] + 1);
                }
#pragma unroll
            for (int m = 0; m < M; ++m)
                if (cell[m] >= 0) {
                    if (ok && ((int)(a[m] >> 32) != e || (int)(d[m] >> 32) != e)) {
                        const long long t0 = clock64();
                        ok = false;
                        for (int it = 0; it < (1 << 26) && !ok; ++it) {
                            a[m] = peek(r[m]);
                            d[m] = peek(r[m] + 1);
                            ok = (int)(a[m] >> 32) == e && (int)(d[m] >> 32) == e;
                            if (clock64() - t0 > 4000000000ll) break;
                        }
                    }
                    const float u = __uint_as_float((unsigned)a[m]), dv = __uint_as_float((unsigned)d[m]);
                    cur[cell[m]] = neg[m] ? -u : u;
                    nxt[cell[m]] = neg[m] ? -dv : dv;
                }
        }
        if (__syncthreads_or(!ok)) {
            if (tid == 0) *(volatile int*)gave_up = 1;
            return;
        }
        // D of the thread's points outside the tile (cells past the halo keep what they hold:
        // they are too far from the tile to reach it within B steps)
#pragma unroll
        for (int k = 0; k < KY; ++k) {
            const int sy = sy0 + k;
            const bool oy = k >= klo && k < khi;
            if (sy < hr) {
                if (!(oy && own_a) && sx < wr) dd[k].x = nxt[sy * PX + cx];
                if (!(oy && own_b) && sx + 1 < wr) dd[k].y = nxt[sy * PX + cx + 1];
            }
        }
        // the step loop's first write to nxt is to the thread's own cells, read above
    }
#pragma unroll
    for (int k = 0; k < KY; ++k) {
        if (k >= klo && k < khi) {
            if (own_a) acc[gbase + (int64_t)k * nx] = accp[k].x;
            if (own_b) acc[gbase + (int64_t)k * nx + 1] = accp[k].y;
        }
    }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct PersistVariant {
    void* fn;
    int R, TX, TY, H, threads, per_sm;
    size_t smem;
    double us[2];  // time of a step with one and with two CTAs an SM
    const char* name;
};
#define EW_PERSIST(R, NWX, NTY, KY, B, MINB, US1, US2)                                                               \
    PersistVariant {                                                                                                \
        (void*)k_persist2d<R, NWX, NTY, KY, B, MINB>, R, PersistShape<R, NWX, NTY, KY, B>::TX,                      \
            PersistShape<R, NWX, NTY, KY, B>::TY, PersistShape<R, NWX, NTY, KY, B>::H,                              \
            PersistShape<R, NWX, NTY, KY, B>::NT, MINB, PersistShape<R, NWX, NTY, KY, B>::SMEM, { US1, US2 },       \
            "k_persist2d<" #R ", " #NWX ", " #NTY ", " #KY ", " #B ", " #MINB ">"                                    \
    }
// Times measured over 400 steps, exchanges included.  A step's time is mostly
// latency (a region of 64 x 32 points takes 0.6 us, 128 x 64 points 1.4 us), so
// each grid takes the smallest region that its tiles fit the SMs with.
static const std::vector<PersistVariant>& persist_variants() {
    static const std::vector<PersistVariant> v = {
        EW_PERSIST(2, 1, 16, 2, 4, 2, 1.13, 1.58), EW_PERSIST(2, 1, 32, 2, 4, 1, 1.44, 0.0),
        EW_PERSIST(2, 1, 16, 4, 3, 2, 1.88, 2.90), EW_PERSIST(2, 1, 16, 4, 4, 2, 1.63, 2.45),
        EW_PERSIST(2, 2, 16, 4, 3, 1, 2.45, 0.0),  EW_PERSIST(2, 2, 16, 4, 4, 1, 2.18, 0.0),
        EW_PERSIST(2, 2, 16, 6, 4, 1, 3.12, 0.0),  EW_PERSIST(1, 1, 16, 2, 8, 2, 0.71, 0.95),
        EW_PERSIST(1, 1, 32, 2, 8, 1, 0.92, 0.0),  EW_PERSIST(1, 1, 16, 4, 6, 2, 1.13, 1.71),
        EW_PERSIST(1, 1, 16, 4, 8, 2, 1.04, 1.53), EW_PERSIST(1, 2, 16, 4, 5, 1, 1.64, 0.0),
        EW_PERSIST(1, 2, 16, 4, 8, 1, 1.37, 0.0),  EW_PERSIST(1, 2, 16, 6, 8, 1, 2.03, 0.0)};
    return v;
}

struct PersistPlan {
    const PersistVariant* v = nullptr;
    int ntx = 0, nty = 0;  // tiles of a vector
    double us = 1e30;      // time of a step
};

static PersistPlan persist_plan(const GridGeom& g, int nvec, int nsm) {
    PersistPlan best;
    const int R = g.order == 2 ? 1 : 2;
    for (const PersistVariant& v : persist_variants()) {
        if (v.R != R) continue;
        const int64_t ntx = (g.n[0] + v.TX - 1) / v.TX, nty = (g.n[1] + v.TY - 1) / v.TY;
        if (ntx > 4096 || nty > 4096 || ntx * nty * nvec > (int64_t)nsm * v.per_sm) continue;
        // every source of a halo cell lies in an adjacent tile
        if ((ntx > 1 && g.n[0] / ntx < v.H + 2) || (nty > 1 && g.n[1] / nty < v.H + 2)) continue;
        const double us = v.us[ntx * nty * nvec > nsm ? 1 : 0];
        if (us < best.us) {
            best.v = &v;
            best.ntx = (int)ntx;
            best.nty = (int)nty;
            best.us = us;
        }
    }
    return best;
}

static int sm_count() {
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nsm;
}

// All vectors of the call fit the chip at once, and the solve is faster than on
// the blocked kernels, whose step does not fall below 3.3 us (order 4; 3.7 us with
// Neumann faces) or 2.8 us (order 2) however small the grid (measured 300 x 250 ...
// 1600 x 700).  The largest order-4 regions take 3.12 us a step and 25 us a solve, so
// with Dirichlet faces they pay only from about 200 steps (blocked against here: 446 x
// 754, 4 vectors, 40 steps 155 and 164 us; 422 x 1364, 2 vectors, 100 steps 334 and 348
// us; 1657 x 700, 240 steps 821 and 809 us; with a Neumann face 340 x 567, 6 vectors,
// 100 steps 441 and 356 us).
bool persist2d_fits(const GridGeom& g, int nvec, int64_t Nt) {
    if (g.dim != 2 || g.map) return false;
    const double most = g.order == 2 ? 2.05 : g.bc != 0 || Nt >= 200 ? 3.2 : 3.0;
    return persist_plan(g, nvec, sm_count()).us <= most;
}

OnChipForm persist2d_form(const GridGeom& g, int nvec) {
    const PersistPlan p = persist_plan(g, nvec, sm_count());
    if (!p.v) return OnChipForm{"", 0, 0, 0};
    return OnChipForm{p.v->name, p.v->H / p.v->R, (int)((g.n[0] + p.ntx - 1) / p.ntx), (int)((g.n[1] + p.nty - 1) / p.nty)};
}

// bytes of the exchange records, which follow the time-level fields
size_t persist2d_room(const GridGeom& g, int nvec) {
    return sizeof(unsigned long long) * 4 * (size_t)g.N * (size_t)nvec;
}

// steps 2 .. Nt: F[0] = D^1, F[1] = W^1 (dense rows), acc holds c_0 W^0 + c_1 W^1.
// *taken = false when the device refuses the launch because its CTAs cannot all be
// resident (a partitioned GPU): nothing was computed and the caller takes the blocked kernels.
ew_status persist2d_advance(const GridGeom& g, const FilterPlan& plan, const float* cdev, float* const* F, float* acc,
                            int nvec, int64_t fstride, void* records, cudaStream_t st, bool* taken) {
    *taken = true;
    if (plan.Nt < 2) return EW_OK;
    const PersistPlan p = persist_plan(g, nvec, sm_count());
    if (!p.v) return set_error(EW_EUNSUPPORTED, "grid does not fit on the chip");
    EW_CUDA_TRY(cudaFuncSetAttribute(p.v->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)p.v->smem));
    Stencil<float> s = make_stencil<float>(g, plan.dt * plan.dt);
    int nx = (int)g.n[0], ny = (int)g.n[1], ntx = p.ntx, nty = p.nty;
    int64_t Nt = plan.Nt;
    const float *D1 = F[0], *W1 = F[1];
    if (!g.gave_up) return set_error(EW_EINVAL, "on-chip wave-solve: the grid has no word for waits that give up");
    int* gave_up = g.gave_up;
    unsigned long long* rec = (unsigned long long*)records;
    int stall = getenv("EW_TEST_RB2D_STALL") ? 1 : 0;  // test hook: the first CTA publishes nothing, so the waits run out
    EW_CUDA_TRY(cudaMemsetAsync(rec, 0, persist2d_room(g, nvec), st));
    void* args[] = {(void*)&nx, (void*)&ny, (void*)&D1,  (void*)&W1,  (void*)&acc,     (void*)&cdev, (void*)&Nt,
                    (void*)&s,  (void*)&ntx, (void*)&nty, (void*)&fstride, (void*)&rec,  (void*)&stall,
                    (void*)&gave_up};
    cudaEvent_t ev = fused_begin(st);
    cudaError_t e = getenv("EW_TEST_COOP_TOO_LARGE")  // test hook: the answer of a device with fewer SMs
                        ? cudaErrorCooperativeLaunchTooLarge
                        : cudaLaunchCooperativeKernel(p.v->fn, dim3((unsigned)(ntx * nty * nvec)),
                                                      dim3((unsigned)p.v->threads), args, p.v->smem, st);
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();
        if (ev) cudaEventDestroy(ev);
        *taken = false;
        return EW_OK;
    }
    EW_CUDA_TRY(e);
    fused_end(ev, st, g.N * nvec, g.N * nvec * (plan.Nt - 1));
    return EW_OK;
}

}  // namespace ew
