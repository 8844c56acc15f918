// ew_reg2d_dev.cuh -- the temporally blocked 2D FP32 step with a tile's time
// levels in registers.
//
// A warp owns 128 columns and KY rows of the staged region, a lane four
// columns in a row: W^n, D^n = W^n - W^{n-1} and the filter sums of its points
// stay in its registers for all steps of the tile.  The neighbours in x come
// from the adjacent lanes (shuffles), those in y from the lane's own rows but
// for the R rows beyond the warp's first and last, which the warps publish to
// one another through shared memory, one barrier a step.  (W in shared memory,
// as in ew_tb2d_dev.cuh, takes three reads and a write of it a point and step:
// 70 % of the shared-memory bandwidth of the whole launch, and the arithmetic
// waits for it.  Here a point takes a quarter of that: 20.5 -> 16.0 ms for 64 boxes
// at order 2.)  What bounds it now is latency: instructions issue on 36 % of the
// cycles, three warps a scheduler, each row's chain of shuffle and seven
// dependent operations.  Tried: 16 warps of 6 rows 16.4 ms, 8 warps of 13 rows 17
// ms, 20 and 24 warps spill; an mbarrier with the edge rows computed first in place
// of the barrier 16.5 ms; descriptors fetched two tiles ahead 16.4 ms.
//
// The region is 128 x NW KY with a halo of H = R B: the lanes and warps at its
// edge compute with zeros for what lies beyond, and the points that this
// reaches in B steps are those of the halo.  Points outside the box hold the
// box closure's extension (ew_bc_dev.cuh), which the steps preserve.
//
// Staging: a warp copies its own rows (D, W and the filter sums) with
// asynchronous copies to its part of shared memory and picks up four columns a
// lane from there; the copies of the next tile are under way while this one is
// computed.  Results go back through the warp's exchange rows, so that the
// stores are contiguous.
//
// The operations of a point and their order are those of tb2d_tile
// (ew_tb2d_dev.cuh): the same bits.
#pragma once

#include "ew_tb2d_dev.cuh"

namespace ew {

template <int R, int NW, int KY, int B>
struct Reg2dShape {
    static constexpr int RX = 128, RY = NW * KY;
    static constexpr int H = R * B;  // halo
    static constexpr int TX = RX - 2 * H, TY = RY - 2 * H;
    static constexpr int NT = 32 * NW;
    static constexpr int PLANE = RX * RY;                // floats of one staged field
    static constexpr int EX = 2 * R * RX;                // floats a warp publishes a step
    static constexpr size_t SMEM = sizeof(float) * (3 * (size_t)PLANE + 2 * (size_t)NW * EX);
    static_assert(TX > 0 && TY > 0, "halo larger than the tile");
    static_assert(KY >= R && 2 * EX >= 3 * RX, "exchange rows, and the room to hand back a row of three fields");
};

// asynchronous copy of one float, or a zero
__device__ __forceinline__ void cp_async4_if(float* dst, const float* src, bool in) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(in ? 4 : 0) : "memory");
}

// a tile to stage: the level pair (D, W) = (Ain, Bin), the sums, and the global
// coordinates of the staged region's corner
struct Reg2dTile {
    int nx, ny, bc;
    int x0, y0;
    const float *Ain, *Bin, *acc;
};

// start the copies of the warp's rows
template <int R, int NW, int KY, int B, bool GEN>
__device__ __forceinline__ void reg2d_stage(const Reg2dTile t, float* stage) {
    using S = Reg2dShape<R, NW, KY, B>;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int nx = t.nx, ny = t.ny, x0 = t.x0, y0 = t.y0;
    const float *Ain = t.Ain, *Bin = t.Bin, *acc = t.acc;
    const bool inside = x0 >= 0 && x0 + S::RX <= nx && y0 >= 0 && y0 + S::RY <= ny;
    float* dst = stage + wy * KY * S::RX + lane;
    // the filter sums are those of the owned points (the others' are not stored)
    auto own = [&](int q) { return lane + 32 * q >= S::H && lane + 32 * q < S::H + S::TX; };
    if (inside) {
        int64_t g = (int64_t)(y0 + wy * KY) * nx + x0 + lane;
#pragma unroll 1
        for (int k = 0; k < KY; ++k, g += nx) {
            const bool owny = wy * KY + k >= S::H && wy * KY + k < S::H + S::TY;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                cp_async4(dst + k * S::RX + 32 * q, Ain + g + 32 * q);
                cp_async4(dst + S::PLANE + k * S::RX + 32 * q, Bin + g + 32 * q);
                if (owny && own(q)) cp_async4(dst + 2 * S::PLANE + k * S::RX + 32 * q, acc + g + 32 * q);
            }
        }
    } else {
        int ix[4], s = 1;  // source columns (-1: zero); the signs are applied when the rows are picked up
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int gx = x0 + lane + 32 * q;
            ix[q] = gx >= 0 && gx < nx ? gx : ext2<GEN>(gx, nx, axis_bc(t.bc, 0), s);
        }
#pragma unroll 1
        for (int k = 0; k < KY; ++k) {
            const int gy = y0 + wy * KY + k;
            const bool iny = gy >= 0 && gy < ny;
            const int iy = iny ? gy : ext2<GEN>(gy, ny, axis_bc(t.bc, 1), s);
            const int64_t row = (int64_t)(iy < 0 ? 0 : iy) * nx;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool in = ix[q] >= 0 && iy >= 0;
                const int64_t g = row + (in ? ix[q] : 0);
                cp_async4_if(dst + k * S::RX + 32 * q, Ain + g, in);
                cp_async4_if(dst + S::PLANE + k * S::RX + 32 * q, Bin + g, in);
                if (iny && own(q) && x0 + lane + 32 * q < nx)
                    cp_async4(dst + 2 * S::PLANE + k * S::RX + 32 * q, acc + g);
            }
        }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}

// the b <= B steps of a staged tile, weights cw; next() starts the copies of the
// tile after it once this one is in registers
template <int R, int NW, int KY, int B, bool GEN, class Next>
__device__ __forceinline__ void reg2d_steps(const Reg2dTile t, float* __restrict__ Aout, float* __restrict__ Bout,
                                            float* __restrict__ acc, const float* __restrict__ cw, int b,
                                            const Stencil<float>& st, float* stage, float* exch, Next next) {
    using S = Reg2dShape<R, NW, KY, B>;
    static_assert(B <= 32, "a lane holds one step's weight");
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, wy = threadIdx.x >> 5;
    const int nx = t.nx, ny = t.ny, x0 = t.x0, y0 = t.y0;
    const float cl = lane < b ? cw[lane] : 0.f;
    float2 w[KY][2], d[KY][2], a[KY][2];
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncwarp();
    {
        const float* src = stage + wy * KY * S::RX + 4 * lane;
#pragma unroll
        for (int k = 0; k < KY; ++k) {
            const float4 v0 = *reinterpret_cast<const float4*>(src + k * S::RX);
            const float4 v1 = *reinterpret_cast<const float4*>(src + S::PLANE + k * S::RX);
            const float4 v2 = *reinterpret_cast<const float4*>(src + 2 * S::PLANE + k * S::RX);
            d[k][0] = make_float2(v0.x, v0.y), d[k][1] = make_float2(v0.z, v0.w);
            w[k][0] = make_float2(v1.x, v1.y), w[k][1] = make_float2(v1.z, v1.w);
            a[k][0] = make_float2(v2.x, v2.y), a[k][1] = make_float2(v2.z, v2.w);
        }
    }
    if (!(x0 >= 0 && x0 + S::RX <= nx && y0 >= 0 && y0 + S::RY <= ny)) {
        int sx[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int gx = x0 + 4 * lane + i;
            sx[i] = 1;
            if (gx < 0 || gx >= nx) ext2<GEN>(gx, nx, axis_bc(t.bc, 0), sx[i]);
        }
#pragma unroll
        for (int k = 0; k < KY; ++k) {
            const int gy = y0 + wy * KY + k;
            int sy = 1;
            if (gy < 0 || gy >= ny) ext2<GEN>(gy, ny, axis_bc(t.bc, 1), sy);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (sx[2 * h] * sy < 0) w[k][h].x = -w[k][h].x, d[k][h].x = -d[k][h].x;
                if (sx[2 * h + 1] * sy < 0) w[k][h].y = -w[k][h].y, d[k][h].y = -d[k][h].y;
            }
        }
    }
    // publish W of the warp's first and last R rows
    auto publish_rows = [&](int p) {
        float* e = exch + (p * NW + wy) * S::EX + 4 * lane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            *reinterpret_cast<float4*>(e + r * S::RX) = make_float4(w[r][0].x, w[r][0].y, w[r][1].x, w[r][1].y);
            const int k = KY - R + r;
            *reinterpret_cast<float4*>(e + (R + r) * S::RX) = make_float4(w[k][0].x, w[k][0].y, w[k][1].x, w[k][1].y);
        }
    };
    __syncwarp();  // the rows are picked up: the next tile's may come
    next();
    publish_rows(0);
    __syncthreads();
    const float2 C0{st.c0, st.c0}, C1X{st.c1[0], st.c1[0]}, C1Y{st.c1[1], st.c1[1]};
    const float2 C2X{st.c2[0], st.c2[0]}, C2Y{st.c2[1], st.c2[1]};
    for (int s = 0; s < b; ++s) {
        const float cs = __shfl_sync(FULL, cl, s);
        const float2 CS{cs, cs};
        // rows above the warp's first (its neighbour's last R) and below its last
        float2 up[R][2], dn[R][2];
        const float* e = exch + ((s & 1) * NW + wy) * S::EX + 4 * lane;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            float4 u = make_float4(0.f, 0.f, 0.f, 0.f), l = u;
            if (wy > 0) u = *reinterpret_cast<const float4*>(e - S::EX + (R + r) * S::RX);
            if (wy < NW - 1) l = *reinterpret_cast<const float4*>(e + S::EX + r * S::RX);
            up[r][0] = make_float2(u.x, u.y), up[r][1] = make_float2(u.z, u.w);
            dn[r][0] = make_float2(l.x, l.y), dn[r][1] = make_float2(l.z, l.w);
        }
#pragma unroll
        for (int k = 0; k < KY; ++k) {
            // up[r]: the old row k - R + r
            const float2 p = w[k][0], q = w[k][1];
            const float ld = __shfl_up_sync(FULL, q.y, 1), ra = __shfl_down_sync(FULL, p.x, 1);
            const float2* n1 = k + 1 < KY ? w[k + 1 < KY ? k + 1 : 0] : dn[k + 1 < KY ? 0 : k + 1 - KY];
            float2 lap[2], nv[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 c = w[k][h];
                const float2 sx1 = h ? make_float2(s_add(p.y, q.y), s_add(q.x, ra))
                                     : make_float2(s_add(ld, p.y), s_add(p.x, q.x));
                lap[h] = p_mul(C0, c);
                lap[h] = p_fma(C1X, sx1, lap[h]);
                lap[h] = p_fma(C1Y, p_add(up[R - 1][h], n1[h]), lap[h]);
            }
            if constexpr (R == 2) {
                const float lc = __shfl_up_sync(FULL, q.x, 1), rb = __shfl_down_sync(FULL, p.y, 1);
                const float2* n2 = k + 2 < KY ? w[k + 2 < KY ? k + 2 : 0] : dn[k + 2 < KY ? 0 : k + 2 - KY];
                lap[0] = p_fma(C2X, p_add(make_float2(lc, ld), q), lap[0]);
                lap[1] = p_fma(C2X, p_add(p, make_float2(ra, rb)), lap[1]);
#pragma unroll
                for (int h = 0; h < 2; ++h) lap[h] = p_fma(C2Y, p_add(up[0][h], n2[h]), lap[h]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                d[k][h] = p_add(d[k][h], lap[h]);  // D^{n+1} = D^n + dt^2 L W^n
                nv[h] = p_add(w[k][h], d[k][h]);   // W^{n+1} = W^n + D^{n+1}
                a[k][h] = p_fma(CS, nv[h], a[k][h]);
                if constexpr (R == 2) up[0][h] = up[1][h];
                up[R - 1][h] = w[k][h];
                w[k][h] = nv[h];
            }
        }
        if (s + 1 < b) {
            publish_rows((s + 1) & 1);
            __syncthreads();
        }
    }
    // the owned points back: a row of the three fields through the warp's exchange
    // rows of both buffers (its neighbours are done with them after this barrier)
    __syncthreads();
    float* e0 = exch + wy * S::EX;
    float* e1 = exch + (NW + wy) * S::EX;
    float* t0 = e0;
    float* t1 = e0 + S::RX;
    float* t2 = 2 * S::EX >= 3 * S::RX && S::EX >= 3 * S::RX ? e0 + 2 * S::RX : e1;
#pragma unroll
    for (int k = 0; k < KY; ++k) {
        const int sy = wy * KY + k, gy = y0 + sy;
        if (sy < S::H || sy >= S::H + S::TY || gy >= ny) continue;
        *reinterpret_cast<float4*>(t0 + 4 * lane) = make_float4(d[k][0].x, d[k][0].y, d[k][1].x, d[k][1].y);
        *reinterpret_cast<float4*>(t1 + 4 * lane) = make_float4(w[k][0].x, w[k][0].y, w[k][1].x, w[k][1].y);
        *reinterpret_cast<float4*>(t2 + 4 * lane) = make_float4(a[k][0].x, a[k][0].y, a[k][1].x, a[k][1].y);
        __syncwarp();
        const int64_t g = (int64_t)gy * nx + x0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int sx = lane + 32 * q;
            if (sx >= S::H && sx < S::H + S::TX && x0 + sx < nx) {
                Aout[g + sx] = t0[sx];
                Bout[g + sx] = t1[sx];
                acc[g + sx] = t2[sx];
            }
        }
        __syncwarp();
    }
}

}  // namespace ew
