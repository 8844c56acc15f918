// ew_krylov.cu -- FP64 tall-skinny kernels of the Krylov eigen-solver (Arnoldi
// section): block Gram products C = A^T B with warp-shuffle reductions (the
// classical Gram-Schmidt coefficients, applied twice), block updates
// B <- beta B + alpha A M (the Gram-Schmidt subtraction, the thick-restart
// basis rotation V Y and the Cholesky-QR scaling), and precision conversions
// between the FP64 basis and the filter's FP32 fields.
//
// Layout: a block of vectors is column-major with leading dimension ld (each
// vector contiguous, vector j at offset j * ld).  The Gram product is
// deterministic: fixed block count, per-block partials summed in order.
#include <algorithm>

#include "ew_internal.h"

namespace ew {

constexpr int kGramTile = 4;    // 4 x 4 output entries per thread
constexpr int kGramThreads = 256;

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// part[(chunk * ma + i) * mb + j] = sum over the chunk's rows of A[r,i] B[r,j];
// with sym (A and B the same block) only the tiles on and above the diagonal.
//
// Bound: FP64 (two multiply-adds a clock and SM).  A thread's sixteen sums go
// through the warp by halves (each step sends the half that the other lane
// keeps): 16 additions a thread, where reducing them one by one took 80, as much
// as the rows' own multiply-adds.  Measured, N = 122 177: 16 x 16 of one block
// 253 us -> 72 us, 112 x 16 1748 -> 381 us (379 us of multiply-adds at full rate).
__global__ void __launch_bounds__(kGramThreads)
    k_gram(int64_t N, const double* __restrict__ A, int64_t lda, int ma, const double* __restrict__ B,
           int64_t ldb, int mb, bool sym, double* __restrict__ part) {
    __shared__ double sh[kGramThreads / 32][kGramTile * kGramTile];
    if (sym && blockIdx.z < blockIdx.y) return;
    const int i0 = blockIdx.y * kGramTile, j0 = blockIdx.z * kGramTile;
    double acc[kGramTile * kGramTile];
#pragma unroll
    for (int a = 0; a < kGramTile * kGramTile; ++a) acc[a] = 0.0;
    const int64_t chunk = (N + gridDim.x - 1) / gridDim.x;
    const int64_t r0 = blockIdx.x * chunk;
    const int64_t r1 = min(N, r0 + chunk);
    for (int64_t r = r0 + threadIdx.x; r < r1; r += kGramThreads) {
        double av[kGramTile], bv[kGramTile];
#pragma unroll
        for (int a = 0; a < kGramTile; ++a) av[a] = (i0 + a < ma) ? A[(int64_t)(i0 + a) * lda + r] : 0.0;
#pragma unroll
        for (int c = 0; c < kGramTile; ++c) bv[c] = (j0 + c < mb) ? B[(int64_t)(j0 + c) * ldb + r] : 0.0;
#pragma unroll
        for (int a = 0; a < kGramTile; ++a)
#pragma unroll
            for (int c = 0; c < kGramTile; ++c)
                acc[a * kGramTile + c] = fma(av[a], bv[c], acc[a * kGramTile + c]);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    static_assert(kGramTile * kGramTile == 16, "four halvings leave one sum a lane pair");
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) {  // lanes with bit 2 h keep the upper half
        const bool up = lane & (2 * h);
#pragma unroll
        for (int a = 0; a < h; ++a) {
            const double send = up ? acc[a] : acc[a + h];
            acc[a] = (up ? acc[a + h] : acc[a]) + __shfl_xor_sync(0xffffffffu, send, 2 * h);
        }
    }
    acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if (!(lane & 1)) sh[wid][lane >> 1] = acc[0];
    __syncthreads();
    if (threadIdx.x < kGramTile * kGramTile) {
        const int a = threadIdx.x / kGramTile, c = threadIdx.x % kGramTile;
        double v = 0.0;
        for (int w = 0; w < kGramThreads / 32; ++w) v += sh[w][threadIdx.x];
        if (i0 + a < ma && j0 + c < mb) part[((int64_t)blockIdx.x * ma + i0 + a) * mb + j0 + c] = v;
    }
}

// C[i * mb + j] = sum over chunks of part, one warp an entry (lanes strided over
// the chunks, then a fixed shuffle tree); with sym an entry below the diagonal's
// tiles is its mirror image's
__global__ void k_gram_finish(const double* __restrict__ part, int nchunks, int ma, int mb, bool sym,
                              double* __restrict__ C) {
    const int e = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
    if (e >= ma * mb) return;
    const int i = e / mb, j = e % mb;
    const int src = sym && i / kGramTile > j / kGramTile ? j * mb + i : e;
    double s = 0.0;
    for (int q = lane; q < nchunks; q += 32) s += part[(int64_t)q * ma * mb + src];
    s = wsum(s);
    if (lane == 0) C[e] = s;
}

constexpr int kGramChunks = 304;

// row chunks: the fewest multiply-adds in a row on an SM (its CTAs, each with its
// rows' sixteen a thread and about two rows' worth for the reduction).  304 chunks
// whatever the number of tiles left a thread one or two rows of a tile
static int gram_chunks(int64_t N, int64_t tiles, int nsm) {
    int best = 1;
    int64_t cost = INT64_MAX;
    for (int c = 1; c <= kGramChunks; ++c) {
        const int64_t rows = ((N + c - 1) / c + kGramThreads - 1) / kGramThreads;
        const int64_t k = (tiles * c + nsm - 1) / nsm * (rows + 2);
        if (k < cost) cost = k, best = c;
    }
    return best;
}

ew_status gram(int64_t N, const double* A, int64_t lda, int ma, const double* B, int64_t ldb, int mb,
               double* part, double* C, cudaStream_t st) {
    int dev = 0, nsm = 0;
    EW_CUDA_TRY(cudaGetDevice(&dev));
    EW_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const bool sym = A == B && lda == ldb && ma == mb;
    const int64_t ti = (ma + kGramTile - 1) / kGramTile, tj = (mb + kGramTile - 1) / kGramTile;
    const int chunks = gram_chunks(N, sym ? ti * (ti + 1) / 2 : ti * tj, nsm);
    dim3 grid((unsigned)chunks, (unsigned)ti, (unsigned)tj);
    k_gram<<<grid, kGramThreads, 0, st>>>(N, A, lda, ma, B, ldb, mb, sym, part);
    k_gram_finish<<<(ma * mb * 32 + 127) / 128, 128, 0, st>>>(part, chunks, ma, mb, sym, C);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch(2);
    return EW_OK;
}

size_t gram_part_doubles(int ma, int mb) { return (size_t)kGramChunks * ma * mb; }

// Out[:, j] = beta * Bin[:, j] + alpha * sum_i A[:, i] M[i * mb + j], j < mb.
// Rows are staged in shared memory first, so Out may alias A or Bin (the
// in-place basis rotation V[:, :k] = V[:, :m] Y).  Staged with the rows of a column
// side by side: a warp's multiply-add reads 32 neighbours and one broadcast.  (With
// a row's columns side by side its lanes met in one bank: 163 us on average over a
// solve with N = 122 177 and up to 112 columns, now 85 us, FP64 bound.)
constexpr int kUpdRows = 32;
constexpr int kUpdThreads = 256;

__global__ void __launch_bounds__(kUpdThreads)
    k_update(int64_t N, const double* A, int64_t lda, int ma, const double* Bin, int64_t ldb, int mb,
             const double* __restrict__ M, double alpha, double beta, double* Out, int64_t ldo) {
    extern __shared__ double sm[];
    double* sA = sm;                    // ma x kUpdRows: a warp (one j, 32 rows) reads 32 in a row
    double* sB = sA + kUpdRows * ma;    // mb x kUpdRows
    double* sM = sB + kUpdRows * mb;    // ma x mb
    const int64_t r0 = (int64_t)blockIdx.x * kUpdRows;
    const int nr = (int)min((int64_t)kUpdRows, N - r0);
    for (int e = threadIdx.x; e < ma * mb; e += kUpdThreads) sM[e] = M[e];
    for (int e = threadIdx.x; e < kUpdRows * ma; e += kUpdThreads) {
        int i = e / kUpdRows, r = e % kUpdRows;
        sA[e] = (r < nr) ? A[(int64_t)i * lda + r0 + r] : 0.0;
    }
    if (beta != 0.0)
        for (int e = threadIdx.x; e < kUpdRows * mb; e += kUpdThreads) {
            int j = e / kUpdRows, r = e % kUpdRows;
            sB[e] = (r < nr) ? Bin[(int64_t)j * ldb + r0 + r] : 0.0;
        }
    __syncthreads();
    for (int e = threadIdx.x; e < kUpdRows * mb; e += kUpdThreads) {
        int j = e / kUpdRows, r = e % kUpdRows;
        if (r >= nr) continue;
        double s = 0.0;
        for (int i = 0; i < ma; ++i) s = fma(sA[i * kUpdRows + r], sM[i * mb + j], s);
        double o = alpha * s;
        if (beta != 0.0) o = fma(beta, sB[e], o);
        Out[(int64_t)j * ldo + r0 + r] = o;
    }
}

ew_status update(int64_t N, const double* A, int64_t lda, int ma, const double* Bin, int64_t ldb, int mb,
                 const double* M, double alpha, double beta, double* Out, int64_t ldo, cudaStream_t st) {
    size_t smem = sizeof(double) * ((size_t)kUpdRows * (ma + mb) + (size_t)ma * mb);
    if (smem > 200 * 1024) return set_error(EW_EINVAL, "basis too wide for the update kernel");
    static bool attr = false;
    if (!attr) {
        EW_CUDA_TRY(cudaFuncSetAttribute(k_update, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr = true;
    }
    unsigned blocks = (unsigned)((N + kUpdRows - 1) / kUpdRows);
    k_update<<<blocks, kUpdThreads, smem, st>>>(N, A, lda, ma, Bin, ldb, mb, M, alpha, beta, Out, ldo);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}

template <typename S, typename D>
__global__ void k_convert(int64_t n, const S* __restrict__ x, D* __restrict__ y) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        y[q] = (D)x[q];
}

template <typename S, typename D>
ew_status convert(int64_t n, const S* x, D* y, cudaStream_t st) {
    int64_t b = (n + 255) / 256;
    k_convert<S, D><<<(unsigned)std::min<int64_t>(b, 152 * 32), 256, 0, st>>>(n, x, y);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}
template ew_status convert<double, float>(int64_t, const double*, float*, cudaStream_t);
template ew_status convert<float, double>(int64_t, const float*, double*, cudaStream_t);

// SplitMix64 (Steele, Lea, Flood 2014): draw i of stream `seed` mapped to
// uniform [-1, 1): 2 (z >> 11) 2^-53 - 1, z = mix(seed + (i + 1) * golden).
__global__ void k_splitmix_uniform(int64_t n, uint64_t seed, double* __restrict__ out) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        uint64_t z = seed + (uint64_t)(q + 1) * 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z = z ^ (z >> 31);
        out[q] = 2.0 * ((double)(z >> 11) * 0x1.0p-53) - 1.0;
    }
}

ew_status splitmix_uniform(int64_t n, uint64_t seed, double* out, cudaStream_t st) {
    int64_t b = (n + 255) / 256;
    k_splitmix_uniform<<<(unsigned)std::min<int64_t>(b, 152 * 32), 256, 0, st>>>(n, seed, out);
    EW_CUDA_TRY(cudaGetLastError());
    count_launch();
    return EW_OK;
}

}  // namespace ew
