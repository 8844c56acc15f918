// ew_small_eig.h -- the Rayleigh-Ritz step's small symmetric eigen-problem (host).
#pragma once

#include <math.h>

#include <algorithm>
#include <cmath>
#include <vector>

namespace ew {

// Eigenvalues w and eigenvectors (columns of V) of a symmetric matrix (row-major
// n x n, destroyed), for the Rayleigh-Ritz step: Householder reflections to
// tridiagonal form, then implicit QR steps with Wilkinson's shift (Golub and Van
// Loan, Matrix Computations, sections 8.3.1 to 8.3.3).  Everything runs along
// rows: the eigenvectors are kept as rows until the end.  For n = 112 1.6
// to 2.1 ms, Jacobi sweeps (ew_arnoldi.cu) 14 to 60 ms, with residuals and loss of
// orthogonality ten times larger than these.  Small eigenvalues are accurate to the matrix's
// norm only, which is all that Ritz values need; svqb() keeps the sweeps.
inline void tridiagonal_eig(int n, std::vector<double>& A, std::vector<double>& V, std::vector<double>& w) {
    auto row = [&](std::vector<double>& M, int i) { return M.data() + (size_t)i * n; };
    std::vector<double> v((size_t)n * n, 0.0), beta(n, 0.0), p(n), e(n, 0.0);
    w.assign(n, 0.0);
    // where squares of the entries would leave the range: entries near 1 (an exact scaling)
    double big = 0.0;
    int ex = 0;
    for (double a : A) big = std::max(big, fabs(a));
    if (big > 0.0 && std::isfinite(big)) frexp(big, &ex);
    if (ex > -300 && ex < 300) ex = 0;
    if (ex)
        for (double& a : A) a = ldexp(a, -ex);
    for (int k = 0; k + 2 < n; ++k) {  // reflection k zeroes column k below the subdiagonal
        double* vk = row(v, k);
        double ss = 0.0;
        for (int i = k + 1; i < n; ++i) {
            vk[i] = A[(size_t)i * n + k];
            if (i > k + 1) ss += vk[i] * vk[i];
        }
        if (ss == 0.0) continue;  // nothing to zero
        const double x0 = vk[k + 1], len = sqrt(x0 * x0 + ss), to = x0 > 0.0 ? -len : len;
        vk[k + 1] = x0 - to;
        beta[k] = 2.0 / (vk[k + 1] * vk[k + 1] + ss);
        A[(size_t)(k + 1) * n + k] = to;
        double pv = 0.0;
        for (int i = k + 1; i < n; ++i) {
            const double* a = row(A, i);
            double s = 0.0;
            for (int j = k + 1; j < n; ++j) s += a[j] * vk[j];
            p[i] = beta[k] * s;
            pv += p[i] * vk[i];
        }
        const double half = 0.5 * beta[k] * pv;
        for (int i = k + 1; i < n; ++i) p[i] -= half * vk[i];
        for (int i = k + 1; i < n; ++i) {
            double* a = row(A, i);
            const double vi = vk[i], pi = p[i];
            for (int j = k + 1; j < n; ++j) a[j] -= vi * p[j] + pi * vk[j];
        }
    }
    for (int i = 0; i < n; ++i) {
        w[i] = A[(size_t)i * n + i];
        if (i + 1 < n) e[i] = A[(size_t)(i + 1) * n + i];
    }
    // product of the reflections, then its transpose: rows that the QR steps rotate
    V.assign((size_t)n * n, 0.0);
    for (int i = 0; i < n; ++i) V[(size_t)i * n + i] = 1.0;
    for (int k = n - 3; k >= 0; --k) {
        if (beta[k] == 0.0) continue;
        const double* vk = row(v, k);
        std::fill(p.begin(), p.end(), 0.0);
        for (int i = k + 1; i < n; ++i) {
            const double* q = row(V, i);
            for (int j = k + 1; j < n; ++j) p[j] += vk[i] * q[j];
        }
        for (int i = k + 1; i < n; ++i) {
            double* q = row(V, i);
            const double f = beta[k] * vk[i];
            for (int j = k + 1; j < n; ++j) q[j] -= f * p[j];
        }
    }
    auto transpose = [&]() {
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < i; ++j) std::swap(V[(size_t)i * n + j], V[(size_t)j * n + i]);
    };
    transpose();
    auto negligible = [&](int i) { return fabs(e[i]) <= 1.1e-16 * (fabs(w[i]) + fabs(w[i + 1])); };
    int hi = n - 1;
    for (int it = 0; hi > 0 && it < 60 * n; ++it) {
        if (negligible(hi - 1)) {
            e[--hi] = 0.0;
            continue;
        }
        int lo = hi - 1;
        while (lo > 0 && !negligible(lo - 1)) --lo;
        const double del = 0.5 * (w[hi - 1] - w[hi]), eh = e[hi - 1];
        const double sq = sqrt(del * del + eh * eh), root = sq > 0.0 ? sq : hypot(del, eh);
        const double shift = w[hi] - eh * (eh / (del >= 0.0 ? del + root : del - root));
        double x = w[lo] - shift, z = e[lo];  // the bulge starts here and is chased to hi
        for (int k = lo; k < hi; ++k) {
            const double r = hypot(x, z), c = r > 0.0 ? x / r : 1.0, s = r > 0.0 ? z / r : 0.0;
            if (k > lo) e[k - 1] = r;
            const double t = s * (w[k + 1] - w[k]) + 2.0 * c * e[k];
            w[k] += s * t;
            w[k + 1] -= s * t;
            e[k] = c * t - e[k];
            x = e[k];
            if (k + 1 < hi) {
                z = s * e[k + 1];
                e[k + 1] *= c;
            }
            double *a = row(V, k), *b = row(V, k + 1);
            for (int j = 0; j < n; ++j) {
                const double aj = a[j], bj = b[j];
                a[j] = c * aj + s * bj;
                b[j] = c * bj - s * aj;
            }
        }
    }
    transpose();
    if (ex)
        for (double& a : w) a = ldexp(a, ex);
}

}  // namespace ew
