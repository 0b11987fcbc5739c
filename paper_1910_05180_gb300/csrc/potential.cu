// potential.cu -- host side of the TI potential's evaluation: the sum over the
// coupling groups as one rational function of q = phi (1 - phi).
//
// Eq. 6 gives, per cell, sum_k beta_k / (1 - A_k s^2) with s = 1 - 2 phi.  Since
// s^2 = 1 - 4 q, every term is (beta_k / e_k) / (1 + g_k q) with e_k = 1 - A_k
// and g_k = 4 A_k / e_k: all weights and all g_k are positive, so for q >= 0
// the sum written as N(q) / D(q), D = prod (1 + g_k q), has positive
// coefficients only and Horner's rule loses nothing to cancellation.  K groups
// cost 2 K - 1 FMAs and one division, where summing them as a running fraction
// costs 4 K - 2 operations and the square of s.
//
// Fewer terms.  As a function of u = s^2 the sum is a Stieltjes function: its
// poles 1 / A_k lie beyond 1.  A rational function of degree N < K that agrees
// with it in 2 N points of [0, u_hi] comes from the Gauss quadrature of the
// measure beta_k / prod_i (1 - u_i A_k) (multipoint Pade approximation of
// Stieltjes functions; see Stahl and Totik, "General Orthogonal Polynomials",
// 1992, ch. 6), here by Lanczos' algorithm on the K masses and QL
// iterations (Golub and Welsch, Math. Comp. 23, 1969).  The nodes stay inside
// the range of the A_k and the weights stay positive, so the form above is
// kept.  The u_i are Chebyshev points in log(1 / A_max - u), which crowds them
// where the nearest pole is felt: the error falls below 2^-30 of the sum with
// N = 3 at lambda = 6 dx, 4 at 3 dx, 5-6 at 2 dx, 7-8 at 1 dx for a generic
// normal (13 groups).  That is far below the FP32 rounding of either form;
// FP64 grids take every group.  u_hi = 1 + min(0.05, a quarter of the way to
// the first pole); cells beyond it (phi outside [0, 1] by more than 1.2 %)
// are summed group by group in the kernel.
#include <math.h>

#include <algorithm>

#include "host_internal.h"

namespace spfm_host {

namespace {

constexpr int kK = spfm::kMaxTerms;
constexpr double kTol = 0x1p-30;
// largest coefficients, with room for q outside [0, 1/4] in the compute type's range
constexpr double kMaxCoef32 = 1e24, kMaxCoef64 = 1e100;

// Eigenvalues d and first components z of the unit eigenvectors of the n x n
// symmetric tridiagonal matrix with diagonal d and off-diagonal e, by QL
// iterations with Wilkinson's shift (Golub and Welsch); false without convergence.
bool eigen(double *d, double *e, double *z, int n)
{
    for (int i = 0; i < n; ++i) z[i] = i == 0 ? 1.0 : 0.0;
    e[n - 1] = 0.0;
    for (int l = 0; l < n; ++l)
        for (int it = 0;; ++it) {
            int m = l;   // the block l..m is unreduced
            while (m < n - 1 && fabs(e[m]) > 1e-17 * (fabs(d[m]) + fabs(d[m + 1]))) ++m;
            if (m == l) break;
            if (it == 50) return false;
            // the shift: the eigenvalue of the leading 2 x 2 block nearer d[l]
            const double h = (d[l + 1] - d[l]) / (2.0 * e[l]);
            const double shift = d[l] - e[l] / (h + copysign(sqrt(h * h + 1.0), h));
            // one sweep of plane rotations from the bottom chases the bulge up
            double x = d[m] - shift, y = e[m - 1];
            for (int i = m - 1; i >= l; --i) {
                const double r = sqrt(x * x + y * y);
                if (r == 0.0) break;
                const double c = x / r, s = y / r;   // rotates (i, i + 1)
                if (i < m - 1) e[i + 1] = r;
                const double a = d[i], b = e[i], f = d[i + 1];
                d[i + 1] = c * c * f + 2.0 * c * s * b + s * s * a;
                d[i] = s * s * f - 2.0 * c * s * b + c * c * a;
                e[i] = c * s * (a - f) + (c * c - s * s) * b;
                const double t = z[i + 1];
                z[i + 1] = c * t + s * z[i];
                z[i] = c * z[i] - s * t;
                if (i > l) {
                    x = e[i];
                    y = s * e[i - 1];
                    e[i - 1] *= c;
                }
            }
        }
    return true;
}

// N nodes and weights whose sum of w / (1 - x u) agrees with that of
// (A, beta) in the 2 N points u
bool reduce(const double *A, const double *beta, int K, int N, const double *u, double *x, double *w)
{
    double Q[kK][kK], off[kK], v0[kK], total = 0.0;
    for (int k = 0; k < K; ++k) {
        double om = 1.0;
        for (int i = 0; i < 2 * N; ++i) om *= 1.0 - u[i] * A[k];
        Q[0][k] = beta[k] / om;
        total += Q[0][k];
    }
    for (int k = 0; k < K; ++k) Q[0][k] = sqrt(Q[0][k] / total);
    for (int n = 0; n < N; ++n) {
        double a = 0.0, r[kK], norm = 0.0;
        for (int k = 0; k < K; ++k) a += A[k] * Q[n][k] * Q[n][k];
        x[n] = a;
        if (n == N - 1) break;
        for (int k = 0; k < K; ++k) r[k] = A[k] * Q[n][k];
        for (int pass = 0; pass < 2; ++pass)   // orthogonal to all before, twice
            for (int j = 0; j <= n; ++j) {
                double d = 0.0;
                for (int k = 0; k < K; ++k) d += r[k] * Q[j][k];
                for (int k = 0; k < K; ++k) r[k] -= d * Q[j][k];
            }
        for (int k = 0; k < K; ++k) norm += r[k] * r[k];
        norm = sqrt(norm);
        if (!(norm > 1e-14 * a)) return false;   // fewer than N distinct masses
        off[n] = norm;
        for (int k = 0; k < K; ++k) Q[n + 1][k] = r[k] / norm;
    }
    if (!eigen(x, off, v0, N)) return false;
    for (int j = 0; j < N; ++j) {
        double om = total * v0[j] * v0[j];
        for (int i = 0; i < 2 * N; ++i) om *= 1.0 - u[i] * x[j];
        w[j] = om;
        if (!(x[j] > 0.0 && x[j] < 1.0 && w[j] > 0.0)) return false;
    }
    return true;
}

// N(q) / D(q) of the nodes x with e = 1 - x and weights w; false above max_coef
bool expand(const double *x, const double *e, const double *w, int N, double max_coef, Rational &r)
{
    r.deg = N;
    for (int i = 0; i < kK; ++i) r.num[i] = 0.0;
    for (int i = 0; i <= kK; ++i) r.den[i] = i == 0 ? 1.0 : 0.0;
    for (int k = 0; k < N; ++k) {
        const double g = 4.0 * x[k] / e[k], wk = w[k] / e[k];
        // N <- N (1 + g q) + wk D, D <- D (1 + g q)
        for (int i = k; i >= 0; --i) r.num[i] += (i > 0 ? g * r.num[i - 1] : 0.0) + wk * r.den[i];
        for (int i = k + 1; i >= 1; --i) r.den[i] += g * r.den[i - 1];
    }
    for (int i = 0; i <= N; ++i)
        if (!(r.den[i] < max_coef) || (i < N && !(r.num[i] < max_coef))) return false;
    return true;
}

}  // namespace

void build_rational(const double *A, const double *E, const double *beta, int K, bool fp32, Rational &r)
{
    const double max_coef = fp32 ? kMaxCoef32 : kMaxCoef64;
    r.deg = 0;
    r.q_lo = -HUGE_VAL;
    if (K < 1) {   // no coupled direction: the sum is 0
        const double x = 0.0, e = 1.0, w = 0.0;
        expand(&x, &e, &w, 1, max_coef, r);
        return;
    }
    if (fp32 && K > 2) {
        double amax = 0.0;
        for (int k = 0; k < K; ++k) amax = std::max(amax, A[k]);
        const double pole = 1.0 / amax, u_hi = 1.0 + std::min(0.05, 0.25 * (pole - 1.0));
        const bool room = pole - u_hi > 0.0;   // none where some A_k is 1
        const double l0 = log(pole), l1 = room ? log(pole - u_hi) : l0;
        // a generic normal needs about 2.7 + log(pole / (pole - u_hi)) terms: the search starts there
        for (int N = std::max(2, (int)(2.7 + l0 - l1)); N < K && room; ++N) {
            double u[2 * kK], x[kK], w[kK], e[kK];
            for (int i = 0; i < 2 * N; ++i)
                u[i] = pole - exp(l0 + (l1 - l0) * 0.5 * (1.0 - cos(M_PI * (2 * i + 1) / (4.0 * N))));
            if (!reduce(A, beta, K, N, u, x, w)) continue;
            // the error peaks between the points of agreement and at the ends
            double worst = 0.0;
            for (int i = 0; i <= 2 * N; ++i) {
                const double v = pole - exp(l0 + (l1 - l0) * 0.5 * (1.0 - cos(M_PI * i / (2.0 * N))));
                double f = 0.0, g = 0.0;
                for (int k = 0; k < K; ++k) f += beta[k] / (1.0 - A[k] * v);
                for (int j = 0; j < N; ++j) g += w[j] / (1.0 - x[j] * v);
                worst = std::max(worst, fabs(g / f - 1.0));
            }
            if (!(worst < kTol)) continue;
            for (int j = 0; j < N; ++j) e[j] = 1.0 - x[j];
            if (expand(x, e, w, N, max_coef, r)) {
                r.q_lo = 0.25 * (1.0 - u_hi);
                return;
            }
        }
    }
    if (!expand(A, E, beta, K, max_coef, r)) r.deg = 0;
}

}  // namespace spfm_host
