// Small dense linear algebra on the host, for the m x m matrices of the
// small-space setup (Gram matrices for Cholesky-QR re-orthonormalisation and
// the Rayleigh-Ritz matrices of the eigensolver), and the Chebyshev
// coefficients of the polynomial P(x) ~ x^{-1/2} (Sec. 2).
//
// Matrices are column-major arrays of (re, im) pairs, A(i, j) = A[i + j n].
#include <algorithm>
#include <cmath>
#include <limits>
#include <numeric>
#include <vector>

#include "ovl_internal.h"

namespace ovl {
namespace {
// Complex arithmetic in plain real operations: std::complex multiplies through a library routine that
// looks for NaNs.
inline HostCplx operator+(HostCplx a, HostCplx b) { return {a.re + b.re, a.im + b.im}; }
inline HostCplx operator-(HostCplx a, HostCplx b) { return {a.re - b.re, a.im - b.im}; }
inline HostCplx operator*(HostCplx a, HostCplx b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
inline HostCplx operator*(double a, HostCplx b) { return {a * b.re, a * b.im}; }
inline HostCplx conj(HostCplx a) { return {a.re, -a.im}; }
inline double norm(HostCplx a) { return a.re * a.re + a.im * a.im; }
// y -= c x over n numbers
inline void subtract(int n, HostCplx c, const HostCplx* x, HostCplx* y) {
    for (int i = 0; i < n; ++i) {
        y[i].re -= c.re * x[i].re - c.im * x[i].im;
        y[i].im -= c.re * x[i].im + c.im * x[i].re;
    }
}
}  // namespace

bool host_cholesky(int n, std::vector<HostCplx>& A) {
    // Left-looking by columns: column j loses its part on the columns before it, then is scaled.
    for (int j = 0; j < n; ++j) {
        HostCplx* cj = &A[(size_t)j * n];
        for (int k = 0; k < j; ++k) {
            const HostCplx* ck = &A[(size_t)k * n];
            subtract(n - j, conj(ck[j]), ck + j, cj + j);
        }
        const double d = cj[j].re;
        if (!(d > 0.0) || !std::isfinite(d)) return false;
        const double r = std::sqrt(d);
        cj[j] = HostCplx{r, 0.0};
        for (int i = j + 1; i < n; ++i) cj[i] = HostCplx{cj[i].re / r, cj[i].im / r};
        for (int i = 0; i < j; ++i) cj[i] = HostCplx{0.0, 0.0};  // clear the upper triangle
    }
    return true;
}

void host_inv_lower_dag(int n, const std::vector<HostCplx>& L, std::vector<HostCplx>& R) {
    // X = L^{-1} (lower) by forward substitution, column by column; R = X^+.
    R.assign((size_t)n * n, HostCplx{0.0, 0.0});
    std::vector<HostCplx> x(n);
    for (int c = 0; c < n; ++c) {
        std::fill(x.begin(), x.end(), HostCplx{0.0, 0.0});
        x[c].re = 1.0;
        for (int k = c; k < n; ++k) {  // x_k is known: it leaves the rows below
            const HostCplx* ck = &L[(size_t)k * n];
            x[k] = HostCplx{x[k].re / ck[k].re, x[k].im / ck[k].re};  // the diagonal is real
            subtract(n - k - 1, x[k], ck + k + 1, x.data() + k + 1);
        }
        for (int i = c; i < n; ++i) R[c + (size_t)i * n] = conj(x[i]);
    }
}

namespace {
// The Hermitian A (n x n, overwritten) becomes Q T Q^+ with T real and tridiagonal (diagonal d,
// subdiagonal e): Q is a product of reflections 1 - tau_k v_k v_k^+, k = 0 .. n - 2, whose v_k (1 at row
// k + 1) are left below the diagonal of column k.  Reflection k maps the column below the diagonal onto a
// real multiple of its first entry, and A - v w^+ - w v^+ is what both sides of it leave of the rest.
void tridiagonalise(int n, std::vector<HostCplx>& A, std::vector<double>& d, std::vector<double>& e,
                    std::vector<HostCplx>& tau) {
    std::vector<HostCplx> w(n);
    for (int k = 0; k + 1 < n; ++k) {
        const int m = n - k - 1, r0 = k + 1;
        HostCplx* v = &A[r0 + (size_t)k * n];
        d[k] = A[k + (size_t)k * n].re;
        double rest = 0.0;
        for (int i = 1; i < m; ++i) rest = std::max(rest, std::max(std::fabs(v[i].re), std::fabs(v[i].im)));
        const double most = std::max(rest, std::max(std::fabs(v[0].re), std::fabs(v[0].im)));
        if (rest == 0.0 && v[0].im == 0.0) {  // already real: no reflection
            e[k] = v[0].re;
            tau[k] = HostCplx{0.0, 0.0};
            continue;
        }
        // The column's largest number is brought near 1: a column may be far below the matrix, and its squares
        // below the smallest double.
        int scale = 0;
        std::frexp(most, &scale);
        double below = 0.0;
        for (int i = 0; i < m; ++i) {
            v[i] = HostCplx{std::ldexp(v[i].re, -scale), std::ldexp(v[i].im, -scale)};
            if (i > 0) below += norm(v[i]);
        }
        const HostCplx a = v[0];
        const double beta = -std::copysign(std::sqrt(norm(a) + below), a.re);
        tau[k] = HostCplx{(beta - a.re) / beta, -a.im / beta};
        const HostCplx t{a.re - beta, a.im};  // v = (x - beta e_1) / (a - beta)
        const double q = 1.0 / norm(t);
        const HostCplx inv{t.re * q, -t.im * q};
        for (int i = 1; i < m; ++i) v[i] = inv * v[i];
        v[0] = HostCplx{1.0, 0.0};
        e[k] = std::ldexp(beta, scale);
        // w = tau A v - 1/2 tau (tau A v, v) v on the trailing block
        std::fill(w.begin(), w.begin() + m, HostCplx{0.0, 0.0});
        for (int j = 0; j < m; ++j) subtract(m, HostCplx{-v[j].re, -v[j].im}, &A[r0 + (size_t)(r0 + j) * n], w.data());
        HostCplx dot{0.0, 0.0};
        for (int i = 0; i < m; ++i) {
            w[i] = tau[k] * w[i];
            dot = dot + conj(w[i]) * v[i];
        }
        subtract(m, 0.5 * (tau[k] * dot), v, w.data());
        for (int j = 0; j < m; ++j) {
            HostCplx* c = &A[r0 + (size_t)(r0 + j) * n];
            const HostCplx vj = conj(v[j]), wj = conj(w[j]);
            for (int i = 0; i < m; ++i) {
                c[i].re -= v[i].re * wj.re - v[i].im * wj.im + w[i].re * vj.re - w[i].im * vj.im;
                c[i].im -= v[i].re * wj.im + v[i].im * wj.re + w[i].re * vj.im + w[i].im * vj.re;
            }
        }
    }
    d[n - 1] = A[(size_t)n * n - 1].re;
}

// Eigenvalues of the tridiagonal (d, e) into d, the rotations accumulated into Z (n x n, column-major):
// implicit QR steps with Wilkinson's shift on unreduced blocks (Golub and Van Loan, Matrix
// Computations, section 8.3).  false: not converged.
bool diagonalise(int n, std::vector<double>& d, std::vector<double>& e, std::vector<double>& Z) {
    const double eps = 2.220446049250313e-16, floor = 1e-280;  // (the largest number is near 1)
    int hi = n - 1;
    for (int steps = 0; hi > 0 && steps < 60 * n; ++steps) {
        if (std::fabs(e[hi - 1]) <= eps * (std::fabs(d[hi - 1]) + std::fabs(d[hi])) + floor) {
            --hi;
            continue;
        }
        int lo = hi - 1;
        while (lo > 0 && std::fabs(e[lo - 1]) > eps * (std::fabs(d[lo - 1]) + std::fabs(d[lo])) + floor) --lo;
        const double h = 0.5 * (d[hi - 1] - d[hi]), b2 = e[hi - 1];
        const double shift = d[hi] - b2 * (b2 / (h + std::copysign(std::hypot(h, b2), h)));
        double x = d[lo] - shift, z = e[lo];
        for (int k = lo; k < hi; ++k) {
            const double r = std::hypot(x, z);
            const double c = r > 0.0 ? x / r : 1.0, s = r > 0.0 ? z / r : 0.0;
            if (k > lo) e[k - 1] = r;
            const double a = d[k], b = e[k], g = d[k + 1];
            d[k] = c * (c * a + s * b) + s * (c * b + s * g);
            d[k + 1] = s * (s * a - c * b) + c * (c * g - s * b);
            e[k] = c * (c * b + s * g) - s * (c * a + s * b);
            if (k + 1 < hi) {
                z = s * e[k + 1];
                e[k + 1] *= c;
                x = e[k];
            }
            double* zk = &Z[(size_t)k * n];
            double* zn = zk + n;
            for (int i = 0; i < n; ++i) {
                const double p = zk[i], q = zn[i];
                zk[i] = c * p + s * q;
                zn[i] = c * q - s * p;
            }
        }
    }
    return hi == 0;
}
}  // namespace

bool host_eigh(int n, std::vector<HostCplx>& A, std::vector<double>& w, std::vector<HostCplx>& Z) {
    // Reflections to real tridiagonal form, its eigenvectors by QR steps, and the reflections applied to
    // them.  32 x 32: 0.4 ms where cyclic Jacobi sweeps took 9; 256 x 256: 0.12 against 5.2 s.
    w.assign(n, 0.0);
    Z.assign((size_t)n * n, HostCplx{0.0, 0.0});
    if (n < 1) return true;
    // the largest number is brought near 1, so that no square overflows
    double most = 0.0;
    bool finite = true;
    for (const HostCplx& v : A) {
        finite = finite && std::isfinite(v.re) && std::isfinite(v.im);
        most = std::max(most, std::max(std::fabs(v.re), std::fabs(v.im)));
    }
    if (!finite) {
        const double nan = std::numeric_limits<double>::quiet_NaN();
        w.assign(n, nan);
        Z.assign((size_t)n * n, HostCplx{nan, nan});
        return false;
    }
    int scale = 0;
    if (most > 0.0) {
        std::frexp(most, &scale);
        for (HostCplx& v : A) v = HostCplx{std::ldexp(v.re, -scale), std::ldexp(v.im, -scale)};
    }
    std::vector<double> d(n), e(n, 0.0), Y((size_t)n * n, 0.0);
    std::vector<HostCplx> tau(n, HostCplx{0.0, 0.0});
    tridiagonalise(n, A, d, e, tau);
    for (int i = 0; i < n; ++i) Y[i + (size_t)i * n] = 1.0;
    const bool converged = diagonalise(n, d, e, Y);
    std::vector<int> order(n);
    std::iota(order.begin(), order.end(), 0);
    std::sort(order.begin(), order.end(), [&](int a, int b) { return d[a] < d[b]; });
    for (int j = 0; j < n; ++j) {
        w[j] = std::ldexp(d[order[j]], scale);
        HostCplx* z = &Z[(size_t)j * n];
        const double* y = &Y[(size_t)order[j] * n];
        for (int i = 0; i < n; ++i) z[i].re = y[i];
        for (int k = n - 2; k >= 0; --k) {  // z -= tau_k v_k (v_k^+ z)
            const HostCplx* v = &A[k + 1 + (size_t)k * n];
            HostCplx dot{0.0, 0.0};
            for (int i = 0; i < n - k - 1; ++i) {
                dot.re += v[i].re * z[k + 1 + i].re + v[i].im * z[k + 1 + i].im;
                dot.im += v[i].re * z[k + 1 + i].im - v[i].im * z[k + 1 + i].re;
            }
            subtract(n - k - 1, tau[k] * dot, v, z + k + 1);
        }
    }
    return converged;
}

namespace {
// Interpolation at the Chebyshev-Gauss nodes y_j = cos(theta_j), theta_j = pi (j + 1/2)/(n + 1),
// mapped to x_j = ((1 - eps) y_j + 1 + eps)/2 in [eps, 1].
template <typename F>
void cheb_interp(int n, double eps, F f, double* out) {
    const double pi = std::acos(-1.0);
    std::vector<double> fv(n + 1), th(n + 1);
    for (int j = 0; j <= n; ++j) {
        th[j] = pi * (j + 0.5) / (n + 1);
        fv[j] = f(((1.0 - eps) * std::cos(th[j]) + 1.0 + eps) / 2.0);
    }
    for (int k = 0; k <= n; ++k) {
        double s = 0.0;
        for (int j = 0; j <= n; ++j) s += fv[j] * std::cos(k * th[j]);
        out[k] = 2.0 * s / (n + 1);
    }
    out[0] *= 0.5;
}
}  // namespace

void host_chebyshev_coeffs(int n, double eps, double* out) {
    cheb_interp(n, eps, [](double x) { return 1.0 / std::sqrt(x); }, out);
}

void host_chebyshev_coeffs_shifted_inverse_root(int n, double eps, double a, double* out) {
    cheb_interp(n, eps, [a](double x) { return 1.0 / (a + std::sqrt(x)); }, out);
}

namespace {
// P(y) = sum_k c_k T_k(y) by Clenshaw.
double cheb_sum(const double* c, int n, double y) {
    double b1 = 0.0, b2 = 0.0;
    for (int k = n; k >= 1; --k) {
        const double b0 = c[k] + 2.0 * y * b1 - b2;
        b2 = b1;
        b1 = b0;
    }
    return c[0] + y * b1 - b2;
}

// Solve A z = r in place (A row-major m x m, destroyed; r becomes z); Gaussian elimination
// with partial pivoting.  False if A is singular to working precision.
bool lu_solve(int m, std::vector<double>& A, std::vector<double>& r) {
    for (int k = 0; k < m; ++k) {
        int piv = k;
        for (int i = k + 1; i < m; ++i)
            if (std::fabs(A[(size_t)i * m + k]) > std::fabs(A[(size_t)piv * m + k])) piv = i;
        if (!(std::fabs(A[(size_t)piv * m + k]) > 0.0)) return false;
        if (piv != k) {
            for (int j = 0; j < m; ++j) std::swap(A[(size_t)k * m + j], A[(size_t)piv * m + j]);
            std::swap(r[k], r[piv]);
        }
        const double inv = 1.0 / A[(size_t)k * m + k];
        for (int i = k + 1; i < m; ++i) {
            const double f = A[(size_t)i * m + k] * inv;
            if (f == 0.0) continue;
            double* ri = &A[(size_t)i * m];
            const double* rk = &A[(size_t)k * m];
            for (int j = k; j < m; ++j) ri[j] -= f * rk[j];
            r[i] -= f * r[k];
        }
    }
    for (int k = m - 1; k >= 0; --k) {
        double s = r[k];
        for (int j = k + 1; j < m; ++j) s -= A[(size_t)k * m + j] * r[j];
        r[k] = s / A[(size_t)k * m + k];
    }
    return true;
}
}  // namespace

double host_minimax_coeffs(int n, double eps, double* out) {
    // Remez exchange for min over P of max over [eps, 1] of |1 - sqrt(x) P(x)|, P = sum_k c_k T_k(y),
    // y = (2x - 1 - eps)/(1 - eps) = -cos(theta).  Reference: n + 2 angles; levelled system
    // sqrt(x_i) P(x_i) + s_i E = 1 with alternating s_i; next reference: the alternating extrema of
    // the error on a grid of 64 points per oscillation, each refined by a parabola in theta.
    const double pi = std::acos(-1.0);
    const int m = n + 2;
    std::vector<double> th(m), sg(m), c(n + 1, 0.0);
    for (int i = 0; i < m; ++i) {
        th[i] = pi * i / (n + 1);
        sg[i] = (i % 2 == 0) ? 1.0 : -1.0;
    }
    const int G = 64 * m;
    const double h = pi / G;
    auto err_at = [&](double t) {
        const double y = -std::cos(t);
        const double x = ((1.0 - eps) * y + 1.0 + eps) / 2.0;
        return 1.0 - std::sqrt(x) * cheb_sum(c.data(), n, y);
    };
    double delta = 1.0, last_gap = 1e300;
    std::vector<double> e(G + 1);
    for (int it = 0; it < 80; ++it) {
        std::vector<double> A((size_t)m * m), r(m, 1.0);
        for (int i = 0; i < m; ++i) {
            const double y = -std::cos(th[i]);
            const double sx = std::sqrt(((1.0 - eps) * y + 1.0 + eps) / 2.0);
            double t0 = 1.0, t1 = y;
            for (int k = 0; k <= n; ++k) {
                const double tk = (k == 0) ? 1.0 : (k == 1 ? y : 2.0 * y * t1 - t0);
                if (k >= 2) {
                    t0 = t1;
                    t1 = tk;
                }
                A[(size_t)i * m + k] = sx * tk;
            }
            A[(size_t)i * m + n + 1] = sg[i];
        }
        if (!lu_solve(m, A, r)) break;
        for (int k = 0; k <= n; ++k) c[k] = r[k];
        const double E = std::fabs(r[n + 1]);
        for (int j = 0; j <= G; ++j) e[j] = err_at(h * j);
        // extrema (ends included), refined, then reduced to an alternating sequence
        std::vector<double> at, av;
        for (int j = 0; j <= G; ++j) {
            const bool end = (j == 0 || j == G);
            if (!end && !((e[j] - e[j - 1]) * (e[j + 1] - e[j]) <= 0.0 && e[j] != e[j - 1])) continue;
            double t = h * j;
            if (!end) {
                const double den = e[j - 1] - 2.0 * e[j] + e[j + 1];
                if (den != 0.0) t += 0.5 * h * (e[j - 1] - e[j + 1]) / den;
            }
            const double v = err_at(t);
            if (!av.empty() && ((v > 0.0) == (av.back() > 0.0))) {
                if (std::fabs(v) > std::fabs(av.back())) {
                    at.back() = t;
                    av.back() = v;
                }
            } else {
                at.push_back(t);
                av.push_back(v);
            }
        }
        while ((int)at.size() > m) {
            if (std::fabs(av.front()) < std::fabs(av.back())) {
                at.erase(at.begin());
                av.erase(av.begin());
            } else {
                at.pop_back();
                av.pop_back();
            }
        }
        delta = 0.0;
        for (double v : av) delta = std::max(delta, std::fabs(v));
        if ((int)at.size() < m) break;
        for (int i = 0; i < m; ++i) {
            th[i] = at[i];
            sg[i] = av[i] > 0.0 ? 1.0 : -1.0;
        }
        // levelled: the gap between the largest error and E is at the rounding of the error
        // function (~1e-14 absolute at delta ~ 1e-10), so also stop once it no longer halves
        const double gap = (delta - E) / E;
        if (gap <= 1e-6 || (gap < 1e-3 && gap > 0.5 * last_gap)) break;
        last_gap = gap;
    }
    for (int k = 0; k <= n; ++k) out[k] = c[k];
    return delta;
}

double host_poly_delta(const double* coeffs, int n, double eps) {
    // max |1 - sqrt(x) P(x)| on a grid uniform in the Chebyshev angle (Clenshaw in FP64)
    const int ng = 4096;
    double worst = 0.0;
    for (int q = 0; q <= ng; ++q) {
        const double y = std::cos(3.141592653589793 * q / ng);
        double b1 = 0.0, b2 = 0.0;
        for (int k = n; k >= 1; --k) {
            const double b0 = coeffs[k] + 2.0 * y * b1 - b2;
            b2 = b1;
            b1 = b0;
        }
        const double P = coeffs[0] + y * b1 - b2;
        const double x = ((1.0 - eps) * y + 1.0 + eps) / 2.0;
        worst = std::max(worst, std::fabs(1.0 - std::sqrt(x) * P));
    }
    return worst;
}

}  // namespace ovl
