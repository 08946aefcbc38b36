// Host construction of grid, quadrature, finite differences, banded LU
// factors, influence/flux responses and base-flow profiles (FP64).
//
// Section 2.4 (Keuchel & Avila): N_r Chebyshev points with optional
// relaxation, high-order radial finite differences, Fourier modes in theta
// and z, influence-matrix wall conditions, flux forcing f_z (Eq. 2.7).
// Eq. 2.3-2.4: steady profile plus the Sexl-Womersley oscillation.
#include "setup.hpp"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>

namespace pnop {

using cd = std::complex<double>;

int parity_index(int m) { return (m % 2 == 0) ? 0 : 1; }

// ---------------------------------------------------------------- grid
static void radial_points(int nr, double stretch, std::vector<double>& r) {
    r.resize(nr);
    const double last = std::cos(M_PI * (nr - 1) / (2.0 * nr - 1.0));
    for (int j = 0; j < nr; ++j) {
        double x = std::cos(M_PI * j / (2.0 * nr - 1.0));
        double rho = 1.0 - j * (1.0 - last) / (nr - 1.0);
        r[j] = (1.0 - stretch) * x + stretch * rho;
    }
    r[0] = 1.0;
}

// Dense LU with partial pivoting (long double), solves A x = b in place.
static bool dense_solve(int n, std::vector<long double>& A, std::vector<long double>& b) {
    std::vector<int> piv(n);
    for (int c = 0; c < n; ++c) {
        int p = c;
        for (int i = c + 1; i < n; ++i)
            if (std::fabs(A[i * n + c]) > std::fabs(A[p * n + c])) p = i;
        if (A[p * n + c] == 0) return false;
        if (p != c) {
            for (int k = 0; k < n; ++k) std::swap(A[p * n + k], A[c * n + k]);
            std::swap(b[p], b[c]);
        }
        for (int i = c + 1; i < n; ++i) {
            long double f = A[i * n + c] / A[c * n + c];
            if (f == 0) continue;
            for (int k = c; k < n; ++k) A[i * n + k] -= f * A[c * n + k];
            b[i] -= f * b[c];
        }
    }
    for (int i = n - 1; i >= 0; --i) {
        long double s = b[i];
        for (int k = i + 1; k < n; ++k) s -= A[i * n + k] * b[k];
        b[i] = s / A[i * n + i];
    }
    return true;
}

// Quadrature for int_0^1 f r dr exact when f is a polynomial of degree < nr
// in s = r^2: half the interpolatory weights of int_0^1 ds on s_j = r_j^2,
// from the Chebyshev moment equations sum_j T_n(2 s_j - 1) w_j = mu_n.
static bool radial_quadrature(const std::vector<double>& r, std::vector<double>& W) {
    const int n = (int)r.size();
    std::vector<long double> A((size_t)n * n), b(n);
    for (int j = 0; j < n; ++j) {
        long double x = 2.0L * (long double)r[j] * (long double)r[j] - 1.0L;
        long double t0 = 1.0L, t1 = x;
        for (int k = 0; k < n; ++k) {
            long double tk = (k == 0) ? t0 : (k == 1 ? t1 : 0.0L);
            if (k >= 2) {
                tk = 2.0L * x * t1 - t0;
                t0 = t1;
                t1 = tk;
            }
            A[(size_t)k * n + j] = tk;
        }
    }
    for (int k = 0; k < n; ++k) b[k] = (k % 2 == 0) ? 1.0L / (1.0L - (long double)k * k) : 0.0L;
    if (!dense_solve(n, A, b)) return false;
    W.resize(n);
    for (int j = 0; j < n; ++j) W[j] = (double)(0.5L * b[j]);
    return true;
}

// Weights of the d-th derivative at x0 from 9 nodes: exactness on (x-x0)^p,
// p = 0..8, solved as a Vandermonde system in the scaled offsets.
static bool fd_weights(double x0, const double* x, int d, double* w) {
    const int n = kStencil;
    long double h = 0;
    for (int i = 0; i < n; ++i) h = std::max(h, std::fabs((long double)x[i] - x0));
    std::vector<long double> A((size_t)n * n), b(n, 0.0L);
    for (int p = 0; p < n; ++p)
        for (int i = 0; i < n; ++i) A[(size_t)p * n + i] = std::pow(((long double)x[i] - x0) / h, p);
    long double fact = 1;
    for (int q = 2; q <= d; ++q) fact *= q;
    b[d] = fact;
    if (!dense_solve(n, A, b)) return false;
    for (int i = 0; i < n; ++i) w[i] = (double)(b[i] / std::pow(h, d));
    return true;
}

bool build_grid(HostOps& h, std::string& err) {
    const Dims& d = h.d;
    const int nr = d.nr;
    radial_points(nr, d.stretch, h.r);
    h.invr.resize(nr);
    for (int j = 0; j < nr; ++j) h.invr[j] = 1.0 / h.r[j];
    if (!radial_quadrature(h.r, h.W)) {
        err = "radial quadrature system is singular";
        return false;
    }
    for (int j = 0; j < nr; ++j)
        if (!(h.W[j] > 0)) {
            err = "radial quadrature weight is not positive (stretch too large?)";
            return false;
        }
    // finite differences on the mirrored grid {r} U {-r}; a mirrored node
    // carries parity * f(r_i).  Rows near the wall are one-sided.
    std::vector<double> ext(2 * nr);
    for (int e = 0; e < nr; ++e) ext[e] = h.r[e];
    for (int e = nr; e < 2 * nr; ++e) ext[e] = -h.r[2 * nr - 1 - e];
    h.D1.assign((size_t)2 * nr * kBand, 0.0);
    h.D2.assign((size_t)2 * nr * kBand, 0.0);
    for (int j = 0; j < nr; ++j) {
        int lo = std::min(std::max(j - kStencil / 2, 0), 2 * nr - kStencil);
        double w1[kStencil], w2[kStencil];
        if (!fd_weights(h.r[j], &ext[lo], 1, w1) || !fd_weights(h.r[j], &ext[lo], 2, w2)) {
            err = "finite-difference system is singular";
            return false;
        }
        for (int pi = 0; pi < 2; ++pi) {
            const double par = pi == 0 ? 1.0 : -1.0;
            for (int t = 0; t < kStencil; ++t) {
                int e = lo + t;
                int col = e < nr ? e : 2 * nr - 1 - e;
                double sg = e < nr ? 1.0 : par;
                int s = col - j + kLo;
                if (s < 0 || s >= kBand) {
                    err = "stencil outside the stored band";
                    return false;
                }
                h.D1[((size_t)pi * nr + j) * kBand + s] += sg * w1[t];
                h.D2[((size_t)pi * nr + j) * kBand + s] += sg * w2[t];
            }
        }
    }
    return true;
}

// ---------------------------------------------------------------- Bessel / base flow
cd bessel_j(int nu, cd z) {
    cd half = 0.5 * z;
    cd term = 1.0;
    for (int i = 0; i < nu; ++i) term *= half / double(i + 1);
    cd sum = term;
    cd q = -half * half;
    for (int k = 1; k < 400; ++k) {
        term *= q / double(k * (k + nu));
        sum += term;
        if (std::abs(term) <= 1e-18 * std::max(std::abs(sum), 1e-300)) break;
    }
    return sum;
}

static void base_profiles(HostOps& h) {
    const int nr = h.d.nr;
    h.Uh.assign(nr, cd(0, 0));
    h.dUh.assign(nr, cd(0, 0));
    h.omega = h.ph.Wo * h.ph.Wo / h.ph.Re;
    if (h.ph.A == 0.0) return;
    const cd kappa = std::polar(h.ph.Wo, 0.75 * M_PI);
    const cd j0k = bessel_j(0, kappa), j1k = bessel_j(1, kappa);
    // bulk of the oscillation = (A/2) sin(omega t): B (1 - 2 J1/(kappa J0)) = -i A / 2
    const cd B = cd(0.0, -0.5 * h.ph.A) / (1.0 - 2.0 * j1k / (kappa * j0k));
    for (int j = 0; j < nr; ++j) {
        cd kr = kappa * h.r[j];
        h.Uh[j] = B * (1.0 - bessel_j(0, kr) / j0k);
        h.dUh[j] = B * kappa * bessel_j(1, kr) / j0k;
    }
}

// ---------------------------------------------------------------- banded LU
// Band row j holds columns j-4 .. j+8 at offsets 0..12.
struct Band {
    int n;
    std::vector<double> a;  // [n][kBand]
    double& at(int j, int col) { return a[(size_t)j * kBand + (col - j + kLo)]; }
    double get(int j, int col) const {
        int s = col - j + kLo;
        if (s < 0 || s >= kBand || col < 0 || col >= n) return 0.0;
        return a[(size_t)j * kBand + s];
    }
};

// Doolittle LU without pivoting.  Output per row: l[0..3] (columns j-4..j-1),
// 1/U_jj, U_{j,j+1..j+8}.
static bool band_lu(const Band& A, std::vector<double>& f, double& growth) {
    const int n = A.n;
    std::vector<double> U((size_t)n * (kUp + 1), 0.0);  // U[j][0..8] = U_{j,j..j+8}
    f.assign((size_t)n * kBand, 0.0);
    double amax = 0, umax = 0;
    for (double v : A.a) amax = std::max(amax, std::fabs(v));
    for (int j = 0; j < n; ++j) {
        double row[kLo + kUp + 1];  // columns j-4 .. j+8
        for (int s = 0; s < kBand; ++s) row[s] = A.get(j, j - kLo + s);
        for (int i = std::max(0, j - kLo); i < j; ++i) {
            double piv = U[(size_t)i * (kUp + 1)];
            double l = row[i - j + kLo] / piv;
            row[i - j + kLo] = 0.0;
            for (int c = i + 1; c <= std::min(n - 1, i + kUp); ++c) {
                int s = c - j + kLo;
                if (s >= kBand) {
                    if (U[(size_t)i * (kUp + 1) + (c - i)] != 0.0 && l != 0.0) return false;  // fill beyond band
                    continue;
                }
                row[s] -= l * U[(size_t)i * (kUp + 1) + (c - i)];
            }
            f[(size_t)j * kBand + (i - (j - kLo))] = l;
        }
        if (row[kLo] == 0.0) return false;
        for (int c = 0; c <= kUp; ++c) {
            double v = (j + c < n) ? row[kLo + c] : 0.0;
            U[(size_t)j * (kUp + 1) + c] = v;
            umax = std::max(umax, std::fabs(v));
        }
        f[(size_t)j * kBand + kLo] = 1.0 / row[kLo];
        for (int c = 1; c <= kUp; ++c) f[(size_t)j * kBand + kLo + c] = U[(size_t)j * (kUp + 1) + c];
    }
    growth = umax / std::max(amax, 1e-300);
    return true;
}

// Solve with factors f (real RHS, in place).
static void band_solve(int n, const std::vector<double>& f, std::vector<double>& x) {
    for (int j = 0; j < n; ++j) {
        double s = x[j];
        for (int e = 0; e < kLo; ++e) {
            int c = j - kLo + e;
            if (c >= 0) s -= f[(size_t)j * kBand + e] * x[c];
        }
        x[j] = s;
    }
    for (int j = n - 1; j >= 0; --j) {
        double s = x[j];
        for (int e = 1; e <= kUp; ++e) {
            int c = j + e;
            if (c < n) s -= f[(size_t)j * kBand + kLo + e] * x[c];
        }
        x[j] = s * f[(size_t)j * kBand + kLo];
    }
}

// Uniform numbers in [0, 1) (splitmix64; a generator with a large state costs more to
// seed than a banded solve)
struct Uniform {
    unsigned long long g;
    double operator()() {
        unsigned long long z = g += 0x9E3779B97F4A7C15ull;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return (double)((z ^ (z >> 31)) >> 11) * 0x1p-53;
    }
};

static double band_backward_error(const Band& A, const std::vector<double>& f, unsigned seed) {
    const int n = A.n;
    Uniform U{seed};
    std::vector<double> b(n), x;
    for (int j = 0; j < n; ++j) b[j] = 2.0 * U() - 1.0;
    x = b;
    band_solve(n, f, x);
    double rmax = 0, amax = 0, xmax = 0;
    for (int j = 0; j < n; ++j) {
        double s = -b[j], arow = 0;
        for (int c = std::max(0, j - kLo); c <= std::min(n - 1, j + kUp); ++c) {
            s += A.get(j, c) * x[c];
            arow += std::fabs(A.get(j, c));
        }
        rmax = std::max(rmax, std::fabs(s));
        amax = std::max(amax, arow);
        xmax = std::max(xmax, std::fabs(x[j]));
    }
    return rmax / (amax * xmax + 1e-300);
}

static void scatter_factors(RawVec& dst, int mat, int k, int nr, int ntile, int nc1,
                            const std::vector<double>& f) {
    for (int j = 0; j < nr; ++j)
        for (int e = 0; e < kBand; ++e) dst[fac_index(mat, k, j, e, nr, ntile, nc1)] = f[(size_t)j * kBand + e];
}

// Row-local coefficients of A^T = U^T L^T from the factors of A: row j holds
// U_{j-8+e, j} (e = 0..7, oldest first), 1/U_jj, L_{j+1+e, j} (e = 0..3).
static std::vector<double> transpose_factors(int nr, const std::vector<double>& f) {
    std::vector<double> t((size_t)nr * kBand, 0.0);
    for (int j = 0; j < nr; ++j) {
        for (int e = 0; e < 8; ++e) {
            const int i = j - 8 + e;  // U_{i, j} = f[i][4 + (j - i)]
            if (i >= 0) t[(size_t)j * kBand + e] = f[(size_t)i * kBand + kLo + (j - i)];
        }
        t[(size_t)j * kBand + 8] = f[(size_t)j * kBand + kLo];
        for (int e = 0; e < 4; ++e) {
            const int i = j + 1 + e;  // L_{i, j} = f[i][j - i + 4]
            if (i < nr) t[(size_t)j * kBand + 9 + e] = f[(size_t)i * kBand + (j - i + kLo)];
        }
    }
    return t;
}

// Unevaluated sums of two doubles (Dekker 1971, Knuth's two-sum; about 106 bits).
struct dd {
    double h = 0.0, l = 0.0;
};
static inline dd dd_norm(double h, double l) {  // |l| <= |h|
    const double s = h + l;
    return {s, l - (s - h)};
}
static inline dd dd_add(dd a, dd b) {
    const double s = a.h + b.h, v = s - a.h;
    return dd_norm(s, (a.h - (s - v)) + (b.h - v) + (a.l + b.l));
}
static inline dd dd_mul(dd a, dd b) {
    const double p = a.h * b.h;
    return dd_norm(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
static inline dd dd_neg(dd a) { return {-a.h, -a.l}; }
static inline dd dd_inv(dd a) {  // 1 / a, one Newton step
    const double q = 1.0 / a.h, r = std::fma(-q, a.h, 1.0) - q * a.l;
    return dd_norm(q, q * r);
}

// s + sum a_i x_i with the roundings of the products and sums carried along
static inline double dd_dot(double s, int n, const double* a, double sign, const dd* x) {
    double c = 0.0;
    for (int i = 0; i < n; ++i) {
        const double ai = sign * a[i], p = ai * x[i].h, t = s + p, z = t - s;
        c += ((s - (t - z)) + (p - z)) + std::fma(ai, x[i].h, -p) + ai * x[i].l;
        s = t;
    }
    return s + c;
}
// x <- A^-1 e_0 by the factors f of A and refinement with exact residuals, until a
// correction stays below the last bits of x.
static void unit_response(const Band& A, const std::vector<double>& f, std::vector<dd>& x) {
    const int n = A.n;
    std::vector<double> r(n, 0.0);
    r[0] = 1.0;
    band_solve(n, f, r);
    x.assign(n, dd{});
    for (int rounds = 0;; ++rounds) {
        double step = 0, size = 0;
        for (int j = 0; j < n; ++j) {
            x[j] = dd_add(x[j], {r[j], 0.0});
            step = std::max(step, std::fabs(r[j]));
            size = std::max(size, std::fabs(x[j].h));
        }
        if (rounds == 3 || (rounds && !(step > std::ldexp(size, -50)))) return;
        for (int j = 0; j < n; ++j) {
            const int lo = std::max(0, j - kLo), hi = std::min(n - 1, j + kUp);
            r[j] = dd_dot(j == 0 ? 1.0 : 0.0, hi - lo + 1, &A.a[(size_t)j * kBand + (lo - j + kLo)], -1.0, &x[lo]);
        }
        band_solve(n, f, r);
    }
}

// value in fixed point, as the two signed digits the device reads (low, high)
static double fx_bits(long long c) {
    if ((unsigned)(c & 0xFFFFFFFFll) == 0x80000000u) ++c;  // keeps the low digit above -2^31 (x_dot4's sums)
    const int lo = (int)(unsigned)(c & 0xFFFFFFFFll);
    const unsigned hi = (unsigned)(int)((c - lo) >> 32);
    const unsigned long long b = ((unsigned long long)hi << 32) | (unsigned)lo;
    double d;
    std::memcpy(&d, &b, sizeof d);
    return d;
}
static double fx_pair(int lo, int hi) {
    const unsigned long long b = ((unsigned long long)(unsigned)hi << 32) | (unsigned)lo;
    double d;
    std::memcpy(&d, &b, sizeof d);
    return d;
}
// v scale to the nearest integer, scale a power of two (halves away from zero)
static inline long long fx_near(double v) { return (long long)(v + std::copysign(0.5, v)); }
static inline long long fx_round(dd v, double scale) {
    const double h = v.h * scale;
    const long long c = std::fabs(h) < 4503599627370496.0 ? fx_near(h) : (long long)h;  // whole from 2^52 on
    return c + fx_near((h - (double)c) + v.l * scale);
}

// v scale as a number with 32 fractional bits: its integer part as two signed digits,
// the fraction as a third one
static double fx_bits(dd v, double scale, int& third) {
    long long c = (long long)(v.h * scale);
    long long f = fx_round({v.h * scale - (double)c, v.l * scale}, 4294967296.0);
    c += (f + (1ll << 31)) >> 32;
    f -= ((f + (1ll << 31)) >> 32) << 32;
    third = (int)f;
    const int lo = (int)(unsigned)(c & 0xFFFFFFFFll);
    return fx_pair(lo, (int)((c - lo) >> 32));
}

// The two-sided factorisation of one matrix (layout notes in setup.hpp), by
// positions: l[s][p][e] = N(p, p-4+e) for the outer columns, u[s][p][e] =
// U(p, p+1+e), d[s][p] = 1/D, all of side s, and the inverse of the middle block.
// Computed in sums of two doubles and rounded once, into the tables: in FP64 the
// elimination and the scaling by 1/D leave several roundings of 2^-53 in every
// factor, which the solver, rounding at 2^-54 and below, would repeat in every
// solve.
struct Twist {
    std::vector<dd> l[2], u[2], d[2];
    dd mid[8][8];  // S^-1 by rows h-4..h+3
};
// G <- G^-1 by Gauss-Jordan elimination with partial pivoting.  The
// solver multiplies by G instead of solving with S, which is as stable only if
// G is accurate far beyond the result: nearly singular matrices (the pressure
// of m = 0 and small k_z in a long pipe, condition number about Lz^2) cancel in
// G r as many bits as their condition number has.
static bool invert8(dd (&G)[8][8]) {
    int perm[8];
    for (int c = 0; c < 8; ++c) {
        int p = c;
        for (int i = c + 1; i < 8; ++i)
            if (std::fabs(G[i][c].h) > std::fabs(G[p][c].h)) p = i;
        if (G[p][c].h == 0.0 || !std::isfinite(G[p][c].h)) return false;
        perm[c] = p;
        for (int j = 0; j < 8 && p != c; ++j) std::swap(G[p][j], G[c][j]);
        const dd inv = dd_inv(G[c][c]);
        G[c][c] = {1.0, 0.0};
        for (int j = 0; j < 8; ++j) G[c][j] = dd_mul(G[c][j], inv);
        for (int i = 0; i < 8; ++i) {
            if (i == c) continue;
            const dd m = dd_neg(G[i][c]);
            G[i][c] = dd{};
            for (int j = 0; j < 8; ++j) G[i][j] = dd_add(G[i][j], dd_mul(m, G[c][j]));
        }
    }
    for (int c = 7; c >= 0; --c)  // the row exchanges, undone as column exchanges
        for (int i = 0; i < 8 && perm[c] != c; ++i) std::swap(G[i][c], G[i][perm[c]]);
    return true;
}
static bool twist_factor(const Band& A, const FxShape& f, Twist& t) {
    const int n = A.n, h = f.h, B = 8, W = 2 * B + 1;
    thread_local std::vector<dd> w;
    w.assign((size_t)n * W, dd{});
    auto at = [&](int i, int j) -> dd& { return w[(size_t)i * W + (j - i + B)]; };
    for (int i = 0; i < n; ++i)
        for (int j = std::max(0, i - kLo); j <= std::min(n - 1, i + kUp); ++j) at(i, j).h = A.get(i, j);
    for (int s = 0; s < 2; ++s) {
        const int np = 4 * f.chunks[s], pad = s ? f.pad : 0;
        t.l[s].assign((size_t)np * 4, dd{});
        t.u[s].assign((size_t)np * 8, dd{});
        t.d[s].assign(np, dd{});
        auto row = [&](int p) { return s ? n - 1 - (p - pad) : p; };
        for (int p = pad; p < np - 4; ++p) {
            const int i = row(p);
            const dd piv = at(i, i);
            if (piv.h == 0.0 || !std::isfinite(piv.h)) return false;
            const dd inv = t.d[s][p] = dd_inv(piv);
            for (int e = 0; e < 8; ++e) {
                const int q = p + 1 + e, j = row(q);
                if (j < 0 || j >= n) break;
                const dd v = at(i, j);
                if (v.h != 0.0 && e >= 4 && (s || p > 3 || q > 8)) return false;
                t.u[s][(size_t)p * 8 + e] = dd_mul(v, inv);
            }
            for (int q = p + 1; q <= p + 4; ++q) {
                const int j = row(q);
                const dd m = dd_mul(at(j, i), inv);
                t.l[s][(size_t)q * 4 + (p - q + 4)] = m;
                if (m.h == 0.0) continue;
                const dd neg = dd_neg(m);
                for (int c = 1; c <= 8; ++c) {
                    const int k = row(p + c);
                    if (k < 0 || k >= n || std::abs(k - j) > B) break;
                    if (at(i, k).h != 0.0) at(j, k) = dd_add(at(j, k), dd_mul(neg, at(i, k)));
                }
            }
        }
    }
    for (int i = 0; i < 8; ++i)
        for (int j = 0; j < 8; ++j) t.mid[i][j] = at(h - 4 + i, h - 4 + j);
    return invert8(t.mid);
}
// positions of a side's half of the middle as rows of the block: own, then the other side's
static int mid_row(int s, int i) { return i < 4 ? (s ? 7 - i : i) : (s ? i - 4 : 11 - i); }

// Backward error of the two-sided solve of A x = b, by rows (Oettli and Prager
// 1964): the residual over |A||x| + |b|.  b = A x for a random x of order one: the
// solution of a random b would lie along the null vector of a nearly singular
// matrix, beside which whatever the middle block loses disappears.
static double twist_backward_error(const Band& A, const FxShape& f, const Twist& t, unsigned seed) {
    const int n = A.n;
    std::vector<double> b(n, 0.0), x(n);
    Uniform U{seed};
    for (double& v : x) v = 0.5 + U();
    for (int j = 0; j < n; ++j)
        for (int c = std::max(0, j - kLo); c <= std::min(n - 1, j + kUp); ++c) b[j] += A.get(j, c) * x[c];
    double mid[8];
    std::vector<double> y[2];
    for (int s = 0; s < 2; ++s) {
        const int np = 4 * f.chunks[s], pad = s ? f.pad : 0;
        y[s].assign(np, 0.0);
        for (int p = pad; p < np; ++p) {
            double v = b[s ? n - 1 - (p - pad) : p];
            for (int e = 0; e < 4; ++e)
                if (p - 4 + e >= 0) v -= t.l[s][(size_t)p * 4 + e].h * y[s][p - 4 + e];
            y[s][p] = v;
        }
        for (int i = 0; i < 4; ++i) mid[mid_row(s, i)] = y[s][np - 4 + i];
    }
    for (int s = 0; s < 2; ++s) {
        const int np = 4 * f.chunks[s], pad = s ? f.pad : 0;
        std::vector<double> xs(np + 8, 0.0);
        for (int i = 0; i < 4; ++i) {
            dd v;
            for (int c = 0; c < 8; ++c) v = dd_add(v, dd_mul(t.mid[mid_row(s, i)][c], {mid[c], 0.0}));
            xs[np - 4 + i] = v.h;
        }
        for (int p = np - 5; p >= pad; --p) {
            double v = y[s][p] * t.d[s][p].h;
            for (int e = 0; e < 8; ++e) v -= t.u[s][(size_t)p * 8 + e].h * xs[p + 1 + e];
            xs[p] = v;
        }
        for (int p = pad; p < np; ++p) x[s ? n - 1 - (p - pad) : p] = xs[p];
    }
    double worst = 0;
    for (int j = 0; j < n; ++j) {
        double r = -b[j], arow = std::fabs(b[j]) + 1e-300;
        for (int c = std::max(0, j - kLo); c <= std::min(n - 1, j + kUp); ++c) {
            r += A.get(j, c) * x[c];
            arow += std::fabs(A.get(j, c) * x[c]);
        }
        worst = std::max(worst, std::fabs(r) / arow);
        if (!std::isfinite(r)) return 1.0;
    }
    return worst;
}

// Largest row sum of the multipliers of one factorisation (column 0 apart,
// which is scaled to at most 1), and the largest entry of that column.
static void fx_measure(const FxShape& f, const Twist& t, double& sum, double& col0) {
    for (int s = 0; s < 2; ++s) {
        const int np = 4 * f.chunks[s];
        for (int p = 0; p < np; ++p) {
            double l = 0, u = 0, lt = 0, ut = 0;  // rows and columns of N and U
            for (int e = 0; e < 4; ++e) {
                const double a = std::fabs(t.l[s][(size_t)p * 4 + e].h);
                const bool first = s == 0 && p - 4 + e == 0;
                if (first) col0 = std::max(col0, a);
                l += first ? std::min(a, 1.0) : a;
                if (p + 1 + e < np) {
                    const double b = std::fabs(t.l[s][(size_t)(p + 1 + e) * 4 + 3 - e].h);
                    lt += s == 0 && p == 0 ? std::min(b, 1.0) : b;
                }
            }
            for (int e = 0; e < 8; ++e) {
                u += std::fabs(t.u[s][(size_t)p * 8 + e].h);
                if (p - 1 - e >= 0) ut += std::fabs(t.u[s][(size_t)(p - 1 - e) * 8 + e].h);
            }
            const double worst = std::max(std::max(l, u), std::max(lt, ut));
            if (!(worst <= sum)) sum = worst;  // NaN included
        }
    }
}

// Writes a factorisation into the tables at (mat, k).  False when 1/D or S^-1 is
// outside the range of its format.
static bool fx_write(FixedTable& tab, int mat, int k, int nht, const FxShape& f, const Twist& t) {
    const size_t base = ((size_t)mat * nht + k / kTileX) * f.tile, kk = k % kTileX;
    const double one = std::ldexp(1.0, kFxBits), col0 = std::ldexp(1.0, kFxBits - tab.shift);
    auto mult = [&](dd v, double scale) { return fx_bits(fx_round(dd_neg(v), scale)); };
    auto pair = [&](size_t row, int e) { return ((row * 2 + e / 2) * kTileX + kk) * 2 + e % 2; };
    for (int s = 0; s < 2; ++s) {
        const int np = 4 * f.chunks[s];
        auto L = [&](int p, int q) {  // N(p, q), q < p
            const bool first = s == 0 && q == 0;
            return q < 0 || p >= np ? 0.0 : mult(t.l[s][(size_t)p * 4 + (q - p + 4)], first ? col0 : one);
        };
        auto U = [&](int p, int q) { return p < 0 || q >= np ? 0.0 : mult(t.u[s][(size_t)p * 8 + (q - p - 1)], one); };
        for (int p = 0; p < np; ++p) {
            const size_t in = base + f.in[s], out = base + f.out[s] + (size_t)(p / 4) * 20 * kTileX;
            for (int e = 0; e < 4; ++e) {
                // the middle rows couple inwards through S alone
                const int q = p - 4 + e;
                const bool inner = q >= np - 4;
                tab.direct[in + pair(p, e)] = inner ? 0.0 : L(p, q);
                tab.transposed[in + pair(p, e)] = inner ? 0.0 : U(q, p);
                if (p < np - 4) {
                    tab.direct[out + pair(p % 4, e)] = U(p, p + 1 + e);
                    tab.transposed[out + pair(p % 4, e)] = L(p + 1 + e, p);
                }
            }
        }
        // 1/D = D' 2^(q - 60), D' of at most 62 bits.  The rows of a chunk of four share
        // q, two bits of q + 128 being the lowest bits of each row's D', except in the
        // first chunk (the wall row), where all eight are the low byte.  The bits above
        // are rounded for these to be part of the value: 2^-54 of 1/D at most, down to
        // rows 2^6 below the largest of their chunk.
        for (int p = 0; p < np - 4;) {
            const int end = p < 4 ? p + 1 : p + 4;
            int lo = 1 << 20, hi = -(1 << 20);
            for (int i = p; i < end; ++i) {
                int q = 0;
                std::frexp(t.d[s][i].h, &q);
                if (t.d[s][i].h == 0.0) continue;  // empty position
                lo = std::min(lo, q);
                hi = std::max(hi, q);
            }
            if (lo > hi) lo = hi = 0;
            const int q = hi - 2;
            if (hi - lo > 6 || q < -127 || q > 127) return false;
            const double unit = std::ldexp(1.0, 60 - q);
            for (; p < end; ++p) {
                const int bits = p < 4 ? 8 : 2, code = p < 4 ? q + 128 : ((q + 128) >> 2 * (p % 4)) & 3;
                const long long scaled = fx_round(t.d[s][p], unit) - code + (1 << bits >> 1);
                const long long c = ((scaled >> bits) << bits) + code;
                const int low = (int)(unsigned)(c & 0xFFFFFFFFll);
                const size_t o = base + f.out[s] + (size_t)(p / 4) * 20 * kTileX + (16 + p % 4) * kTileX + kk;
                tab.direct[o] = tab.transposed[o] = fx_pair(low, (int)((c - low) >> 32));
            }
        }
        // S^-1 scaled by a power of two to row sums of at most 1, with 32 further
        // fractional bits in a third digit
        for (int tr = 0; tr < 2; ++tr) {
            auto& dst = tr ? tab.transposed : tab.direct;
            auto entry = [&](int i, int c) {  // row i of this side, column c: own rows, then the other side's
                const int a = mid_row(s, i), b = mid_row(s, c);
                return tr ? t.mid[b][a] : t.mid[a][b];
            };
            double sum = 0;
            for (int i = 0; i < 4; ++i) {
                double r = 0;
                for (int c = 0; c < 8; ++c) r += std::fabs(entry(i, c).h);
                if (!(r <= sum)) sum = r;
            }
            int q = 0;
            if (!std::isfinite(sum) || sum == 0.0) return false;
            std::frexp(sum, &q);
            if (q < -900 || q > 900) return false;
            const size_t o = base + f.mid[s];
            const double unit = std::ldexp(1.0, kFxBits - q);
            for (int i = 0; i < 4; ++i)
                for (int c = 0; c < 8; c += 2) {
                    int third[2];
                    for (int e = 0; e < 2; ++e)
                        dst[o + ((size_t)(i * 4 + c / 2) * kTileX + kk) * 2 + e] =
                            fx_bits(entry(i, c + e), unit, third[e]);
                    dst[o + ((size_t)(32 + i * 4 + c / 2) * kTileX) + kk] = fx_pair(third[0], third[1]);
                }
            dst[o + 48 * kTileX + kk] = fx_pair(q, 0);
        }
    }
    for (int i = 0; i < 4; ++i)
        for (int e = 0; e < 4; ++e) {  // U(i, 5 + e), the part beyond four columns
            const int c = 5 + e;
            const double v = c - i > 4 ? mult(t.u[0][(size_t)i * 8 + (c - i - 1)], one) : 0.0;
            tab.direct[base + f.wall + (size_t)(i * 4 + e) * kTileX + kk] = v;
            tab.transposed[base + f.wall + (size_t)(e * 4 + i) * kTileX + kk] = v;
        }
    return true;
}

static Band laplacian_band(const HostOps& h, int mabs, double kz) {
    const int nr = h.d.nr;
    Band L{nr, std::vector<double>((size_t)nr * kBand, 0.0)};
    for (int j = 0; j < nr; ++j)
        for (int s = 0; s < kBand; ++s) L.a[(size_t)j * kBand + s] = h.Lb[((size_t)mabs * nr + j) * kBand + s];
    for (int j = 0; j < nr; ++j) L.at(j, j) -= kz * kz;
    return L;
}

static Band helmholtz_band(const HostOps& h, int mabs, double kz) {
    const int nr = h.d.nr;
    Band A = laplacian_band(h, mabs, kz);
    const double c = -1.0 / (2.0 * h.ph.Re);
    for (double& v : A.a) v *= c;
    for (int j = 0; j < nr; ++j) A.at(j, j) += 1.0 / h.ph.dt;
    for (int s = 0; s < kBand; ++s) A.a[s] = 0.0;
    A.at(0, 0) = 1.0;  // Dirichlet row
    return A;
}

static Band pressure_band(const HostOps& h, int mabs, double kz) {
    const int nr = h.d.nr;
    Band A = laplacian_band(h, mabs, kz);
    const int pi = parity_index(mabs);
    for (int s = 0; s < kBand; ++s) A.a[s] = h.D1[((size_t)pi * nr + 0) * kBand + s];  // Neumann row
    return A;
}

// fn(i, thread) for i = 0..n-1 on up to 16 host threads; fn touches only data of its own i.
template <class F> static void parallel_k(int n, F&& fn) {
    const int T = std::max(1, std::min<int>({n, 16, (int)std::max(1u, std::thread::hardware_concurrency())}));
    if (T == 1) {
        for (int k = 0; k < n; ++k) fn(k, 0);
        return;
    }
    std::vector<std::thread> th;
    for (int t = 0; t < T; ++t)
        th.emplace_back([&, t] {
            for (int k = t; k < n; k += T) fn(k, t);
        });
    for (auto& x : th) x.join();
}

// Factors nmat matrices per k: calls each(ma, k, f) with the LU factors (FP64,
// without pivoting; worst: its largest backward error) and fills the device
// tables, in fixed point where every row of every matrix fits and the two-sided
// elimination is as stable as the LU has to be, else in FP64.  Work is split by
// (matrix, table tile), so that a host thread writes whole tiles.  False when a
// LU breaks down.
template <class F, class E>
static bool factor_tables(const HostOps& h, FixedTable& t, RawVec& fac, RawVec& facT,
                          int nmat, F&& matrix, E&& each, double& worst) {
    const int nr = h.d.nr, nk = h.d.nk, nht = (nk + kTileX - 1) / kTileX;
    const FxShape shape = fx_shape(nr);
    auto kz = [&](int k) { return 2.0 * M_PI * k / h.d.Lz; };
    t.ok = nr >= kFxMinRows && std::max(shape.chunks[0], shape.chunks[1]) <= kFxMaxChunks;
    t.shift = 0;
    fac.clear();
    facT.clear();
    t.direct.clear();
    t.transposed.clear();
    if (t.ok) {
        // column 0 of N is column 0 of A over the wall row's diagonal: the
        // wall-side rows of A off its diagonal depend on neither m (but for its
        // parity, which does not reach them) nor k
        const Band A = matrix(std::min(1, nmat - 1), kz(0));
        double col = 0;
        for (int j = 1; j <= kLo; ++j) col = std::max(col, std::fabs(A.get(j, 0) / A.get(0, 0)));
        if (std::isfinite(col))
            while (std::ldexp(col, -t.shift) > 1.0) ++t.shift;
        t.direct.resize((size_t)nmat * nht * shape.tile);
        t.transposed.resize(t.direct.size());
    }
    std::vector<double> err_t(16, 0.0), sum(16, 0.0), col(16, 0.0);
    std::vector<int> fail(16, 0), unfit(16, 0);
    parallel_k(nmat * nht, [&](int item, int th) {
        const int ma = item / nht, k0 = item % nht * kTileX;
        std::vector<double> f;
        Twist w;
        double growth = 0;
        for (RawVec* v : {&t.direct, &t.transposed})
            if (t.ok) std::fill_n(v->begin() + (size_t)item * shape.tile, shape.tile, 0.0);
        for (int k = k0; k < std::min(nk, k0 + kTileX) && !fail[th]; ++k) {
            const Band A = matrix(ma, kz(k));
            if (!band_lu(A, f, growth)) {
                fail[th] = 1;
                return;
            }
            err_t[th] = std::max(err_t[th], band_backward_error(A, f, 1234u + ma * 977u + k));
            each(ma, k, A, f);
            if (!t.ok || unfit[th]) continue;
            if (!twist_factor(A, shape, w) || !(twist_backward_error(A, shape, w, 99u + ma * 977u + k) < kFxBackward)) {
                unfit[th] = 1;
                continue;
            }
            fx_measure(shape, w, sum[th], col[th]);
            if (!(sum[th] <= kFxRowSum) || !(std::ldexp(col[th], -t.shift) <= 1.0) ||
                !fx_write(t, ma, k, nht, shape, w))
                unfit[th] = 1;
        }
    });
    bool ok = t.ok;
    for (int th = 0; th < 16; ++th) {
        if (fail[th]) return false;
        ok = ok && !unfit[th];
        worst = std::max(worst, err_t[th]);
    }
    t.ok = ok;
    if (ok) return true;
    t = FixedTable{};
    const int nt = h.ntile;
    const size_t tile = (size_t)nr * kBand * kTileK;
    fac.resize((size_t)nmat * nt * tile);
    facT.resize(fac.size());
    parallel_k(nmat * nt, [&](int item, int) {
        const int ma = item / nt, k0 = item % nt * kTileK;
        for (RawVec* v : {&fac, &facT}) std::fill_n(v->begin() + (size_t)item * tile, tile, 0.0);
        std::vector<double> f;
        double growth = 0;
        for (int k = k0; k < std::min(nk, k0 + kTileK); ++k) {
            band_lu(matrix(ma, kz(k)), f, growth);
            scatter_factors(fac, ma, k, nr, nt, kNc1Direct, f);
            scatter_factors(facT, ma, k, nr, nt, kNc1Transposed, transpose_factors(nr, f));
        }
    });
    return true;
}

bool build_operators(HostOps& h, std::string& err, bool reuse_pressure) {
    const Dims& d = h.d;
    const int nr = d.nr, nk = d.nk, M = d.M;
    if (!(h.ph.Re > 0) || !(h.ph.dt > 0)) {
        err = "Re and dt must be positive";
        return false;
    }
    base_profiles(h);
    // L band for |m'| = 0..M+1: D2 + D1/r - m'^2/r^2, parity of m'
    h.Lb.assign((size_t)(M + 2) * nr * kBand, 0.0);
    for (int ma = 0; ma <= M + 1; ++ma) {
        const int pi = parity_index(ma);
        for (int j = 0; j < nr; ++j) {
            for (int s = 0; s < kBand; ++s) {
                size_t src = ((size_t)pi * nr + j) * kBand + s;
                h.Lb[((size_t)ma * nr + j) * kBand + s] = h.D2[src] + h.invr[j] * h.D1[src];
            }
            h.Lb[((size_t)ma * nr + j) * kBand + kLo] -= (double)ma * ma * h.invr[j] * h.invr[j];
        }
    }
    h.ntile = (nk + kTileK - 1) / kTileK;
    double worst = 0;
    // Pressure factors, and the pressure phi of a unit wall datum with its radial
    // derivative for every (|m|, k): they depend on the grid only, a caller that
    // built them for this grid before may keep them.  They are as accurate as the
    // solver's tables (an LU alone leaves 2^-53 times the condition number, about
    // Lz^2 for m = 0, k = 1, and the wall correction would not match the solves).
    const size_t sys = (size_t)(M + 1) * nk * nr;
    auto at = [&](int ma, int k) { return ((size_t)ma * nk + k) * nr; };
    if (!(reuse_pressure && h.phi.size() == sys)) {
        h.phi.assign(sys, 0.0);
        h.dphi.assign(sys, 0.0);
        const bool done = factor_tables(
            h, h.fxP, h.facP, h.facPT, M + 1,
            [&](int ma, double kz) {
                if (ma || kz != 0.0) return pressure_band(h, ma, kz);
                Band I{nr, std::vector<double>((size_t)nr * kBand, 0.0)};  // singular mean mode: never used (p = 0)
                for (int j = 0; j < nr; ++j) I.at(j, j) = 1.0;
                return I;
            },
            [&](int ma, int k, const Band& A, const std::vector<double>& f) {
                if (ma == 0 && k == 0) return;
                thread_local std::vector<dd> x;
                unit_response(A, f, x);
                for (int j = 0; j < nr; ++j) {
                    const int lo = std::max(0, j - kLo), hi = std::min(nr - 1, j + kUp);
                    const double* row = &h.D1[((size_t)parity_index(ma) * nr + j) * kBand + (lo - j + kLo)];
                    h.phi[at(ma, k) + j] = x[j].h;
                    h.dphi[at(ma, k) + j] = dd_dot(0.0, hi - lo + 1, row, 1.0, &x[lo]);
                }
            },
            worst);
        if (!done) {
            err = "pressure band LU failed";
            return false;
        }
    }
    // Helmholtz factors, and the Helmholtz responses to -grad(phi) with u = 0 at
    // the wall: u+ and u- of m >= 0 (those of -m are the other one's of m) and
    // the imaginary part of u_z.
    std::vector<double> hp(sys, 0.0), hm(sys, 0.0), hz(sys, 0.0);
    const bool done = factor_tables(
        h, h.fxH, h.facH, h.facHT, M + 2, [&](int ma, double kz) { return helmholtz_band(h, ma, kz); },
        [&](int mu, int k, const Band&, const std::vector<double>& f) {
            const double kz = 2.0 * M_PI * k / d.Lz;
            std::vector<double> x(nr);
            auto solve = [&](int m, int kind, std::vector<double>& to) {  // kind +1, -1: u+-, 0: u_z
                if (m < 0 || m > M || (m == 0 && k == 0)) return;
                const double *phi = &h.phi[at(m, k)], *dphi = &h.dphi[at(m, k)];
                for (int j = 0; j < nr; ++j)
                    x[j] = kind == 0 ? -kz * phi[j] : -dphi[j] + kind * m * h.invr[j] * phi[j];
                x[0] = 0.0;
                band_solve(nr, f, x);
                std::copy(x.begin(), x.end(), to.begin() + at(m, k));
            };
            solve(mu - 1, 1, hp);
            solve(mu + 1, -1, hm);
            if (mu == 1) solve(0, -1, hm);
            solve(mu, 0, hz);
        },
        worst);
    if (!done) {
        err = "Helmholtz band LU failed";
        return false;
    }
    if (!(worst < 1e-12)) {
        char buf[160];
        std::snprintf(buf, sizeof buf, "banded LU without pivoting is unstable here (backward error %.3g)", worst);
        err = buf;
        return false;
    }
    // influence responses, stored scaled by -1/delta, delta = d/dr(h_r) at the
    // wall; k fastest, [im][component][j][k], so that the device reads them
    // coalesced across the k of a block
    h.infl.assign((size_t)d.nm * nk * 3 * nr, 0.0);
    std::vector<int> zero_t(16, 0);
    const int nkt = (nk + kTileX - 1) / kTileX;
    parallel_k((M + 1) * nkt, [&](int item, int t) {
        const int m = item / nkt, k0 = item % nkt * kTileX, pv = parity_index(m + 1);
        for (int k = k0; k < std::min(nk, k0 + kTileX); ++k) {
            if (m == 0 && k == 0) continue;
            const double *fp = &hp[at(m, k)], *fm = &hm[at(m, k)], *fz = &hz[at(m, k)];
            double delta = 0;
            for (int c = 0; c <= kUp && c < nr; ++c)
                delta += h.D1[((size_t)pv * nr + 0) * kBand + (c + kLo)] * (0.5 * (fp[c] + fm[c]));
            if (!(std::fabs(delta) > 1e-300) || !std::isfinite(delta)) {
                zero_t[t] = 1;
                return;
            }
            for (int side = 0; side < (m ? 2 : 1); ++side) {
                double* out = &h.infl[(size_t)(side ? M - m : M + m) * 3 * nr * nk + k];
                for (int j = 0; j < nr; ++j) {
                    const double ht = -0.5 * (fp[j] - fm[j]);
                    out[(size_t)j * nk] = -(0.5 * (fp[j] + fm[j])) / delta;
                    out[((size_t)nr + j) * nk] = (side ? ht : -ht) / delta;
                    out[((size_t)2 * nr + j) * nk] = -fz[j] / delta;
                }
            }
        }
    });
    for (int t = 0; t < 16; ++t)
        if (zero_t[t]) {
            err = "influence response has zero wall divergence";
            return false;
        }
    // flux response of mode (0,0): Helmholtz of u_z with unit forcing
    {
        std::vector<double> f;
        double growth = 0;
        band_lu(helmholtz_band(h, 0, 0.0), f, growth);
        h.fluxg.assign(nr, 1.0);
        h.fluxg[0] = 0.0;
        band_solve(nr, f, h.fluxg);
        double s = 0;
        for (int j = 0; j < nr; ++j) s += h.W[j] * h.fluxg[j];
        h.flux_inv = 1.0 / s;
    }
    return true;
}

// ---------------------------------------------------------------- checkpoint counts
long long binom_beta(int s, long long t) {
    if (t < 0) return 0;
    // C(s + t, s) = C(s + t, t) with saturation, over the shorter product
    const long long a = std::max<long long>(s, t), b = std::min<long long>(s, t);
    long double v = 1;
    for (long long i = 1; i <= b; ++i) {
        v = v * (long double)(a + i) / (long double)i;
        if (v > 4.0e18L) return (long long)4e18;
    }
    return (long long)(v + 0.5L);
}

bool build_projection(const HostOps& h, std::vector<double>& L, std::string& err) {
    const int nr = h.d.nr, M = h.d.M, nk = h.d.nk, B = kProjBand, W1 = B + 1;
    // A_par = D_r W^-1 D_r^T over the columns i >= 1, banded, for both parities
    std::vector<double> A[2];
    for (int par = 0; par < 2; ++par) {
        A[par].assign((size_t)nr * W1, 0.0);  // A[j][j' - j + B] for j' in [j - B, j]
        std::vector<std::vector<std::pair<int, double>>> col(nr);  // column i: (row j, D_r(j, i))
        for (int j = 0; j < nr; ++j)
            for (int e = 0; e < kBand; ++e) {
                const int i = j - kLo + e;
                if (i < 1 || i >= nr) continue;
                double v = h.D1[((size_t)par * nr + j) * kBand + e];
                if (i == j) v += h.invr[j];
                if (v != 0.0) col[i].push_back({j, v});
            }
        for (int i = 1; i < nr; ++i)
            for (auto& a : col[i])
                for (auto& b : col[i]) {
                    if (b.first > a.first) continue;
                    if (a.first - b.first > B) {
                        err = "admissible projection: divergence stencil wider than the factor band";
                        return false;
                    }
                    A[par][(size_t)a.first * W1 + (b.first - a.first + B)] += a.second * b.second / h.W[i];
                }
    }
    L.assign((size_t)(M + 1) * nk * nr * W1, 0.0);
    std::vector<double> S((size_t)nr * W1);
    for (int ma = 0; ma <= M; ++ma) {
        const int par = parity_index(ma + 1);
        for (int k = 0; k < nk; ++k) {
            if (ma == 0 && k == 0) continue;  // mean mode: diagonal constraints, no factor
            const double kz = 2.0 * M_PI * k / h.d.Lz;
            S = A[par];
            for (int j = 1; j < nr; ++j)
                S[(size_t)j * W1 + B] += ((double)ma * ma * h.invr[j] * h.invr[j] + kz * kz) / h.W[j];
            double* F = &L[(((size_t)ma * nk + k) * nr) * W1];
            for (int j = 0; j < nr; ++j) {
                for (int i = std::max(0, j - B); i <= j; ++i) {
                    double v = S[(size_t)j * W1 + (i - j + B)];
                    for (int q = std::max(0, j - B); q < i; ++q)
                        if (q >= i - B) v -= F[(size_t)j * W1 + (q - j + B)] * F[(size_t)i * W1 + (q - i + B)];
                    if (i < j) {
                        F[(size_t)j * W1 + (i - j + B)] = v * F[(size_t)i * W1 + B];
                    } else {
                        if (!(v > 0) || !std::isfinite(v)) {
                            err = "admissible projection: constraint system is not positive definite";
                            return false;
                        }
                        F[(size_t)j * W1 + B] = 1.0 / std::sqrt(v);
                    }
                }
            }
        }
    }
    return true;
}

int revolve_repetitions(long long nsteps, int snaps) {
    int r = 0;
    while (binom_beta(snaps, r) < nsteps) ++r;
    return r;
}

long long revolve_advances(long long nsteps, int snaps) {
    if (nsteps <= 1) return 0;
    int r = revolve_repetitions(nsteps, snaps);
    return (long long)r * nsteps - binom_beta(snaps + 1, r - 1);
}

}  // namespace pnop
