// FP64 spherical basis functions on the device (Sec. 3.3.1, Eq. shft0):
//   R_n^m(r) = j_n(k|r|) Y_n^m(theta, phi),  S_n^m = h_n Y_n^m,
//   Y_n^m = sqrt((2n+1)/(4pi) (n-|m|)!/(n+|m|)!) P_n^{|m|}(cos theta) e^{i m phi}
// with P_n^{|m|} free of the Condon-Shortley phase (so Y_n^{-m} = conj Y_n^m).
// Coefficient vectors use the flat index n^2 + n + m.
#pragma once

#include "quad.cuh"

__device__ __forceinline__ int nm_idx(int n, int m) { return n * n + n + m; }

// a_n^m and b_n^m of the translation recursions (zero outside their range).
__device__ __forceinline__ double coef_a(int n, int m) {
    int am = abs(m);
    if (n < am || n < 0) return 0.0;
    return sqrt((double)((n + 1 + am) * (n + 1 - am)) / (double)((2 * n + 1) * (2 * n + 3)));
}
__device__ __forceinline__ double coef_b(int n, int m) {
    if (n < 0 || abs(m) > n) return 0.0;
    double v = sqrt((double)((n - m - 1) * (n - m)) / (double)((2 * n - 1) * (2 * n + 1)));
    return m >= 0 ? v : -v;
}

// Normalised associated Legendre functions (no Condon-Shortley phase) for
// n < P at x = cos theta, s = sin theta: out[n(n+1)/2 + m], 0 <= m <= n.
//   Q_0^0 = 1/sqrt(4pi);  Q_m^m = sqrt((2m+1)/(2m)) s Q_{m-1}^{m-1};
//   Q_{m+1}^m = sqrt(2m+3) x Q_m^m;
//   Q_n^m = A x Q_{n-1}^m - B Q_{n-2}^m,
//     A = sqrt((4n^2-1)/(n^2-m^2)),  B = sqrt(((n-1)^2-m^2)(2n+1)/((2n-3)(n^2-m^2))).
__device__ inline void legendre_q(int P, double x, double s, double* out) {
    out[0] = 0.28209479177387814347;   // 1/sqrt(4 pi)
    double diag = out[0];
    for (int m = 0; m < P; ++m) {
        if (m > 0) {
            diag *= sqrt((2.0 * m + 1.0) / (2.0 * m)) * s;
            out[m * (m + 1) / 2 + m] = diag;
        }
        if (m + 1 < P) out[(m + 1) * (m + 2) / 2 + m] = sqrt(2.0 * m + 3.0) * x * diag;
        for (int n = m + 2; n < P; ++n) {
            double nn = (double)n * n, mm = (double)m * m;
            double A = sqrt((4.0 * nn - 1.0) / (nn - mm));
            double B = sqrt(((n - 1.0) * (n - 1.0) - mm) * (2.0 * n + 1.0) / ((2.0 * n - 3.0) * (nn - mm)));
            out[n * (n + 1) / 2 + m] = A * x * out[(n - 1) * n / 2 + m] - B * out[(n - 2) * (n - 1) / 2 + m];
        }
    }
}

// Spherical Bessel j_n(x), n = 0..nmax, by downward recurrence (Miller)
// normalised with j_0 or j_1, whichever is larger in magnitude.
__device__ inline void sph_bessel_j(int nmax, double x, double* j) {
    if (x == 0.0) {
        j[0] = 1.0;
        for (int n = 1; n <= nmax; ++n) j[n] = 0.0;
        return;
    }
    int start = nmax + 24 + (int)x;
    // (2n + 1) / x as a multiple of 1/x in two parts: one part alone is the
    // functions at a rounded argument, 4 to 8 times the error for n, x of 20 to 160
    const double ix = 1.0 / x, ir = fma(-x, ix, 1.0) * ix;
    double fp = 0.0, f = 1e-280;
    for (int n = 0; n <= nmax; ++n) j[n] = 0.0;
    for (int n = start; n >= 1; --n) {
        const double c = 2.0 * n + 1.0;
        double fm = fma(c, ix, c * ir) * f - fp;
        fp = f;
        f = fm;             // f = f_{n-1}, fp = f_n
        if (n - 1 <= nmax) j[n - 1] = f;
        if (n <= nmax) j[n] = fp;
        if (fabs(f) > 1e200) {
            f *= 1e-200;
            fp *= 1e-200;
            for (int q = n - 1; q <= nmax; ++q) j[q] *= 1e-200;
        }
    }
    double sn, cs;
    sincos(x, &sn, &cs);
    double j0 = sn / x;
    double j1 = sn / (x * x) - cs / x;
    double scale = (fabs(j0) >= fabs(j1) || nmax < 1) ? j0 / j[0] : j1 / j[1];
    for (int n = 0; n <= nmax; ++n) j[n] *= scale;
}

// Spherical Bessel y_n(x), n = 0..nmax, by upward recurrence (stable for y).
__device__ inline void sph_bessel_y(int nmax, double x, double* y) {
    double sn, cs;
    sincos(x, &sn, &cs);
    y[0] = -cs / x;
    if (nmax >= 1) y[1] = -cs / (x * x) - sn / x;
    for (int n = 1; n < nmax; ++n) y[n + 1] = (2.0 * n + 1.0) / x * y[n] - y[n - 1];
}

// Y_n^m(u) for n < P at unit vector u: out[nm_idx(n,m)].  q: scratch of
// P(P+1)/2 doubles.
__device__ inline void ylm_unit(int P, double ux, double uy, double uz, double* q, cd* out) {
    double s = sqrt(ux * ux + uy * uy);
    cd e1 = s > 0.0 ? mk(ux / s, uy / s) : mk(1.0, 0.0);
    legendre_q(P, uz, s, q);
    cd em = mk(1.0, 0.0);
    for (int m = 0; m < P; ++m) {
        for (int n = m; n < P; ++n) {
            double v = q[n * (n + 1) / 2 + m];
            out[nm_idx(n, m)] = v * em;
            if (m > 0) out[nm_idx(n, -m)] = v * conjg(em);
        }
        em = em * e1;
    }
}
