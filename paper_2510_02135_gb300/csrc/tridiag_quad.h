// sqrt(T) e1 of a positive definite symmetric tridiagonal T on the host, in
// O(m) operations per quadrature node: the host part of the Krylov square
// root (libMobility paper, Sec. 3.3) when the Ritz values are safely positive.
//
// From sqrt(T) = (2 / pi) int_0^inf T (w^2 + T)^{-1} dw with
// w = sqrt(lo) sc(u; k'), k^2 = lo / hi, [lo, hi] a range that holds the
// spectrum: the integrand is analytic and periodic in u, so the midpoint rule
// with n nodes on (0, K'(k)) converges like exp(-2 pi^2 n / (log(hi / lo) +
// 2.8)) (Hale, Higham & Trefethen, SIAM J. Numer. Anal. 46, 2008, the change
// of variables of their Sec. 4).  20 to 50 nodes reach FP64 rounding.  One
// node is one tridiagonal solve; all nodes run side by side in the inner loop.
// Implicit QR (tridiag.cuh) takes about 1.5 m^2 dependent rotations instead:
// 206 us at m = 68 against 6 us, while an iteration of a system of a thousand
// particles takes 70 us on the GPU.
#pragma once

#include <cmath>
#include <vector>

namespace lmk {

struct SqrtQuadrature {
    std::vector<double> s, wt, x, dl, big, small;
    double lo_hint = 0.0;   // a lower bound of the previous T's spectrum

    // T - sigma I positive definite (no pivot of its L D L^T below zero)?
    static bool definite(int m, const double* al, const double* be, double sigma) {
        double q = al[0] - sigma;
        for (int i = 1; i < m; ++i) {
            if (!(q > 0.0)) return false;
            q = (al[i] - sigma) - be[i - 1] * be[i - 1] / q;
        }
        return q > 0.0;
    }

    // Nodes s_j = w_j^2 and weights for the spectrum in [lo, hi], n even.
    // Nodes j and n + 1 - j satisfy w w' = sqrt(lo hi), so only u < K'/2 is
    // evaluated, where cn stays away from zero; sn, cn, dn by the arithmetic-
    // geometric mean (Abramowitz & Stegun 16.4).
    void nodes(double lo, double hi, int n) {
        const double kPi = 3.14159265358979323846;
        s.resize(n);
        wt.resize(n);
        double a[16], c[16];
        const double k = std::sqrt(lo / hi);
        a[0] = 1.0;
        c[0] = std::sqrt(1.0 - k * k);
        double b = k;
        int L = 0;
        while (L < 15 && std::fabs(c[L]) > 1e-17 * a[L]) {
            a[L + 1] = 0.5 * (a[L] + b);
            c[L + 1] = 0.5 * (a[L] - b);
            b = std::sqrt(a[L] * b);
            ++L;
        }
        const double Kp = kPi / (2.0 * a[L]);
        const double step = 2.0 * Kp / (kPi * n);   // (2 / pi) h
        for (int j = 0; j < n / 2; ++j) {
            const double u = (j + 0.5) * Kp / n;
            double phi = std::ldexp(a[L] * u, L), prev = phi;
            for (int l = L; l >= 1; --l) {
                prev = phi;
                phi = 0.5 * (phi + std::asin(c[l] / a[l] * std::sin(phi)));
            }
            const double sn = std::sin(phi), cn = std::cos(phi);
            const double dn = L > 0 ? cn / std::cos(prev - phi) : 1.0;
            const double w = std::sqrt(lo) * sn / cn, dw = std::sqrt(lo) * dn / (cn * cn);
            s[j] = w * w;
            wt[j] = step * dw;
            s[n - 1 - j] = lo * hi / s[j];
            wt[n - 1 - j] = step * dw * std::sqrt(lo * hi) / s[j];
        }
    }

    // z = sqrt(T) e1, T with diagonal al[0..m) and off-diagonal be[0..m-1).
    // Returns false (z untouched) when T is not safely definite: its smallest
    // eigenvalue below 1e-10 of its largest; the caller then takes QR, which
    // clamps negative Ritz values.
    bool solve(int m, const double* al, const double* be, double* z) {
        double hi = 0.0;
        for (int i = 0; i < m; ++i) {
            const double r = std::fabs(al[i]) + (i > 0 ? std::fabs(be[i - 1]) : 0.0) + (i + 1 < m ? std::fabs(be[i]) : 0.0);
            hi = r <= hi ? hi : r;
        }
        if (!(hi > 1e-100 && hi < 1e100)) return false;   // no over- or underflow of products below
        double lo = m > 1 && lo_hint > 0.0 && lo_hint < 0.5 * hi ? lo_hint : 0.5 * hi;
        while (!definite(m, al, be, lo)) {
            lo *= 0.5;
            if (lo < 1e-10 * hi) {
                lo_hint = 0.0;
                return false;
            }
        }
        lo_hint = lo;   // the smallest Ritz value only falls as T grows
        const double kPi = 3.14159265358979323846;
        const int n = 2 * (int)std::ceil(0.5 * 39.0 * (std::log(hi / lo) + 2.8) / (2.0 * kPi * kPi));
        nodes(lo, hi, n);
        // pivots from the last row up: dl[i][j] = 1 / (al_i + s_j - be_i^2 dl[i+1][j])
        dl.resize((size_t)m * n);
        x.resize(n);
        big.assign(m, 0.0);
        small.assign(m, 0.0);
        double* D = dl.data();
        const double* S = s.data();
        for (int j = 0; j < n; ++j) D[(size_t)(m - 1) * n + j] = 1.0 / (al[m - 1] + S[j]);
        for (int i = m - 2; i >= 0; --i) {
            const double a = al[i], b2 = be[i] * be[i];
            const double* below = D + (size_t)(i + 1) * n;
            double* row = D + (size_t)i * n;
            for (int j = 0; j < n; ++j) row[j] = 1.0 / ((a + S[j]) - b2 * below[j]);
        }
        // x = (T + s)^{-1} e1 from the first row down.  Nodes up to hi enter as
        // T (T + s)^{-1} e1 = e1 - s x, the larger ones as T x: neither form
        // cancels there.  s ascends with j.
        int split = 0;
        while (split < n && S[split] < hi) ++split;
        double c0 = 0.0;
        for (int j = 0; j < n; ++j) {
            x[j] = wt[j] * (j < split ? S[j] : 1.0) * D[j];
            if (j < split) c0 += wt[j];
        }
        for (int i = 0; i < m; ++i) {
            if (i > 0) {
                const double b = -be[i - 1];
                const double* row = D + (size_t)i * n;
                for (int j = 0; j < n; ++j) x[j] = b * x[j] * row[j];
            }
            double t0 = 0.0, t1 = 0.0;
            for (int j = 0; j < split; ++j) t0 += x[j];
            for (int j = split; j < n; ++j) t1 += x[j];
            small[i] = t0;
            big[i] = t1;
        }
        for (int i = 0; i < m; ++i) {
            double t = al[i] * big[i] - small[i];
            if (i > 0) t += be[i - 1] * big[i - 1];
            if (i + 1 < m) t += be[i] * big[i + 1];
            z[i] = t;
        }
        z[0] += c0;
        return true;
    }
};

}  // namespace lmk
