// Float64 evaluation of the far field's expansion, column by column, with the gradient as an
// expansion of its own.
//
// The gradient of a regular solid harmonic of degree N is a combination of those of degree N - 1.
// With Z_N^m = R^_N^m + i R^_N^-m and s = (N-m)!, (N+m)! divided out as in Eq. 1.7, differentiating the
// generating recurrences of Eq. 1.6 (zeta = -x + iy: (dx + i dy) zeta = -2, (dx - i dy) zeta = 0) gives
//   dz Z_N^m              = -sqrt((N-m)(N+m))     Z_{N-1}^m,
//   (dx + i dy) Z_N^m     = -sqrt((N+m)(N+m-1))   Z_{N-1}^{m-1}     (m >= 1),
//   (dx - i dy) Z_N^m     =  sqrt((N-m)(N-m-1))   Z_{N-1}^{m+1},
// so sum_t C_t grad R^_t = sum_t (Cx, Cy, Cz)_t R^_t with coefficients formed once per evaluation, and
// a point costs about 7 float64 operations per term (the value and four products) where carrying the
// gradient through the recurrence took 27.
#pragma once

#include "launch.cuh"

namespace psum {

// sqrt((N+m)(N+m-1)), sqrt((N-m)(N-m-1)), sqrt((N-m)(N+m)) for 0 <= m <= N <= p
__host__ __device__ __forceinline__ int grad_tab_size(int p) { return 3 * (p + 1) * (p + 2) / 2; }
__host__ __device__ __forceinline__ int grad_tab_at(int N, int m) { return 3 * (N * (N + 1) / 2 + m); }
inline void grad_tab_fill(int p, double* t) {
    for (int N = 0; N <= p; ++N)
        for (int m = 0; m <= N; ++m) {
            double* g = t + grad_tab_at(N, m);
            g[0] = std::sqrt((double)(N + m) * (double)(N + m > 0 ? N + m - 1 : 0));
            g[1] = std::sqrt((double)(N - m) * (double)(N - m > 0 ? N - m - 1 : 0));
            g[2] = std::sqrt((double)(N - m) * (double)(N + m));
        }
}

// The gradient's coefficients of term t (degree n, order k) from the expansion's: what the terms of
// degree n + 1 contribute.
__host__ __device__ __forceinline__ void grad_coeffs(const double* __restrict__ C, const double* __restrict__ gt, int p,
                                                     int t, double& cx, double& cy, double& cz) {
    cx = cy = cz = 0.0;
    int n = 0;
    while ((n + 1) * (n + 1) <= t) ++n;
    const int N = n + 1;
    if (N > p) return;
    const int k = t - n * (n + 1), a = k < 0 ? -k : k;
    const double* Cn = C + N * (N + 1);
    cz = -gt[grad_tab_at(N, a) + 2] * Cn[k];
    const double up = 0.5 * gt[grad_tab_at(N, a + 1)];           // from order a + 1
    if (k >= 0) {
        cx = -up * Cn[a + 1];
        cy = up * Cn[-(a + 1)];
    } else {
        cx = -up * Cn[-(a + 1)];
        cy = -up * Cn[a + 1];
    }
    if (a >= 1) {                                                 // from order a - 1
        const double dn = (a == 1 ? 1.0 : 0.5) * gt[grad_tab_at(N, a - 1) + 1];
        const double p_ = Cn[a - 1], m_ = a == 1 ? 0.0 : Cn[-(a - 1)];
        if (k >= 0) {
            cx += dn * p_;
            cy += dn * m_;
        } else {
            cx += dn * m_;
            cy -= dn * p_;
        }
    }
}

// A warp's share of the expansion at its lanes' points: the columns m and p - m of both signs (equal
// work for every pair).  visit(t, v) once per term; Z_m comes by repeated multiplication by
// c_j (-x + iy) (tab: sh_tab_fill's).
template <class Visit>
__device__ __forceinline__ void harmonic_columns(double x, double y, double z, int p, int w, const double* tab,
                                                 Visit&& visit) {
    const double r2 = fma(z, z, fma(y, y, x * x));
    const double* e12 = tab + 2 * (p + 1);
    double re = 1.0, im = 0.0;
    int j = 0;
    for (int col = 0; col < 2; ++col) {
        const int m = col ? p - w : w;
        if (col && m <= w) break;
        for (; j < m;) {
            ++j;
            const double c = tab[j], a = -c * x, b = c * y;
            const double t = fma(a, re, -b * im);
            im = fma(b, re, a * im);
            re = t;
        }
        double a2 = re, b2 = im;
        visit(sh_index(m, m), a2);
        if (m) visit(sh_index(m, -m), b2);
        if (m + 1 > p) continue;
        const double zc = -z * tab[p + 1 + m];
        double a1 = zc * a2, b1 = zc * b2;
        visit(sh_index(m + 1, m), a1);
        if (m) visit(sh_index(m + 1, -m), b1);
        for (int n = m + 2; n <= p; ++n) {
            const double* e = e12 + 2 * (n * (n + 1) / 2 + m);
            const double ez = -e[0] * z, er = -e[1] * r2;
            const double a0 = fma(ez, a1, er * a2);
            a2 = a1;
            a1 = a0;
            visit(sh_index(n, m), a0);
            if (m) {
                const double b0 = fma(ez, b1, er * b2);
                b2 = b1;
                b1 = b0;
                visit(sh_index(n, -m), b0);
            }
        }
    }
}
// warps that share the columns of degree p
__host__ __device__ __forceinline__ int harmonic_warps(int p) { return (p + 2) / 2; }

}  // namespace psum
