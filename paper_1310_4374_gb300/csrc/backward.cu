// Energy E = 1/2 sum_j q_j phi(x_j) and its exact derivatives for the discrete method.
//
// phi = phi_near + phi_far, phi_far = C_1 + sum_{t>=2} C_t R_t(x/R0), C_{2..P} = A^+ f and
// f_l = phi_near(y~_l) - phi_near(y_l) is linear in q (Eqs. 3, 8-10).  The adjoint of the
// least-squares fit gives, with the moments w_t = sum_j q_j R_t(x_j/R0) and u = (A^+)^T w,
//   psi(x)   = sum_l u_l [G(y~_l - x) - G(y_l - x)]   (G: the near-block image kernel),
//   dE/dq_k  = phi(x_k) - phi_far(x_k)/2 + psi(x_k)/2,
//   dE/dx_k  = q_k [grad phi - grad phi_far/2 + grad psi/2](x_k).
// psi is a near-field sum of check-point charges at the charges, done by the same pair kernels
// as the forward sum: 2M charges (+u at y~, -u at y) with the near block's images, or, as the
// right-hand side's two image layers, M points twice (+u_l with the upper layer's images, -u_l
// with the lower's; float32 packing with plans that take the layers).
#include "harmonics.cuh"

namespace psum {

constexpr int kMomThreads = 128;

// phi_far (with C_1) and grad phi_far at every charge, and per-block partial moments: degrees above
// kMomColDegree.
__global__ void __launch_bounds__(kMomThreads) k_moments(const double* __restrict__ x, const double* __restrict__ q,
                                                         int64_t n, const double* __restrict__ C, int p,
                                                         double inv_R0, const double* __restrict__ tab,
                                                         double* __restrict__ far_phi,
                                                         double* __restrict__ far_grad,
                                                         double* __restrict__ w_partial) {
    extern __shared__ double sm[];
    const int P = (p + 1) * (p + 1);
    constexpr int W = kMomThreads / 32;
    double* s_C = sm;
    double* s_w = sm + P;                                   // [warps][P]
    double* s_tab = s_w + W * P;
    for (int t = threadIdx.x; t < P; t += kMomThreads) s_C[t] = C[t];
    for (int t = threadIdx.x; t < sh_tab_size(p); t += kMomThreads) s_tab[t] = tab[t];
    for (int t = threadIdx.x; t < W * P; t += kMomThreads) s_w[t] = 0.0;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t i = (int64_t)blockIdx.x * kMomThreads + threadIdx.x;
    const bool valid = i < n;
    const double qi = valid ? q[i] : 0.0;
    const double ux = valid ? x[3 * i] * inv_R0 : 0.0;
    const double uy = valid ? x[3 * i + 1] * inv_R0 : 0.0;
    const double uz = valid ? x[3 * i + 2] * inv_R0 : 0.0;
    double f = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    double* ws = s_w + warp * P;
    sh_visit_tab<true>(ux, uy, uz, p, s_tab, [&](int nn, int mm, double v, double vx, double vy, double vz) {
        const int t = sh_index(nn, mm);
        const double c = s_C[t];
        f = fma(c, v, f);
        gx = fma(c, vx, gx);
        gy = fma(c, vy, gy);
        gz = fma(c, vz, gz);
        double m = qi * v;
        for (int o = 16; o > 0; o >>= 1) m += __shfl_down_sync(0xffffffffu, m, o);
        if (lane == 0) ws[t] += m;
    });
    if (valid) {
        far_phi[i] = f;
        far_grad[3 * i] = gx * inv_R0;
        far_grad[3 * i + 1] = gy * inv_R0;
        far_grad[3 * i + 2] = gz * inv_R0;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < P; t += kMomThreads) {
        double s = 0.0;
        for (int w = 0; w < W; ++w) s += s_w[w * P + t];
        w_partial[(int64_t)blockIdx.x * P + t] = s;
    }
}

// The same with the columns of the expansion shared out to the warps of a block of 32 charges
// (harmonics.cuh).  Each warp leaves its terms' values in shared memory, and a thread per term sums
// them over the charges, q in the multiply-add: one float64 warp operation per term where a shuffle
// reduction of every term took five and carrying the gradient 27 (2000 charges, degree 8: 89 us).
// A block takes every gridDim.x'th group of 32 charges and keeps its terms' sums in registers.
// Degrees up to kMomColDegree, whose values fit the shared memory of an SM; k_moments above.
constexpr int kMomOwn = 3;               // terms per thread: (p+1)^2 / (32 harmonic_warps(p)) < p/16 + 1
constexpr int kMomPad = 33;

__global__ void k_moments_columns(const double* __restrict__ x, const double* __restrict__ q, int64_t n,
                                  const double4_32a* __restrict__ C4, int p, double inv_R0,
                                  const double* __restrict__ tab, double* __restrict__ far_phi,
                                  double* __restrict__ far_grad, double* __restrict__ w_partial) {
    extern __shared__ double4_32a s_C4[];
    const int P = (p + 1) * (p + 1), nt = sh_tab_size(p), W = blockDim.x / 32;
    double* s_red = (double*)(s_C4 + P);              // [W][4][32]
    double* s_tab = s_red + W * 4 * 32;
    double* s_q = s_tab + nt;                         // [32]
    double* s_v = s_q + 32;                           // [P][kMomPad]
    for (int t = threadIdx.x; t < P; t += blockDim.x) s_C4[t] = C4[t];
    for (int t = threadIdx.x; t < nt; t += blockDim.x) s_tab[t] = tab[t];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double acc[kMomOwn] = {};
    for (int64_t g = blockIdx.x; g * 32 < n; g += gridDim.x) {
        const int64_t i = g * 32 + lane;
        const bool live = i < n;
        const double ux = live ? x[3 * i] * inv_R0 : 0.0, uy = live ? x[3 * i + 1] * inv_R0 : 0.0,
                     uz = live ? x[3 * i + 2] * inv_R0 : 0.0;
        __syncthreads();                              // tables in; the last group's values are used up
        if (w == 0) s_q[lane] = live ? q[i] : 0.0;
        double f = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
        harmonic_columns(ux, uy, uz, p, w, s_tab, [&](int t, double v) {
            const double4_32a c = s_C4[t];
            f = fma(c.x, v, f);
            gx = fma(c.y, v, gx);
            gy = fma(c.z, v, gy);
            gz = fma(c.w, v, gz);
            s_v[t * kMomPad + lane] = v;
        });
        s_red[(w * 4) * 32 + lane] = f;
        s_red[(w * 4 + 1) * 32 + lane] = gx;
        s_red[(w * 4 + 2) * 32 + lane] = gy;
        s_red[(w * 4 + 3) * 32 + lane] = gz;
        __syncthreads();
        for (int c = w; c < 4 && live; c += W) {
            double v = s_red[c * 32 + lane];
            for (int k = 1; k < W; ++k) v += s_red[(k * 4 + c) * 32 + lane];
            if (c == 0)
                far_phi[i] = v;
            else
                far_grad[3 * i + c - 1] = v * inv_R0;
        }
#pragma unroll
        for (int o = 0; o < kMomOwn; ++o) {
            const int t = threadIdx.x + o * blockDim.x;
            if (t < P) {
                double s = 0.0;
#pragma unroll 8
                for (int j = 0; j < 32; ++j) s = fma(s_q[j], s_v[t * kMomPad + j], s);
                acc[o] += s;
            }
        }
    }
#pragma unroll
    for (int o = 0; o < kMomOwn; ++o) {
        const int t = threadIdx.x + o * blockDim.x;
        if (t < P) w_partial[(int64_t)blockIdx.x * P + t] = acc[o];
    }
}

// the coefficients with those of the gradient (harmonics.cuh)
__global__ void k_grad_coeffs(const double* __restrict__ C, const double* __restrict__ gt, int p,
                              double4_32a* __restrict__ C4) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (p + 1) * (p + 1)) return;
    double4_32a c = make_double4_32a(C[t], 0.0, 0.0, 0.0);
    grad_coeffs(C, gt, p, t, c.y, c.z, c.w);
    C4[t] = c;
}

// Sums over rows with a lane per column: the warps take every kColWarps'th row and are added in a
// fixed order (one thread per column walked 100 to 300 rows one after another).
constexpr int kColWarps = 8;
template <class Row>
__device__ __forceinline__ double column_sum(int rows, Row&& row) {
    __shared__ double s_part[kColWarps][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double s = 0.0;
#pragma unroll 4
    for (int r = w; r < rows; r += kColWarps) s = row(r, s);
    s_part[w][lane] = s;
    __syncthreads();
    s = s_part[0][lane];
#pragma unroll
    for (int k = 1; k < kColWarps; ++k) s += s_part[k][lane];
    return s;
}

__global__ void __launch_bounds__(32 * kColWarps) k_moments_reduce(const double* __restrict__ w_partial, int nblk, int P,
                                                                  double* __restrict__ w) {
    const int t = blockIdx.x * 32 + (threadIdx.x & 31);
    const double s = column_sum(nblk, [&](int b, double a) { return t < P ? a + w_partial[(int64_t)b * P + t] : 0.0; });
    if (threadIdx.x < 32 && t < P) w[t] = s;
}

// u = (A^+)^T w over the non-constant moments t = 2..P.
__global__ void __launch_bounds__(32 * kColWarps) k_adjoint(const double* __restrict__ pinv, int rows, int M,
                                                           const double* __restrict__ w, double* __restrict__ u) {
    const int l = blockIdx.x * 32 + (threadIdx.x & 31);
    const double s = column_sum(rows, [&](int r, double a) {
        return l < M ? fma(pinv[(int64_t)r * M + l], w[1 + r], a) : 0.0;
    });
    if (threadIdx.x < 32 && l < M) u[l] = s;
}

// The check points as sources of psi with charges from u (packed positions from the plan).
// Point form (layers == 0): slot s holds point j = inv[s] (j < M: y_j, charge -u_j; else
// y~_{j-M}, charge +u_{j-M}).  Two-layer form: inv[s] = 2 l + side, charge +u_l with the upper
// layer's images (side 0), -u_l with the lower layer's (side 1).  -1: padding, charge 0.  With
// out_lo (float-float plans) the lo parts are copied too, with the charges' float32 remainders.
__global__ void k_check_sources32(const float4* __restrict__ chk_hi, const float4* __restrict__ chk_lo,
                                  const int* __restrict__ inv, int64_t n_pts, int M, const double* __restrict__ u,
                                  float4* __restrict__ out_hi, float4* __restrict__ out_lo, int layers) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_pts) return;
    const int j = inv[s];
    double cd = 0.0;
    if (j >= 0) {
        if (layers)
            cd = (j & 1) ? -u[j >> 1] : u[j >> 1];
        else
            cd = j < M ? -u[j] : u[j - M];
    }
    const float c = (float)cd;
    const float4 A = chk_hi[2 * s], B = chk_hi[2 * s + 1];
    out_hi[2 * s] = A;
    out_hi[2 * s + 1] = make_float4(B.x, B.y, c, c);
    if (out_lo) {
        const float cl = (float)(cd - (double)c);
        const float4 C = chk_lo[2 * s], D = chk_lo[2 * s + 1];
        out_lo[2 * s] = C;
        out_lo[2 * s + 1] = make_float4(D.x, D.y, cl, cl);
    }
}

__global__ void k_check_sources64(const double4_32a* __restrict__ chk, int64_t n_pts, int M,
                                  const double* __restrict__ u, double4_32a* __restrict__ out) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_pts) return;
    const double4_32a P = chk[s];
    double c = 0.0;
    if (s < 2 * M) c = s < M ? -u[s] : u[s - M];
    out[s] = make_double4_32a(P.x, P.y, P.z, c);
}

__global__ void k_backward_combine(int64_t n, const int* __restrict__ perm, const double* __restrict__ q,
                                   const double* __restrict__ phi, const double* __restrict__ grad,
                                   const double* __restrict__ far_phi, const double* __restrict__ far_grad,
                                   const double* __restrict__ psi, const double* __restrict__ gpsi,
                                   const double* __restrict__ gE, double* __restrict__ dEdq,
                                   double* __restrict__ dEdx) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int64_t i = perm ? (int64_t)perm[s] : s;
    const double g = gE ? *gE : 1.0;
    if (dEdq) dEdq[i] = g * (phi[i] - 0.5 * far_phi[i] + 0.5 * psi[s]);
    if (dEdx) {
        const double qi = g * q[i];
        for (int c = 0; c < 3; ++c)
            dEdx[3 * i + c] = qi * (grad[3 * i + c] - 0.5 * far_grad[3 * i + c] + 0.5 * gpsi[3 * s + c]);
    }
}

// E = 1/2 sum q phi, fixed-order reduction
constexpr int kEnThreads = 256;
__global__ void __launch_bounds__(kEnThreads) k_energy_partial(const double* __restrict__ q,
                                                               const double* __restrict__ phi, int64_t n,
                                                               double* __restrict__ partial) {
    __shared__ double sh[kEnThreads / 32];
    double s = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * kEnThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kEnThreads)
        s = fma(q[i], phi[i], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kEnThreads / 32; ++w) t += sh[w];
        partial[blockIdx.x] = t;
    }
}

// the partial sums in a fixed order: each thread every 256th, then the block as above
__global__ void __launch_bounds__(kEnThreads) k_energy_finish(const double* __restrict__ partial, int nblk,
                                                              double* __restrict__ E) {
    __shared__ double sh[kEnThreads / 32];
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += kEnThreads) s += partial[b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kEnThreads / 32; ++w) t += sh[w];
        *E = 0.5 * t;
    }
}

// ---------------------------------------------------------------------------
size_t moments_smem(int p) {
    const size_t P = (size_t)(p + 1) * (p + 1);
    if (p <= kMomColDegree)
        return sizeof(double4_32a) * P +
               sizeof(double) * (harmonic_warps(p) * 128 + sh_tab_size(p) + 32 + P * kMomPad);
    return sizeof(double) * (P * (1 + kMomThreads / 32) + sh_tab_size(p));
}

// blocks of the moments' launch: resident ones (two an SM up to degree 16) that share the charges, or
// one per kMomThreads charges
int moments_blocks(int64_t n, int p, int num_sms) {
    if (p > kMomColDegree) return (int)((n + kMomThreads - 1) / kMomThreads);
    const int64_t nb = (n + 31) / 32, cap = 2LL * num_sms;
    return (int)(nb < cap ? nb : cap);
}

cudaError_t launch_moments(const double* x, const double* q, int64_t n, const double* C, double4_32a* C4, int p,
                           double inv_R0, const double* tab, const double* grad_tab, double* far_phi, double* far_grad,
                           double* w_partial, int nblk, double* w, cudaStream_t st) {
    const int P = (p + 1) * (p + 1);
    const size_t smem = moments_smem(p);
    const bool cols = p <= kMomColDegree;
    if (smem > 48 * 1024) {
        const cudaError_t e = cols ? cudaFuncSetAttribute(k_moments_columns, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                                   : cudaFuncSetAttribute(k_moments, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    if (cols) {
        k_grad_coeffs<<<(P + 127) / 128, 128, 0, st>>>(C, grad_tab, p, C4);
        k_moments_columns<<<nblk, 32 * harmonic_warps(p), smem, st>>>(x, q, n, C4, p, inv_R0, tab, far_phi, far_grad,
                                                                     w_partial);
    } else {
        k_moments<<<nblk, kMomThreads, smem, st>>>(x, q, n, C, p, inv_R0, tab, far_phi, far_grad, w_partial);
    }
    k_moments_reduce<<<(P + 31) / 32, 32 * kColWarps, 0, st>>>(w_partial, nblk, P, w);
    return cudaGetLastError();
}

cudaError_t launch_adjoint(const double* pinv, int rows, int M, const double* w, double* u, cudaStream_t st) {
    k_adjoint<<<(M + 31) / 32, 32 * kColWarps, 0, st>>>(pinv, rows, M, w, u);
    return cudaGetLastError();
}

cudaError_t launch_check_sources32(const float4* chk_hi, const float4* chk_lo, const int* inv, int64_t n_pts, int M,
                                   const double* u, float4* out_hi, float4* out_lo, cudaStream_t st, bool layers) {
    k_check_sources32<<<(unsigned)((n_pts + 255) / 256), 256, 0, st>>>(chk_hi, chk_lo, inv, n_pts, M, u, out_hi,
                                                                         out_lo, layers ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_check_sources64(const double4_32a* chk, int64_t n_pts, int M, const double* u,
                                   double4_32a* out, cudaStream_t st) {
    k_check_sources64<<<(unsigned)((n_pts + 255) / 256), 256, 0, st>>>(chk, n_pts, M, u, out);
    return cudaGetLastError();
}

cudaError_t launch_backward_combine(int64_t n, const int* perm, const double* q, const double* phi,
                                    const double* grad, const double* far_phi, const double* far_grad,
                                    const double* psi, const double* gpsi, const double* gE, double* dEdq,
                                    double* dEdx, cudaStream_t st) {
    k_backward_combine<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, perm, q, phi, grad, far_phi, far_grad, psi,
                                                                    gpsi, gE, dEdq, dEdx);
    return cudaGetLastError();
}

cudaError_t launch_energy(const double* q, const double* phi, int64_t n, double* partial, int nblk, double* E,
                          cudaStream_t st) {
    k_energy_partial<<<nblk, kEnThreads, 0, st>>>(q, phi, n, partial);
    k_energy_finish<<<1, kEnThreads, 0, st>>>(partial, nblk, E);
    return cudaGetLastError();
}

}  // namespace psum
