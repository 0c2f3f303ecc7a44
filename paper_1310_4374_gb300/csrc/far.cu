// Everything in algorithm "get" (Sec. 2.3.2) around the near-field sum:
//   validation (Eq. 1: neutral box, positions inside it), with the sort keys,
//   the right-hand side f and the least-squares coefficients (steps 4-5, Eqs. 8-10),
//   the constant C_1 from the zero-mean condition (step 6, Eqs. pfx3-pfx4, App. C),
//   the far field and its gradient at the charges and the final sum, with the pair sums'
//   partial slots (steps 7-8, Eqs. 1.6-1.9).
// All of it runs in float64 but the far field of FP32C plans, which is float32.
#include "launch.cuh"
#include "diffuse.cuh"
#include "harmonics.cuh"
#include "mean.cuh"

namespace psum {

// ---------------------------------------------------------------------------
// block reduction of two doubles (fixed order for a fixed block size)
// ---------------------------------------------------------------------------
template <int BS>
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double sa[BS / 32], sb[BS / 32];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { sa[w] = a; sb[w] = b; }
    __syncthreads();
    if (w == 0) {
        a = l < BS / 32 ? sa[l] : 0.0;
        b = l < BS / 32 ? sb[l] : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
    }
}

constexpr int kRedThreads = 256;

// Eq. 1: charges must sum to zero; positions must lie in [-d/2, d/2).  Without charges (kCharges
// false): evaluation points, inside the half-open box and finite.  `keys` (optional) receives the
// points' places on the spatial curve, so that validation adds no launch before the sort.
// The range test runs on ordered integers and the blocks are small: the float64 pipe of an SM is two
// lanes wide, so a few large blocks would queue on a few SMs' pipes.
constexpr int kPrepThreads = 64;

template <bool kCharges>
__global__ void __launch_bounds__(kPrepThreads) k_prepare(const double* __restrict__ x, const double* __restrict__ q,
                                                          int64_t n, CurveBox box, double* __restrict__ partial,
                                                          int* __restrict__ status, uint32_t* __restrict__ keys) {
    long long lo[3], hi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        lo[c] = ordered_bits(__double_as_longlong(-0.5 * box.d[c]));
        hi[c] = ordered_bits(__double_as_longlong(0.5 * box.d[c]));
    }
    double s = 0.0, sa = 0.0;
    int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * kPrepThreads + threadIdx.x; i < n; i += (int64_t)gridDim.x * kPrepThreads) {
        const double p[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long b = ordered_bits(__double_as_longlong(p[c]));
            if (!(b >= lo[c] && b < hi[c])) bad |= kStatOutOfBox;      // NaN positions too
        }
        if (keys) keys[i] = stored_key(p, box);
        if constexpr (kCharges) {
            const double qi = q[i];
            if (exp_field(__double_as_longlong(qi)) == 0x7ff) bad |= kStatNonFinite;
            s += qi;
            sa += fabs(qi);
        }
    }
    if (bad) atomicOr(status, bad);
    if constexpr (kCharges) {
        block_sum2<kPrepThreads>(s, sa);
        if (threadIdx.x == 0) {
            partial[2 * blockIdx.x] = s;
            partial[2 * blockIdx.x + 1] = sa;
        }
    }
}

// One (charge, term) pair per work item: sum_i q_i U(x_i) with U the regrouped corner sum
// over the block (12 terms, each one logarithm and one two-argument arctangent; every charge
// of the box lies inside the block).  Twelve items per
// charge in blocks of 64 threads keep small systems from running a handful of blocks through
// the float64 pipes of a few SMs (4000 charges: 148 us with one 256-thread block per 256
// charges).
constexpr int kMeanThreads = 64;
constexpr int kMeanTerms = 12;

__global__ void __launch_bounds__(kMeanThreads) k_box_mean(const double* __restrict__ x, const double* __restrict__ q,
                                                           int64_t n, double H0, double H1, double H2,
                                                           double* __restrict__ partial) {
    const double H[3] = {H0, H1, H2};
    double s = 0.0, dummy = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * kMeanThreads + threadIdx.x; k < kMeanTerms * n;
         k += (int64_t)gridDim.x * kMeanThreads) {
        const int64_t i = k / kMeanTerms;
        const int j = (int)(k - i * kMeanTerms);
        const double X[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
        s += q[i] * box_potential_paired_term(X, H, j);
    }
    block_sum2<kMeanThreads>(s, dummy);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// With the near set trimmed to the ball S_b (get step 2) every kept source image x + p
// (|x + p| <= Rb, the same float64 test as the pair kernels) contributes the potential of the
// box at x + p.  Along a line of images (fixed offsets on axes 0 and 1) the kept ones come in
// runs, and a run of boxes is one rod-shaped box: its potential is one regrouped corner sum
// (12 logarithms, 12 arctangents) instead of one per box.  The covering block's lattice is
// walked directly (i d_k is the image table's float64 value), so every kept test matches the
// pair kernels'.  Which images are kept depends on the charge, so the threads of a warp take
// charges in Hilbert order when a permutation is given: neighbours see nearly the same runs.
__global__ void __launch_bounds__(kRedThreads) k_box_mean_ball(const double* __restrict__ x,
                                                               const double* __restrict__ q,
                                                               const uint32_t* __restrict__ perm, int64_t n,
                                                               double d0, double d1, double d2, int K0, int K1,
                                                               int K2, double Rb, double* __restrict__ partial) {
    const double Rb2 = __dmul_rn(Rb, Rb);
    double s = 0.0, dummy = 0.0;
    for (int64_t k = (int64_t)blockIdx.x * kRedThreads + threadIdx.x; k < n; k += (int64_t)gridDim.x * kRedThreads) {
        const int64_t i = perm ? (int64_t)perm[k] : k;
        const double x0 = x[3 * i], x1 = x[3 * i + 1], x2 = x[3 * i + 2];
        double u = 0.0;
        for (int i1 = -K0; i1 <= K0; ++i1) {
            const double a = __dadd_rn(x0, i1 * d0);
            for (int i2 = -K1; i2 <= K1; ++i2) {
                const double b = __dadd_rn(x1, i2 * d1);
                const double ab = __dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b));
                if (ab > Rb2) continue;            // c^2 >= 0: no image of this line is kept
                int lo = 0;
                bool run = false;
                for (int i3 = -K2; i3 <= K2 + 1; ++i3) {
                    bool kept = false;
                    if (i3 <= K2) {
                        const double c = __dadd_rn(x2, i3 * d2);
                        kept = __dadd_rn(ab, __dmul_rn(c, c)) <= Rb2;
                    }
                    if (kept && !run) {
                        lo = i3;
                        run = true;
                    } else if (!kept && run) {
                        // the run lo .. i3 - 1: one box of i3 - lo images along axis 2
                        const double X[3] = {a, b, x2 + 0.5 * (double)(lo + i3 - 1) * d2};
                        const double H[3] = {0.5 * d0, 0.5 * d1, 0.5 * (double)(i3 - lo) * d2};
                        u += box_potential_paired(X, H);
                        run = false;
                    }
                }
            }
        }
        s += q[i] * u;
    }
    block_sum2<kRedThreads>(s, dummy);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// ---------------------------------------------------------------------------
// Steps 4-5: f_l = phi_near(y~_l) - phi_near(y_l), C_{2..P} = A^+ f.
// One warp per row of the (P-1) x M pseudo-inverse.
// ---------------------------------------------------------------------------
constexpr int kProjThreads = 256;

// With `layers` the check sums already hold the difference (the two image layers at y_l), at
// packed position check_pos[l].  Each row gathers f itself (it stays in cache): no launch for it.
__global__ void __launch_bounds__(kProjThreads) k_project(const double* __restrict__ pinv, int rows, int M,
                                                          const double* __restrict__ phi_check,
                                                          const int* __restrict__ check_pos, int layers,
                                                          double* __restrict__ C) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = blockIdx.x * (kProjThreads / 32) + w;
    if (row >= rows) return;
    const double* a = pinv + (int64_t)row * M;
    double s = 0.0;
#pragma unroll 4
    for (int l = lane; l < M; l += 32) {
        const double f = layers ? phi_check[check_pos[l]] : phi_check[check_pos[M + l]] - phi_check[check_pos[l]];
        s = fma(a[l], f, s);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) C[1 + row] = s;
}

// The box mean of phi_near (Eq. pfx4) from its partial sums, and the end of the validation: the
// charges' total against their absolute sum (Eq. 1).
__global__ void __launch_bounds__(kRedThreads) k_totals(const double* __restrict__ mean_partial, int nblk,
                                                        double inv_V0, const double* __restrict__ val_partial,
                                                        int nblk_val, int* __restrict__ status,
                                                        double* __restrict__ mean) {
    double m = 0.0, dummy = 0.0, qs = 0.0, qa = 0.0;
    for (int b = threadIdx.x; b < nblk; b += kRedThreads) m += mean_partial[b];
    for (int b = threadIdx.x; b < nblk_val; b += kRedThreads) {
        qs += val_partial[2 * b];
        qa += val_partial[2 * b + 1];
    }
    block_sum2<kRedThreads>(m, dummy);
    if (threadIdx.x == 0) *mean = m * inv_V0;
    __syncthreads();                           // block_sum2's shared sums are free again
    block_sum2<kRedThreads>(qs, qa);
    if (threadIdx.x == 0 && !(fabs(qs) <= 1e-12 * qa)) atomicOr(status, kStatNonNeutral);
}

// Step 6 (Eq. pfx3 with phi_mean = 0): C_1 = -<phi_near> - sum_{t>=2} C_t R_t^(0), by one warp; every
// lane returns it.
__device__ __forceinline__ double constant_term(const double* __restrict__ C, const double* __restrict__ Rbox, int P,
                                                const double* __restrict__ mean, int zero_mean) {
    if (!zero_mean) return 0.0;
    double s = 0.0;
#pragma unroll 4
    for (int t = 1 + (threadIdx.x & 31); t < P; t += 32) s = fma(C[t], Rbox[t], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return -*mean - s;
}
__global__ void k_constant(double* __restrict__ C, const double* __restrict__ Rbox, int P,
                           const double* __restrict__ mean, int zero_mean) {
    const double c = constant_term(C, Rbox, P, mean, zero_mean);
    if (threadIdx.x == 0) C[0] = c;
}

// The evaluation's status joins the plan's (psum_sync reads it): what was flagged before this
// kernel by its first thread, what a thread finds itself at once.
__device__ __forceinline__ void merge_status(const int* status, int* plan_status) {
    if (blockIdx.x == 0 && threadIdx.x == 0 && *status) atomicOr(plan_status, *status);
}
__device__ __forceinline__ void flag_nonfinite(int* status, int* plan_status) {
    atomicOr(status, kStatNonFinite);
    atomicOr(plan_status, kStatNonFinite);
}

// ---------------------------------------------------------------------------
// Steps 7-8: phi = phi_near + C_1 + sum_t C_t R_t(x/R0), grad likewise
// (the gradient of the expansion by differentiating the recurrence), written
// back to the caller's order.
// ---------------------------------------------------------------------------
constexpr int kFarThreads = 128;

//
// The kernels also add up the pair sums' partial slots (NearSlots): a block of 32 points has eight
// warps for the slots (every eighth each, combined in a fixed order) beside those that evaluate the
// expansion, so neither a reduction launch nor its latency stands before the far field, and C_1 is
// formed by each block for itself (the first one stores it).  As launches of their own the reduction
// and the constant took 5 to 12 us each on the way of a small evaluation.
struct SlotRow {
    int64_t r1, e1, r2, n;      // entries [0, e1) sit at r1 + e, the others at r2 + e - e1
};

// A point's slots: the work items that touch its tile (one-sided kernels), or the tile's row of the
// symmetric kernels' last band (see k_sym_reduce).
__device__ __forceinline__ SlotRow slot_row(const NearSlots& a, int64_t tile) {
    if (!a.sym) {
        const int64_t upt = a.near.n_chunks * a.near.n_img, first = tile * upt;
        const int64_t n = sk_owner(first + upt - 1, a.U, a.W) - sk_owner(first, a.U, a.W) + 1;
        return SlotRow{tile * a.max_contrib, n, 0, n};
    }
    const SymSys& S = a.symsys;
    if (tile < S.a0) return SlotRow{0, 0, 0, 0};
    const int64_t bw = S.a1 - S.a0, n_out = tile < S.a1 ? S.n_tiles - S.a1 : 0;
    return SlotRow{sym_slot(S, tile, S.a0) * S.n_g, bw * S.n_g, n_out > 0 ? sym_slot(S, tile, S.a1) * S.n_g : 0,
                   (bw + n_out) * S.n_g};
}

// Warp w's share of the sums of packed point i: potential, then field components with kGrad.
template <bool kGrad>
__device__ __forceinline__ void slot_sums(const NearSlots& a, int64_t i, int w, double (&acc)[4]) {
    const int64_t tile = i / a.tile;
    const SlotRow r = slot_row(a, tile);
    const double* base = a.partial + (i - tile * a.tile);
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = 0.0;
#pragma unroll 4
    for (int64_t k = w; k < r.n; k += kSlotWarps) {
        const int64_t off = (k < r.e1 ? r.r1 + k : r.r2 + (k - r.e1)) * 4 * a.tile;
        if (!debug_in_range(off, 4 * a.tile, a.limit, a.status, 1)) continue;
#pragma unroll
        for (int c = 0; c < (kGrad ? 4 : 1); ++c) acc[c] += base[off + c * a.tile];
    }
}

// One output of one point (c = 0: the potential, 1..3: the field) from the slot sums of the eight
// warps, the earlier bands' sums and the far field's value.
__device__ __forceinline__ void write_point(const NearSlots& a, const double* s_part, int lane, int64_t s, int64_t i,
                                            int c, double far, bool failed, double* phi, double* grad, int* status,
                                            int* plan_status) {
    double v = s_part[c * 32 + lane];
#pragma unroll
    for (int w = 1; w < kSlotWarps; ++w) v += s_part[(w * 4 + c) * 32 + lane];
    if (a.phi_acc) v = (c == 0 ? a.phi_acc[s] : a.grad_acc[3 * s + c - 1]) + v;
    const double r = failed ? __longlong_as_double(0x7ff8000000000000ll) : v + far;
    if (c == 0)
        phi[i] = r;
    else
        grad[3 * i + c - 1] = r;
    if (!failed && !(fabs(r) <= 1.7976931348623157e308)) {
        atomicOr(status, kStatNonFinite);
        atomicOr(plan_status, kStatNonFinite);
    }
}
constexpr int kStatFailed = kStatNonNeutral | kStatOutOfBox | kStatNonFinite | kStatTimeout | kStatBounds;

// FP32C plans: the far field in float32, a smooth, slowly varying part of phi (its float32
// evaluation errors sit well below the pair sum's), by the block's ninth warp.
template <bool kGrad>
__global__ void __launch_bounds__(32 * (kSlotWarps + 1)) k_sum_far32(FarArgs f, NearSlots a,
                                                                     const float* __restrict__ tab) {
    merge_status(a.status, f.plan_status);
    extern __shared__ unsigned char s_raw[];
    const int p = f.p, P = (p + 1) * (p + 1), nt = sh_tab_size(p);
    double* s_part = (double*)s_raw;                   // [8][4][32], then the far field's [4][32]
    double* s_far = s_part + kSlotWarps * 4 * 32;
    float* s_C = (float*)(s_far + 4 * 32);
    float* s_tab = s_C + P;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * 32 + lane;
    const bool live = s < f.n;
    const int64_t i = live ? (f.perm ? (int64_t)f.perm[s] : s) : 0;
    // every warp loads its part of the tables at once; the slot warps then go on without waiting
    for (int t = threadIdx.x; t < P; t += 32 * (kSlotWarps + 1))
        if (t) s_C[t] = (float)f.C[t];
    for (int t = threadIdx.x; t < nt; t += 32 * (kSlotWarps + 1)) s_tab[t] = tab[t];
    if (w == kSlotWarps) {
        const double x0 = f.x[3 * i], x1 = f.x[3 * i + 1], x2 = f.x[3 * i + 2];
        const double c1 = constant_term(f.C, f.Rbox, P, f.mean, f.zero_mean);
        if (lane == 0) {
            if (blockIdx.x == 0) f.C[0] = c1;
            s_C[0] = (float)c1;
        }
        asm volatile("bar.sync 1, %0;" ::"r"(32 * (kSlotWarps + 1)) : "memory");
        const float ux = (float)(x0 * f.inv_R0), uy = (float)(x1 * f.inv_R0), uz = (float)(x2 * f.inv_R0);
        float v = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
        // the t = 1 term of the sum is C_1 R^_0^0 = C_1: included by the visitor
        sh_visit_tab<kGrad>(ux, uy, uz, p, s_tab, [&](int nn, int mm, float h, float hx, float hy, float hz) {
            const float c = s_C[sh_index(nn, mm)];
            v = fma(c, h, v);
            if (kGrad) {
                gx = fma(c, hx, gx);
                gy = fma(c, hy, gy);
                gz = fma(c, hz, gz);
            }
        });
        s_far[lane] = (double)v;
        if (kGrad) {
            s_far[32 + lane] = (double)gx * f.inv_R0;
            s_far[64 + lane] = (double)gy * f.inv_R0;
            s_far[96 + lane] = (double)gz * f.inv_R0;
        }
    } else {
        asm volatile("bar.arrive 1, %0;" ::"r"(32 * (kSlotWarps + 1)) : "memory");
        if (live) {
            double acc[4];
            slot_sums<kGrad>(a, s, w, acc);
#pragma unroll
            for (int c = 0; c < (kGrad ? 4 : 1); ++c) s_part[(w * 4 + c) * 32 + lane] = acc[c];
        }
    }
    __syncthreads();
    if (w < (kGrad ? 4 : 1) && live)
        write_point(a, s_part, lane, s, i, w, s_far[w * 32 + lane], (*a.status & kStatFailed) != 0, f.phi, f.grad,
                    a.status, f.plan_status);
}

// FP64 and FF plans: in float64, the columns of the expansion shared out to the other warps of the
// block (harmonics.cuh), which form each coefficient with the gradient's first.  One thread per point
// with the gradient carried through the recurrence kept the float64 pipes of a few SMs busy for
// 61 us at 1000 charges and degree 8 (a float64 warp instruction takes a scheduler 64 cycles); by
// columns, a launch of its own, 12 us.
constexpr int kFar64Threads = 32 * (kSlotWarps + (kMaxDegree + 2) / 2);

template <bool kGrad>
__global__ void __launch_bounds__(kFar64Threads) k_sum_far64(FarArgs f, NearSlots a, const double* __restrict__ tab,
                                                             const double* __restrict__ grad_tab) {
    merge_status(a.status, f.plan_status);
    extern __shared__ double4_32a s_C4[];
    const int p = f.p, P = (p + 1) * (p + 1), nt = sh_tab_size(p), W = blockDim.x / 32 - kSlotWarps;
    double* s_part = (double*)(s_C4 + P);              // [8][4][32]
    double* s_red = s_part + kSlotWarps * 4 * 32;      // [W][4][32]
    double* s_tab = s_red + W * 4 * 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t s = (int64_t)blockIdx.x * 32 + lane;
    const bool live = s < f.n;
    const int64_t i = live ? (f.perm ? (int64_t)f.perm[s] : s) : 0;
    if (w >= kSlotWarps) {
        const int t0 = threadIdx.x - 32 * kSlotWarps;
        if (w == kSlotWarps) {
            const double c1 = constant_term(f.C, f.Rbox, P, f.mean, f.zero_mean);
            if (lane == 0) {
                s_C4[0].x = c1;
                if (blockIdx.x == 0) f.C[0] = c1;
            }
        }
        for (int t = t0; t < P; t += 32 * W) {
            double cx = 0.0, cy = 0.0, cz = 0.0;
            if (kGrad) grad_coeffs(f.C, grad_tab, p, t, cx, cy, cz);
            if (t) s_C4[t].x = f.C[t];
            s_C4[t].y = cx;
            s_C4[t].z = cy;
            s_C4[t].w = cz;
        }
        for (int t = t0; t < nt; t += 32 * W) s_tab[t] = tab[t];
        const double ux = f.x[3 * i] * f.inv_R0, uy = f.x[3 * i + 1] * f.inv_R0, uz = f.x[3 * i + 2] * f.inv_R0;
        asm volatile("bar.sync 1, %0;" ::"r"(32 * W) : "memory");    // the column warps among themselves
        double v = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
        harmonic_columns(ux, uy, uz, p, w - kSlotWarps, s_tab, [&](int t, double h) {
            const double4_32a c = s_C4[t];
            v = fma(c.x, h, v);
            if (kGrad) {
                gx = fma(c.y, h, gx);
                gy = fma(c.z, h, gy);
                gz = fma(c.w, h, gz);
            }
        });
        double* r = s_red + (w - kSlotWarps) * 4 * 32 + lane;
        r[0] = v;
        if (kGrad) {
            r[32] = gx;
            r[64] = gy;
            r[96] = gz;
        }
    } else if (live) {
        double acc[4];
        slot_sums<kGrad>(a, s, w, acc);
#pragma unroll
        for (int c = 0; c < (kGrad ? 4 : 1); ++c) s_part[(w * 4 + c) * 32 + lane] = acc[c];
    }
    __syncthreads();
    if (w < (kGrad ? 4 : 1) && live) {
        double v = s_red[w * 32 + lane];
        for (int k = 1; k < W; ++k) v += s_red[(k * 4 + w) * 32 + lane];
        write_point(a, s_part, lane, s, i, w, w == 0 ? v : v * f.inv_R0, (*a.status & kStatFailed) != 0, f.phi, f.grad,
                    a.status, f.plan_status);
    }
}

// Steps 7-8 with the RBF basis of Eq. 5: phi_far(y) = C_1 + sum_t C_{t+1} / |y - x_t| and
// its gradient, a pair sum of the targets against the n_rbf centres in float64 (the
// least-squares coefficients of kernel functions cancel strongly: a float32 sum would
// lose digits to that cancellation).  Centres with their coefficients are staged in
// shared memory in blocks of kRbfBlock.
constexpr int kRbfBlock = 256;

template <bool kGrad>
__global__ void __launch_bounds__(kFarThreads) k_far_rbf(const double* __restrict__ x, int64_t n,
                                                         const int* __restrict__ perm,
                                                         const double* __restrict__ phi_near,
                                                         const double* __restrict__ grad_near,
                                                         const double* __restrict__ C,
                                                         const double* __restrict__ centres, int S,
                                                         const int* __restrict__ status,
                                                         double* __restrict__ phi, double* __restrict__ grad,
                                                         int* __restrict__ status_out, int* __restrict__ plan_status) {
    merge_status(status, plan_status);
    __shared__ double4_32a s_c[kRbfBlock];
    const int64_t s = (int64_t)blockIdx.x * kFarThreads + threadIdx.x;
    const bool live = s < n;
    const int64_t i = live ? (perm ? (int64_t)perm[s] : s) : 0;
    const double y0 = live ? x[3 * i] : 0.0, y1 = live ? x[3 * i + 1] : 0.0, y2 = live ? x[3 * i + 2] : 0.0;
    double f = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    for (int t0 = 0; t0 < S; t0 += kRbfBlock) {
        const int nb = S - t0 < kRbfBlock ? S - t0 : kRbfBlock;
        __syncthreads();
        for (int t = threadIdx.x; t < nb; t += kFarThreads) {
            const double* c = centres + 3 * (size_t)(t0 + t);
            s_c[t] = make_double4_32a(c[0], c[1], c[2], C[1 + t0 + t]);
        }
        __syncthreads();
        for (int t = 0; t < nb; ++t) {
            const double4_32a c = s_c[t];
            const double a = y0 - c.x, b = y1 - c.y, e = y2 - c.z;
            const double ri = rsqrt(fma(e, e, fma(b, b, a * a)));
            const double cr = c.w * ri;
            f += cr;
            if (kGrad) {
                const double cr3 = cr * ri * ri;
                gx = fma(-cr3, a, gx);
                gy = fma(-cr3, b, gy);
                gz = fma(-cr3, e, gz);
            }
        }
    }
    if (!live) return;
    const bool failed = (*status & (kStatNonNeutral | kStatOutOfBox | kStatNonFinite | kStatTimeout | kStatBounds)) != 0;
    if (failed) {
        phi[i] = __longlong_as_double(0x7ff8000000000000ll);
        if (grad) grad[3 * i] = grad[3 * i + 1] = grad[3 * i + 2] = __longlong_as_double(0x7ff8000000000000ll);
        return;
    }
    const double ph = phi_near[s] + (C[0] + f);
    phi[i] = ph;
    bool finite = fabs(ph) <= 1.7976931348623157e308;
    if (kGrad) {
        const double g0 = grad_near[3 * s] + gx, g1 = grad_near[3 * s + 1] + gy, g2 = grad_near[3 * s + 2] + gz;
        grad[3 * i] = g0;
        grad[3 * i + 1] = g1;
        grad[3 * i + 2] = g2;
        finite = finite && fabs(g0) <= 1.7976931348623157e308 && fabs(g1) <= 1.7976931348623157e308 &&
                 fabs(g2) <= 1.7976931348623157e308;
    }
    if (!finite) flag_nonfinite(status_out, plan_status);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_far_rbf(const double* x, int64_t n, const int* perm, const double* phi_near,
                           const double* grad_near, const double* C, const double* centres, int S, const int* status,
                           double* phi, double* grad, int* status_out, int* plan_status, cudaStream_t st) {
    const unsigned nb = (unsigned)((n + kFarThreads - 1) / kFarThreads);
    if (grad)
        k_far_rbf<true><<<nb, kFarThreads, 0, st>>>(x, n, perm, phi_near, grad_near, C, centres, S, status, phi,
                                                    grad, status_out, plan_status);
    else
        k_far_rbf<false><<<nb, kFarThreads, 0, st>>>(x, n, perm, phi_near, grad_near, C, centres, S, status, phi,
                                                     grad, status_out, plan_status);
    return cudaGetLastError();
}

int reduce_blocks(int64_t n, int num_sms) {
    int64_t nb = (n + kPrepThreads - 1) / kPrepThreads;
    const int64_t cap = 16LL * num_sms;
    if (nb > cap) nb = cap;
    return nb < 1 ? 1 : (int)nb;
}

cudaError_t launch_prepare(const double* x, const double* q, int64_t n, const double d[3], double* partial, int nblk,
                           int* status, uint32_t* keys, cudaStream_t st) {
    if (q)
        k_prepare<true><<<nblk, kPrepThreads, 0, st>>>(x, q, n, curve_box(d, n), partial, status, keys);
    else
        k_prepare<false><<<nblk, kPrepThreads, 0, st>>>(x, q, n, curve_box(d, n), partial, status, keys);
    return cudaGetLastError();
}

// At most four blocks an SM: two warps a scheduler keep its float64 pipe busy, and the mean, which
// starts first, leaves registers for the sort and the packing beside it (with sixteen they waited for
// its first wave: 117 us until the pair sum at 20 000 charges, of which 62 us of their own).
int mean_blocks(int64_t n, int num_sms) {
    int64_t nb = (kMeanTerms * n + kMeanThreads - 1) / kMeanThreads;
    const int64_t cap = 4LL * num_sms;
    if (nb > cap) nb = cap;
    return nb < 1 ? 1 : (int)nb;
}

cudaError_t launch_box_mean(const double* x, const double* q, int64_t n, const double H[3], double* partial,
                            int nblk, cudaStream_t st) {
    k_box_mean<<<nblk, kMeanThreads, 0, st>>>(x, q, n, H[0], H[1], H[2], partial);
    return cudaGetLastError();
}

cudaError_t launch_box_mean_ball(const double* x, const double* q, const uint32_t* perm, int64_t n,
                                 const double d[3], const int K[3], double Rb, double* partial, int nblk,
                                 cudaStream_t st) {
    k_box_mean_ball<<<nblk, kRedThreads, 0, st>>>(x, q, perm, n, d[0], d[1], d[2], K[0], K[1], K[2], Rb, partial);
    return cudaGetLastError();
}

cudaError_t launch_project(const double* pinv, int rows, int M, const double* phi_check, const int* check_pos,
                           double* C, cudaStream_t st, bool layers) {
    const int per = kProjThreads / 32;
    k_project<<<(rows + per - 1) / per, kProjThreads, 0, st>>>(pinv, rows, M, phi_check, check_pos, layers ? 1 : 0, C);
    return cudaGetLastError();
}

cudaError_t launch_totals(const double* mean_partial, int nblk, double inv_V0, const double* val_partial, int nblk_val,
                          int* status, double* mean, cudaStream_t st) {
    k_totals<<<1, kRedThreads, 0, st>>>(mean_partial, nblk, inv_V0, val_partial, nblk_val, status, mean);
    return cudaGetLastError();
}

cudaError_t launch_constant(double* C, const double* Rbox, int P, const double* mean, int zero_mean, cudaStream_t st) {
    k_constant<<<1, 32, 0, st>>>(C, Rbox, P, mean, zero_mean);
    return cudaGetLastError();
}

// Debug builds: a slot read refused inside the kernel before (debug_in_range) is known to all of it only when it
// has ended, so it reaches the outputs and the plan's status here, as a refused write does in that kernel.
#if PSUM_DEBUG_CHECKS
__global__ void k_refused_reads(FarArgs f, const int* __restrict__ status) {
    if (!(*status & kStatBounds)) return;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) atomicOr(f.plan_status, kStatBounds);
    if (i >= f.n) return;
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    f.phi[i] = nan;
    if (f.grad) f.grad[3 * i] = f.grad[3 * i + 1] = f.grad[3 * i + 2] = nan;
}
#endif
static cudaError_t finish_sum_far(const FarArgs& f, const NearSlots& a, cudaStream_t st) {
#if PSUM_DEBUG_CHECKS
    k_refused_reads<<<(unsigned)((f.n + 255) / 256), 256, 0, st>>>(f, a.status);
#endif
    return cudaGetLastError();
}

cudaError_t launch_sum_far32(const FarArgs& f, const NearSlots& a, const float* tab32, cudaStream_t st) {
    const int P = (f.p + 1) * (f.p + 1);
    const size_t smem = sizeof(double) * (kSlotWarps + 1) * 128 + sizeof(float) * (P + sh_tab_size(f.p));
    const auto kernel = f.grad ? k_sum_far32<true> : k_sum_far32<false>;
    kernel<<<(unsigned)((f.n + 31) / 32), 32 * (kSlotWarps + 1), smem, st>>>(f, a, tab32);
    return finish_sum_far(f, a, st);
}

cudaError_t launch_sum_far64(const FarArgs& f, const NearSlots& a, const double* tab64, const double* grad_tab,
                             cudaStream_t st) {
    const int P = (f.p + 1) * (f.p + 1), W = harmonic_warps(f.p);
    const size_t smem = sizeof(double4_32a) * P + sizeof(double) * ((W + kSlotWarps) * 128 + sh_tab_size(f.p));
    const auto kernel = f.grad ? k_sum_far64<true> : k_sum_far64<false>;
    if (smem > 48 * 1024) {              // high degrees
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    kernel<<<(unsigned)((f.n + 31) / 32), 32 * (W + kSlotWarps), smem, st>>>(f, a, tab64, grad_tab);
    return finish_sum_far(f, a, st);
}

}  // namespace psum
