// Host-side launchers of the device kernels (one definition each in near.cu, sort.cu,
// far.cu, backward.cu, batch.cu).
#pragma once

#include "psum_internal.cuh"

namespace psum {
// near.cu
cudaError_t launch_near32(bool grad, const float4* src_hi, const float4* src_lo, const double* src_org,
                          const float4* tgt_hi, const float4* tgt_lo, const double* tgt_org, const double* shifts,
                          double* partial, const NearPlanLaunch& L, cudaStream_t st, int variant = 0,
                          const double* src_x = nullptr, double Rb = 0.0, bool ff = false,
                          const int* grp_cls = nullptr, const float* img_w = nullptr, int n_cls = 1,
                          const double* grp_sub = nullptr, const int* chunk_img0 = nullptr,
                          const int* chunk_nimg = nullptr);
cudaError_t launch_near64(bool grad, const double4_32a* src, const double4_32a* tgt, const double* shifts,
                          double* partial, const NearPlanLaunch& L, cudaStream_t st, double Rb = 0.0,
                          const float* img_w = nullptr, int n_cls = 1);
constexpr int kCheckClasses = 6;   // two-layer check sums: partner axis and side
// dynamic shared memory of k_near32 for n_img images and n_cls image lists per target group;
// the launches stay within the 48 KiB that needs no opt-in
size_t near32_dyn_smem(int n_img, bool trimmed, bool grad, int n_cls);
constexpr size_t kNear32DynSmemMax = 48 * 1024;
cudaError_t launch_near_reduce(const double* partial, int64_t n_valid, int tile_size, int nq,
                               const NearPlanLaunch& L, double* out_phi, double* out_grad, cudaStream_t st);
int near32_occupancy_ctas(int n_img, int variant = 0, bool trimmed = false, bool ff = false, bool grad = true,
                          int n_cls = 1);
// register budget of the check-point (potential-only) launch of block plans: 0 = 4 CTAs/SM, 1 = 6
#ifndef PSUM_CHECK_VARIANT
#define PSUM_CHECK_VARIANT 0
#endif
constexpr int kCheckVariant = PSUM_CHECK_VARIANT;
cudaError_t launch_near32s(const float4* pk_hi, const float4* pk_lo, const double* org, const float4* ext,
                           const double* shifts, double* partial, const NearSymLaunch& S, cudaStream_t st,
                           bool ff = false, bool refine = false);
cudaError_t launch_sym_reduce(const double* partial, int64_t n_valid, const NearSymLaunch& S, double* out_phi,
                              double* out_grad, cudaStream_t st, bool fp64 = false, bool accumulate = false);
cudaError_t launch_near64s(const double4_32a* pk, const double* shifts, double* partial, const NearSymLaunch& S,
                           cudaStream_t st);
int near64s_occupancy_ctas(int64_t n_tiles);
int near32s_occupancy_ctas(int img_per_g, bool ff = false, bool refine = false);
constexpr int kNear32Variants = 2;
int near64_occupancy_ctas();
// sort.cu
// The box as the keys need it, and how they are stored: as float32 numbers where the points are
// ordered by counting (up to kRankMax of them; k_rank_order), as integers for the radix sort.  At
// kRankMax points counting takes about half of the radix sort's nine launches.
struct CurveBox {
    double d[3], inv[3];
    int as_float;
};
constexpr int64_t kRankSms = 152;                // SMs of the chip
constexpr int64_t kRankMax = 5 * 32 * kRankSms;  // up to five points a lane, one block an SM
inline CurveBox curve_box(const double d[3], int64_t n) {
    return CurveBox{{d[0], d[1], d[2]}, {256.0 / d[0], 256.0 / d[1], 256.0 / d[2]}, n <= kRankMax ? 1 : 0};
}
__device__ __forceinline__ uint32_t stored_key(const double* p, const CurveBox& box) {
    const uint32_t k = curve_key(p, box.d, box.inv);
    return box.as_float ? __float_as_uint((float)k) : k;
}
int sort_blocks(int64_t n);
int curve_order_launches(int64_t n);   // kernels launch_curve_order queues for n points
cudaError_t launch_curve_order(int64_t n, uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb, uint32_t* hist,
                               cudaStream_t st);
cudaError_t launch_curve_sort(const double* x, int64_t n, const double d[3], uint32_t* ka, uint32_t* va,
                               uint32_t* kb, uint32_t* vb, uint32_t* hist, cudaStream_t st);
cudaError_t launch_pack32(const double* x, const double* q, const uint32_t* perm, int64_t n, int64_t n_groups,
                          float4* pk_hi, float4* pk_lo, double* org, cudaStream_t st, double* xs = nullptr,
                          float4* ext = nullptr);
cudaError_t launch_pack64(const double* x, const double* q, int64_t n, int64_t n_pad, double4_32a* pk, cudaStream_t st);
cudaError_t launch_radix_sort(uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb, uint32_t* hist, int64_t n,
                              int passes, cudaStream_t st, uint32_t* spare = nullptr);
cudaError_t launch_pack32_groups(const double* x, const double* q, const uint32_t* perm, int64_t n_groups,
                                 const int64_t* grp_start, const int* grp_count, float4* pk_hi, float4* pk_lo,
                                 double* org, cudaStream_t st, float4* ext = nullptr);
cudaError_t launch_pack64_groups(const double* x, const double* q, int64_t n_pts, const int64_t* grp_start,
                                 const int* grp_count, double4_32a* pk, cudaStream_t st);
// far.cu
int reduce_blocks(int64_t n, int num_sms);
// validation of the charges (q) or of evaluation points (q null), with their curve keys where
// `keys` is given; launch_totals finishes the charges' neutrality test
cudaError_t launch_prepare(const double* x, const double* q, int64_t n, const double d[3], double* partial, int nblk,
                           int* status, uint32_t* keys, cudaStream_t st);
int mean_blocks(int64_t n, int num_sms);   // grid of launch_box_mean for n charges
cudaError_t launch_box_mean(const double* x, const double* q, int64_t n, const double H[3], double* partial,
                            int nblk, cudaStream_t st);
// far field of the RBF basis (Eq. 5): phi = phi_near + C_1 + sum_t C_{t+1} / |y - x_t|, float64
cudaError_t launch_far_rbf(const double* x, int64_t n, const int* perm, const double* phi_near,
                           const double* grad_near, const double* C, const double* centres, int S, const int* status,
                           double* phi, double* grad, int* status_out, int* plan_status, cudaStream_t st);
// trimmed near set: sum over the kept images x + p (|x + p| <= Rb) of the single box's potential
cudaError_t launch_box_mean_ball(const double* x, const double* q, const uint32_t* perm, int64_t n,
                                 const double d[3], const int K[3], double Rb, double* partial, int nblk,
                                 cudaStream_t st);
cudaError_t launch_project(const double* pinv, int rows, int M, const double* phi_check, const int* check_pos,
                           double* C, cudaStream_t st, bool layers = false);
// the box mean of phi_near from its partial sums (nblk of them; 0 without the mean condition) and the
// end of the validation
cudaError_t launch_totals(const double* mean_partial, int nblk, double inv_V0, const double* val_partial, int nblk_val,
                          int* status, double* mean, cudaStream_t st);
// C_1 as a launch of its own (RBF plans)
cudaError_t launch_constant(double* C, const double* Rbox, int P, const double* mean, int zero_mean, cudaStream_t st);
// the pair sums' partial slots as the far-field kernels read them
struct NearSlots {
    const double* partial;
    int sym;                    // 1: the symmetric kernels' last band (symsys), 0: one-sided (near, U, W)
    int tile;                   // targets per tile
    NearSys near;
    SymSys symsys;
    int64_t U, W;
    int max_contrib;
    const double *phi_acc, *grad_acc;   // sums of the earlier bands (null: none)
    int64_t limit;              // doubles of the partial buffer (debug bounds checks)
    int* status;
};
struct FarArgs {
    const double* x;            // the points, caller order
    int64_t n;
    const int* perm;            // packed order (null: the caller's)
    double* C;                  // C_2..C_P in, C_1 out
    const double* Rbox;
    const double* mean;
    int zero_mean, p;
    double inv_R0;
    double *phi, *grad;
    int* plan_status;
};
// the sum of near and far field at the points, written in the caller's order: the far field in
// float32 (FP32C plans) or float64
cudaError_t launch_sum_far32(const FarArgs& f, const NearSlots& a, const float* tab32, cudaStream_t st);
cudaError_t launch_sum_far64(const FarArgs& f, const NearSlots& a, const double* tab64, const double* grad_tab,
                             cudaStream_t st);
int64_t sym_limit(const NearSymLaunch& S);   // doubles of the partial buffer as the debug checks see it
constexpr int kSlotWarps = 8;

// Debug builds (-DPSUM_DEBUG_CHECKS=1) check the pair kernels' writes of their partial sums (the one-sided
// float64 kernel's aside) and the symmetric reductions' and the far field's reads of them against the
// buffer's size: an access outside it is skipped and flagged in the
// launch's status words (kStatBounds, PSUM_ERR_INTERNAL at psum_sync) instead of faulting.
__device__ __forceinline__ bool debug_in_range(int64_t off, int64_t n, int64_t limit, int* status, int n_status) {
#if PSUM_DEBUG_CHECKS
    if (off < 0 || off + n > limit) {
        for (int k = 0; k < n_status; ++k) atomicOr(status + k, kStatBounds);
        return false;
    }
#endif
    return true;
}

// backward.cu
// the moments w (P) of the charges and the far field of the coefficients C at them; C4: P scratch
cudaError_t launch_moments(const double* x, const double* q, int64_t n, const double* C, double4_32a* C4, int p,
                           double inv_R0, const double* tab, const double* grad_tab, double* far_phi, double* far_grad,
                           double* w_partial, int nblk, double* w, cudaStream_t st);
int moments_blocks(int64_t n, int p, int num_sms);
constexpr int kMomColDegree = 25;   // the moments by columns up to this degree (backward.cu)
cudaError_t launch_adjoint(const double* pinv, int rows, int M, const double* w, double* u, cudaStream_t st);
cudaError_t launch_check_sources32(const float4* chk_hi, const float4* chk_lo, const int* inv, int64_t n_pts, int M,
                                   const double* u, float4* out_hi, float4* out_lo, cudaStream_t st,
                                   bool layers = false);
cudaError_t launch_check_sources64(const double4_32a* chk, int64_t n_pts, int M, const double* u,
                                   double4_32a* out, cudaStream_t st);
cudaError_t launch_backward_combine(int64_t n, const int* perm, const double* q, const double* phi,
                                    const double* grad, const double* far_phi, const double* far_grad,
                                    const double* psi, const double* gpsi, const double* gE, double* dEdq,
                                    double* dEdx, cudaStream_t st);
cudaError_t launch_energy(const double* q, const double* phi, int64_t n, double* partial, int nblk, double* E,
                          cudaStream_t st);
}  // namespace psum

