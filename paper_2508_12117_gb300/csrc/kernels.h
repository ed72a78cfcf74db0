// Launchers of the device kernels (private to the library).
#pragma once
#include <cuda_runtime.h>

#include "view.h"

namespace spider {

// message returned by spider_last_error(NULL)
void set_static_error(const char* msg);

// travel times (k_tt.cu, k_mlp_tc.cu)
bool tt_supported_width(int H);
size_t tt_scratch_floats(const NetView& net, int num_sms);
// ctas_per_sm (1 or 2) shapes the FP32 MLP grid; scratch holds 2 x num_sms slots
cudaError_t launch_tt(const NetView& net, const PairSource& src, TTOut out, int num_sms, float* scratch,
                      cudaStream_t st, int ctas_per_sm);
// The same for the caller's arrays (raw pairs): the kernels write T_hi and T_lo
// themselves.  Splitting staged (hi, lo) pairs afterwards cost an allocation and
// two strided copies (47 pairs: 200 us a call that is waited for, 1.57 M pairs:
// 0.12 ms); it is left for times that overlap another array, where a pair's
// result may not be written before every pair has been read.  stage: P float2 of
// the caller's, or null to allocate them on the stream.
cudaError_t launch_times(const NetView& net, const PairSource& src, float* T_hi, float* T_lo, float* J, float2* stage,
                         int num_sms, float* scratch, cudaStream_t st);
cudaError_t launch_mlp_tc(const NetView& net, const PairSource& src, TTOut out, int num_sms,
                          float* scratch, cudaStream_t st);
bool mlp_tc_supported(int H, int precision);
// builds the tensor-core operand images (the first layer's split BF16 image,
// then the hidden layers) on the device
cudaError_t mlp_tc_prepare(const float* W1_host, const float* const Wn_host[3], const float* w5_host, int H,
                           int precision, void** image, float** scales, cudaStream_t st);

// step (k_step.cu)
cudaError_t configure_step_kernels();
cudaError_t launch_select(const StepView& v, int64_t n_b, cudaStream_t st, int bthreads = 256);
// bthreads: threads per CTA of the per-block kernels k_resid and k_final (a
// multiple of 32 up to 1024; results do not depend on it except the rounding
// order of the FP64 r.q sums)
cudaError_t launch_resid(const StepView& v, int64_t n_b, int gu, cudaStream_t st, const cudaEvent_t* ev,
                         int bthreads = 256);
cudaError_t launch_finish(const StepView& v, int64_t n_b, int gu, bool logpost, cudaStream_t st,
                          const cudaEvent_t* ev, int bthreads = 256);
// theta_0 + state (or a stored sample) in FP64, caller order (M x 4)
cudaError_t launch_state_out(const StepView& v, const float4* src, double* out, int grid, cudaStream_t st);
// the last gradient (FP32), caller order (M x 4)
cudaError_t launch_grad_out(const StepView& v, float4* out, int grid, cudaStream_t st);
cudaError_t launch_diag(const StepView& v, const float4* g, const float4* G, double* norms, double* part,
                        int grid, cudaStream_t st);
// whitening (k_whiten.cu: components of the step, stored piece inverses;
// k_solve.cu: conjugate gradients on the other components)
int piece_max_nodes();
int components_grid(int num_sms);
int whiten_clean_grid(int num_sms);
int solve_multi_grid(int num_sms);
cudaError_t configure_solve_kernels();
// branch streams on which independent kernels of one stage run side by side:
// `fork` is recorded on the launching stream and waited on by each branch,
// join[i] is recorded on branch i and waited on by the launching stream
constexpr int kBranches = 5;
struct Branches {
  cudaStream_t s[kBranches];
  cudaEvent_t fork;
  cudaEvent_t join[kBranches];
};
struct WhitenPlan {
  int use_inv;                 // clean pieces through their stored inverses
  int num_sms, cc_grid, clean_grid, multi_grid;
  int top_class;               // largest class that a component of the catalog can be of
  int clean_share;             // quarters of clean_grid on the branch stream (0: on the launching stream)
  int warp_mult, cta_mult;     // CTAs per SM of the one-warp class / of the CTA classes
};
// ev (nullable): four events recorded after the components, the one-warp and
// one-CTA classes, the multi-CTA class, and the join with the clean pieces
// (timed evaluations only); br null: everything in turn on st
cudaError_t launch_whiten(const StepView& v, int64_t n_b, const WhitenPlan& w, int max_it, float tol,
                          cudaStream_t st, const Branches* br, const cudaEvent_t* ev);
cudaError_t launch_solve_class(const StepView& v, int cls, int max_it, float tol, int ctas, cudaStream_t st);
cudaError_t launch_solve_multi(const StepView& v, int max_it, float tol, int grid, cudaStream_t st);
// stage-1 outlier mask (k_outlier.cu)
size_t outlier_scratch_bytes(int n_sub);
// ord (nullable: the same): the caller's index of each observation, the order of keep
cudaError_t launch_outlier(const StepView& v, int n_sub, float kmad, void* scratch, const int32_t* ord, uint8_t* keep,
                           int num_sms, cudaStream_t st, float* med_host, float* mad_host, int64_t* n_kept);
cudaError_t launch_linfilter(const StepView& v, int64_t n_b, float max_rel, const int32_t* ord, uint8_t* keep,
                             unsigned long long* kept, cudaStream_t st);
// posterior summaries (k_uq.cu)
int uq_max_samples();
// truth and results: M x 4 FP64 on the device, the caller's event order
cudaError_t launch_uq(const StepView& v, int64_t first, int n, const double* truth, double lo_pct,
                      double hi_pct, double* med, double* half, double* calib, double* ess, cudaStream_t st);
cudaError_t launch_philox_words(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                int64_t n, uint32_t* out, cudaStream_t st);

}  // namespace spider
