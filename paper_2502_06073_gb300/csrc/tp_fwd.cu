// Launches of the environment embedding + tensor product kernels (tp_kernels.cuh).
#include "tp_kernels.cuh"

namespace {

template <int LMAX, int INK, int OUTK, int CT, bool WB, typename... A>
void fwd_w(int n_atoms, int C, cudaStream_t s, A... args) {
  const long long teams = (long long)n_atoms * (C / CT);
  if (use_small(teams))
    ff_launch(k_env_tp_fwd<LMAX, INK, OUTK, CT, WB, true>, (int)teams, 128, 0, s, n_atoms, C,
              args...);
  else
    ff_launch(k_env_tp_fwd<LMAX, INK, OUTK, CT, WB, false>, ff_cdiv(teams * CT, 128), 128, 0, s,
              n_atoms, C, args...);
}

template <int LMAX, int INK, int OUTK, int CT>
void fwd_one(int n_atoms, int C, const int* row_ptr, int e0, const float* ef, const void* W,
             int wb, int ldw, const float* Vin, const float* thetaT, float* X,
             __nv_bfloat16* Xb, int ldx, int D, float* Vout, float* Gam, float inv_sqrt_nu,
             cudaStream_t s) {
  if (wb)
    fwd_w<LMAX, INK, OUTK, CT, true>(n_atoms, C, s, row_ptr, e0, ef, (const __nv_bfloat16*)W, ldw,
                                     Vin, thetaT, X, Xb, ldx, D, Vout, Gam, inv_sqrt_nu);
  else
    fwd_w<LMAX, INK, OUTK, CT, false>(n_atoms, C, s, row_ptr, e0, ef, (const float*)W, ldw, Vin,
                                      thetaT, X, Xb, ldx, D, Vout, Gam, inv_sqrt_nu);
}

}  // namespace

void launch_env_tp_fwd(int lmax, int in_kind, int out_kind, int C, int n_atoms,
                       const int* row_ptr, int e0, const float* ef, const void* W, int w_bf16,
                       int ldw,
                       const float* Vin, const float* theta, float* X, __nv_bfloat16* Xb,
                       int ldx, int D, float* Vout, float* Gam, float inv_sqrt_nu,
                       cudaStream_t s) {
  ProfScope ps_(PC_TP_FWD, s);
  if (n_atoms <= 0) return;
  FF_TP_DISPATCH(fwd_one, n_atoms, C, row_ptr, e0, ef, W, w_bf16, ldw, Vin, theta, X, Xb, ldx,
                 D, Vout, Gam, inv_sqrt_nu, s);
  ff_count_launch(1);
}
