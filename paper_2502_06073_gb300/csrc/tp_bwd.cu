// Launches of the adjoint of the environment embedding + tensor product (tp_kernels.cuh).
#include "tp_kernels.cuh"

namespace {

template <int LMAX, int INK, int OUTK, int CT, bool WB, typename... A>
void bwd_w(int n_atoms, int C, cudaStream_t s, A... args) {
  const long long teams = (long long)n_atoms * (C / CT);
  if (use_small(teams))
    ff_launch(k_env_tp_bwd<LMAX, INK, OUTK, CT, WB, true>, (int)teams, 128, 0, s, n_atoms, C,
              args...);
  else
    ff_launch(k_env_tp_bwd<LMAX, INK, OUTK, CT, WB, false>, ff_cdiv(teams * CT, 128), 128, 0, s,
              n_atoms, C, args...);
}

template <int LMAX, int INK, int OUTK, int CT>
void bwd_one(int n_atoms, int C, const int* row_ptr, int e0, const float* ef, const void* W,
             int wb, int ldw, const float* Vin, const float* thetaT, const float* GX, int ldx,
             int D, const float* gVout, float* gVin, float* GW, __nv_bfloat16* GWb,
             float* gY_v0, float* gY_env, int gy_stride, const float* Gam, float inv_sqrt_nu,
             cudaStream_t s) {
  if (wb)
    bwd_w<LMAX, INK, OUTK, CT, true>(n_atoms, C, s, row_ptr, e0, ef, (const __nv_bfloat16*)W, ldw,
                                     Vin, thetaT, GX, ldx, D, gVout, gVin, GW, GWb, gY_v0, gY_env,
                                     gy_stride, Gam, inv_sqrt_nu);
  else
    bwd_w<LMAX, INK, OUTK, CT, false>(n_atoms, C, s, row_ptr, e0, ef, (const float*)W, ldw, Vin,
                                      thetaT, GX, ldx, D, gVout, gVin, GW, GWb, gY_v0, gY_env,
                                      gy_stride, Gam, inv_sqrt_nu);
}

}  // namespace

void launch_env_tp_bwd(int lmax, int in_kind, int out_kind, int C, int n_atoms,
                       const int* row_ptr, int e0, const float* ef, const void* W, int w_bf16,
                       int ldw,
                       const float* Vin, const float* theta, const float* GX, int ldx, int D,
                       const float* gVout, float* gVin, float* GW, __nv_bfloat16* GWb, float* gY_v0, float* gY_env,
                       int gy_stride, const float* Gam, float inv_sqrt_nu, cudaStream_t s) {
  ProfScope ps_(PC_TP_BWD, s);
  if (n_atoms <= 0) return;
  FF_TP_DISPATCH(bwd_one, n_atoms, C, row_ptr, e0, ef, W, w_bf16, ldw, Vin, theta, GX, ldx, D,
                 gVout, gVin, GW, GWb, gY_v0, gY_env, gy_stride, Gam, inv_sqrt_nu, s);
  ff_count_launch(1);
}
