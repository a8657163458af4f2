// Host-side declarations of the Kalman-smoother assembly (Sec. 4.2), internal
// to the library.
#pragma once
#include <cuda_runtime.h>

#include "bdss_device.cuh"

namespace bdss {

// Normal equations assembled on the device.  U (N m n), v (N m), w (N n) are
// workspace; B == nullptr skips the right-hand side; rinv_diag: Rinv holds
// only the diagonals (N x m) of diagonal observation precisions.
struct KalmanArgs {
  long long N;
  int n, m, rinv_diag;
  const double *G, *H, *Qinv, *Rinv, *z, *zeta;
  double *A_diag, *A_sub, *B;
  double *U, *v, *w;
  // scaling along the products' common index (bdss_kalman.cu), 16-byte aligned:
  // N x kalman_pad(n) twice, N x kalman_pad(m); whether any step needs it (cleared
  // by the caller)
  short *EQ, *EG, *ER;
  int *scaled;
};
__host__ __device__ inline long long kalman_pad(int n) { return ((long long)n + 63) / 64 * 64; }
// Whether an assembly is small enough for the FP64-ALU tiles, which use neither the
// scaling nor a status.
bool kalman_on_alu(long long N, int n, int m);
// A product whose wait runs out sets st->status (cleared by the caller).
cudaError_t launch_kalman_assemble(const KalmanArgs &a, DevStatus *st, int sms, cudaStream_t s);
long long kalman_max_steps(int n, int m);  // largest N whose grids fit one launch

}  // namespace bdss
