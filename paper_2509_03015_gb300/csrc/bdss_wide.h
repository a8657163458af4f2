// Factorisation of blocks 64 < n <= 256 with its products on the tensor cores
// (internal to the library; see bdss_wide.cu).
#pragma once
#include <cuda_runtime.h>

#include "bdss_device.cuh"

namespace bdss {

// Panels of a block: nt of them, nb columns each (the last may be narrower).
struct WidePanels {
  int nt, nb;
};
WidePanels wide_panels(int n);

template <typename T>
struct WideBuf {
  T *X;  // [m][64][64]: inverse of the current panel's diagonal tile, per eliminated block of the level
  // [m][64]: exponents of the square roots of the current panel's diagonal; the
  // columns of X are scaled by 2^E, what it multiplies by 2^-E as it is cut
  short *E;
  // both or neither (FP32, whose solve passes stream L^{-1}):
  T *Li;  // L^{-1} of every eliminated block (slot of its original index), zero above the diagonal
  T *V;   // [m][n][n]: L^{-T} of the level's blocks, as far as formed
};

// Bytes of WideBuf::X for a system of N blocks.
template <typename T> size_t wide_x_bytes(long long N);
template <typename T> cudaError_t wide_configure();

// Level 0: sym(A_diag) into Ld, the couplings into region 0 of Wb, B into Y.
template <typename T> cudaError_t launch_wide_ingest(const Args<T> &a, int sms, cudaStream_t s);
// Panel k of level l's eliminated blocks: the diagonal tile's Cholesky factor
// and inverse; then every row below it and the rows of W^T and y^T.
template <typename T> cudaError_t launch_wide_diag(const Args<T> &a, const WideBuf<T> &w, int l, int k, cudaStream_t s);
template <typename T>
cudaError_t launch_wide_panel(const Args<T> &a, const WideBuf<T> &w, int l, int k, int sms, cudaStream_t s);
// The separators' D, the next level's couplings and the separators' b.
template <typename T> cudaError_t launch_wide_schur(const Args<T> &a, int l, int sms, cudaStream_t s);
// The top block of an FP32 factorisation is factored in FP64: D_0 and b_0 (in
// a.Y) to FP64; its factor (a.Ltop), inverse and solution back.
cudaError_t launch_wide_top_in(const Args<float> &a, double *D, double *y, cudaStream_t s);
cudaError_t launch_wide_top_out(const Args<float> &a, const double *Li, const double *x, cudaStream_t s);
// Downward pass of level l.
template <typename T> cudaError_t launch_wide_down(const Args<T> &a, int l, cudaStream_t s);

}  // namespace bdss
