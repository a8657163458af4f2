// Factorisation of blocks up to n = 64 with the coupling solves and the Schur
// products on the tensor cores (internal to the library; see bdss_tcf.cu).
#pragma once
#include <cuda_runtime.h>

#include "bdss_device.cuh"

namespace bdss {

// Buffers of the current level, one set per eliminated block m: L^{-1}, and the
// updates it leaves pending on its left and its right separator (n x n
// diagonal update, lower triangle; n x d right-hand-side update).
template <typename T>
struct TcfLevel {
  T *X;   // [m][n][n], zero above the diagonal
  T *C;   // [m][2][n][n]
  T *cb;  // [m][2][n][d]
  // every block, by its original index: exponents of sqrt(D_kk) when its turn
  // comes to be factored (zero from n on), kept with the factors
  short *E;  // [N][64]
};

template <typename T> cudaError_t tcf_configure(int n, int d);
// Positions of level l: apply the pending updates of level l - 1 to every
// position; factor the odd ones (L, L^{-1}, y).  fold_all: the updates only
// (the last level's blocks, before the top block or sweep).
template <typename T>
cudaError_t launch_tcf_diag(const Args<T> &a, const TcfLevel<T> &c, int l, int fold_all, int sms, cudaStream_t s);
// W of level l's eliminated blocks, the updates they leave on their
// separators and the next level's couplings.
template <typename T>
cudaError_t launch_tcf_schur(const Args<T> &a, const TcfLevel<T> &c, int l, int sms, cudaStream_t s);
// The top block of the last level (one block): factor, and x_0 if d > 0.
template <typename T> cudaError_t launch_tcf_top(const Args<T> &a, const TcfLevel<T> &c, cudaStream_t s);
// FP64 solve passes with more right-hand sides than this are digit products
// (n = 64, N = 4096, d = 16, both ways: 4.2 -> 1.74 ms; with nine columns, in a
// tile of 16, they take 0.5 to 0.9 of the persistent kernel's time from n = 32 on,
// where the ALU kernel takes 0.9 to 2.4 of it with eight).
constexpr int kTcfMinRhsTc = 8;
// One level of a solve pass over stored factors that hold X (after launch_tcf_diag;
// in FP32 after any factorisation): up (first: y of level 0) and down.  E: the
// factorisation's exponents (FP64).
template <typename T> cudaError_t launch_tcf_up(const Args<T> &a, int l, int first, int sms, cudaStream_t s);
template <typename T> cudaError_t launch_tcf_down(const Args<T> &a, const short *E, int l, int sms, cudaStream_t s);

}  // namespace bdss
