// Assembly of the Kalman-smoother normal equations of Sec. 4.2 on the device,
// so that a smoother built on the solver never forms its Hessian on the host.
// Step k (0-based) has transition G_k (n x n), observation H_k (m x n),
// precisions Qinv_k (n x n), Rinv_k (m x m), measurement z_k and process
// offset zeta_k; with G_N = 0 the MAP normal equations are block tridiagonal:
//   A_kk      = Qinv_k + G_{k+1}^T Qinv_{k+1} G_{k+1} + H_k^T Rinv_k H_k
//   A_{k+1,k} = -Qinv_{k+1} G_{k+1}
//   b_k       = H_k^T Rinv_k z_k + Qinv_k zeta_k - G_{k+1}^T Qinv_{k+1} zeta_{k+1}
// The n x n and m x n products run on the tensor cores as digit products
// (bdss_slice.cuh; small assemblies on the FP64 ALU, kalman_on_alu), two launches:
//   products  A_{k+1,k} = -Qinv G and, for a full Rinv, U_k = Rinv_k H_k;
//   diagonal  A_kk = Qinv_k + H_k^T U_k - G_{k+1}^T A_{k+1,k} (a diagonal Rinv
//             scales the rows of H as they are cut).
// The products' common index runs over the states of step k + 1 (Qinv G and
// G^T A_{k+1,k}) or the measurements of step k (Rinv H and H^T U), whose units
// enter the operands oppositely, so the operands are scaled along it by the
// exponents of the square roots of the precisions' diagonals (bdss_slice.cuh;
// without it a spread of units of 1e8 cost nine digits).  An entry is then off by
// 2^-57 .. 2^-53 of sqrt(Qinv_rr) max_k sqrt(Qinv_kk) |G_kc|, which is nothing beside
// the geometric mean of the diagonal entries of the normal equations it couples.
// A launch before the products (k_kalman_prepare) finds the exponents and forms
// the vectors v_k = Rinv_k z_k and w_k = Qinv_k zeta_k; where no step's exponents
// differ by more than kKmSpread the products run unscaled, at that loss of the 2^-57
// (N = 16384, n = 64, m = 32: 7.6 ms, and 8.4 ms scaled).  b_k is a small launch
// after them.
//
// Every product is formed transposed (TMEM lane = column of the result), so
// that a warp stores 32 consecutive entries of a row, and its A operand is a
// matrix read by columns: thread (c, g) takes the eight K entries 8 g .. of
// column c, coalesced over c, and cuts them to 16 bytes of every digit.
// With n <= 64 the 128 A rows of a tile are two steps, each multiplied by 32
// of its own B rows at a time; above, two blocks of 64 columns of one step.
//
// FP64-ALU tiles took 23.2 ms at N = 16384, n = 64, m = 32 (0.82 of the FP64
// pipe's rate).
#include "bdss_kalman.h"
#include "bdss_large.cuh"
#include "bdss_launch.h"
#include "bdss_slice_cta.cuh"

namespace bdss {

namespace {

// Work units: pairs of steps (n <= 64) or steps, and per unit the tiles of 128
// result columns.
__host__ __device__ inline long long kalman_groups(long long N, int n) { return n <= 64 ? (N + 1) / 2 : N; }
__host__ __device__ inline int kalman_row_tiles(int n) { return n <= 64 ? 1 : (n + 127) / 128; }
constexpr long long kKalmanTimeoutNs = 10000000000LL;  // bound of a product's wait

constexpr int kKmGroups = 8;  // K groups of eight in a chunk
constexpr size_t kKmSmem = wd_smem<double>();

// 64 rows of an operand by K index: entry (k, c) at p[k ld + c], c < cols
// (rows of B operands read by rows: entry (k, c) at p[c ld + k]); scale:
// factors of the K entries, or null.
struct KmSlot {
  const double *p;
  const double *scale;
  int cols;
};

// Entries k0 + 8 g .. of column c of a slot (zero past the ends).
__device__ __forceinline__ void km_load_col(const KmSlot &s, int ld, int k0, int K, int c, int g, double (&v)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = k0 + 8 * g + i;
    const bool in = c < s.cols && k < K;
    v[i] = in ? ldcg(s.p + (size_t)k * ld + c) : 0.0;
    if (s.scale && in) v[i] *= ldcg(s.scale + k);
  }
}
// Exponent of eight entries that count as v 2^(kSign e), poison included; kSign = 0:
// as they are, without it (km_row_exp).
template <int kSign>
__device__ __forceinline__ int km_exp(const double (&v)[8], const SlScale8 &sc) {
  int raw = 0, ex = kSlNoEx;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    raw = max(raw, sl_exp(v[i]));
    if (kSign) ex = max(ex, sl_exp(v[i]) + kSign * sc.at(i));
  }
  return kSign == 0 ? raw : raw == 0x7FF ? kSlPoisonEx : ex;
}
template <int kSign>
__device__ __forceinline__ int km_row_exp(int ex) {
  return kSign == 0 ? sl_row_exp<double>(ex) : ex;
}

// What a CTA multiplies: out[c][r] (+)= sum_k A(k, c) B(k, r) over K.
struct KmProduct {
  KmSlot a[2];   // A columns 64 b .. (two steps, or two blocks of one)
  int lda, K;
  KmSlot b[2];   // the B of each (the same matrix unless two steps)
  int ldb;
  bool brows;    // B read by rows (K contiguous)
  double sign;
  const short *e[2];  // exponents along K of each
};

// acc += sign x product: this thread's row and 8 columns.  pair: two steps, 32
// columns each per round (column 32 h + 4 hw + i at acc[4 h + i]); else 64
// columns from the first B slot (column 8 hw + i).  ncols: columns in use.  The A
// columns are scaled by 2^(kSign e) along K, the B columns by the inverse (kSign =
// 0: neither).
template <bool kPair, int kSign>
__device__ __forceinline__ bool km_product(WdCta<double> &w, const KmProduct &P, int ncols, int row, int hw,
                                           uint32_t lane_base, int *exK, double (&acc)[8]) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c = tid & 63, g = (tid >> 6) & 7, half = tid >> 9;  // half: this thread's A slot
  constexpr int kR = 64 / kWdWarps<double>;
  int *exKB = exK + kKmGroups * kSlRows;
#pragma unroll 1
  for (int k0 = 0; k0 < P.K; k0 += kSlK) {
    const int kc = min(kSlK, P.K - k0), ks = (kc + 15) >> 4;
    const int halves = kPair && ncols > 32 ? 2 : 1;
#pragma unroll 1
    for (int h = 0; h < halves; ++h) {
      double v[8], vb[8], r2[kR][2];
      const KmSlot sa = half ? P.a[1] : P.a[0];
      SlScale8 sca = {}, scb = {};
      short2 ke[2] = {};
      if (h == 0) {
        if (kSign) sca = sl_scale8((half ? P.e[1] : P.e[0]) + k0 + 8 * g);
        km_load_col(sa, P.lda, k0, P.K, c, g, v);
      }
      // B row rr of 64: column 32 h + (rr & 31) of its step, or column rr
      if (P.brows) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
          if (kSign) ke[b] = *reinterpret_cast<const short2 *>(P.e[b] + k0 + 2 * lane);
#pragma unroll
        for (int u = 0; u < kR; ++u) {
          const int rr = u * kWdWarps<double> + warp, k = 2 * lane;
          const KmSlot s = kPair && rr >= 32 ? P.b[1] : P.b[0];
          const int col = kPair ? 32 * h + (rr & 31) : rr;
          r2[u][0] = r2[u][1] = 0.0;
          if (col < s.cols) {
            const double *p = s.p + (size_t)col * P.ldb + k0 + k;
            if (k < kc) r2[u][0] = ldcg(p);
            if (k + 1 < kc) r2[u][1] = ldcg(p + 1);
          }
        }
      } else if (half == 0) {
        const KmSlot sb = kPair && c >= 32 ? P.b[1] : P.b[0];
        if (kSign) scb = sl_scale8((kPair && c >= 32 ? P.e[1] : P.e[0]) + k0 + 8 * g);
        km_load_col(sb, P.ldb, k0, P.K, kPair ? 32 * h + (c & 31) : c, g, vb);
        exKB[g * 64 + c] = km_exp<-kSign>(vb, scb);
      }
      if (h == 0) exK[g * kSlRows + 64 * half + c] = km_exp<kSign>(v, sca);
      __syncthreads();
      if (h == 0) {
        int ex = kSign == 0 ? 0 : kSlNoEx;
#pragma unroll
        for (int q = 0; q < kKmGroups; ++q) ex = max(ex, exK[q * kSlRows + 64 * half + c]);
        if (g == 0) w.exA[64 * half + c] = km_row_exp<kSign>(ex);
        store8<double, kSign>(v, ex, w.A + sl_off(64 * half + c, g), kSlASlab, sca);
      }
      if (P.brows) {
#pragma unroll
        for (int u = 0; u < kR; ++u) {
          const int rr = u * kWdWarps<double> + warp, k = 2 * lane;
          const short2 kb = ke[kPair && rr >= 32 ? 1 : 0];
          const int e0 = -kSign * kb.x, e1 = -kSign * kb.y;
          int ex;
          if constexpr (kSign != 0) ex = __reduce_max_sync(0xffffffffu, max(sl_exp_at(r2[u][0], e0), sl_exp_at(r2[u][1], e1)));
          else ex = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(sl_exp(r2[u][0]), sl_exp(r2[u][1])));
          if (lane == 0) w.exB[rr] = kSign != 0 ? ex : sl_row_exp<double>(ex);
          sl_store2<double>(r2[u][0], r2[u][1], ex,
                            w.B + (rr >> 5) * kWdBBytes<double> + sl_off(rr & 31, k >> 3) + 2 * (k & 7), kSlBSlab, e0, e1);
        }
      } else if (half == 0) {
        int ex = kSign == 0 ? 0 : kSlNoEx;
#pragma unroll
        for (int q = 0; q < kKmGroups; ++q) ex = max(ex, exKB[q * 64 + c]);
        if (g == 0) w.exB[c] = km_row_exp<kSign>(ex);
        store8<double, -kSign>(vb, ex, w.B + (c >> 5) * kWdBBytes<double> + sl_off(c & 31, g), kSlBSlab, scb);
      }
      const bool cols2 = kPair || ncols > 32;
      wd_issue<double>(w, cols2, ks, ks);
      const int ea = w.exA[row];
      bool ok = true;
      if constexpr (kPair) {
        if (32 * h + 4 * hw < ncols) {  // the same for a warp
          ok = wd_wait<double>(w, row >> 6);
          double x[4];
          if (ok)
            wd_drain4<double>(lane_base + (uint32_t)(row >> 6) * kWdBufCols<double> + (uint32_t)(4 * hw), ea,
                              w.exB + (row >> 6) * 32 + 4 * hw, x);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (h == 0) acc[e] = fma(P.sign, x[e], acc[e]);
            else acc[4 + e] = fma(P.sign, x[e], acc[4 + e]);
          }
        }
      } else if (8 * hw < ncols) {
        ok = wd_wait<double>(w, hw >> 2);
#pragma unroll
        for (int i = 0; i < 8; i += 4) {
          double x[4];
          if (ok)
            wd_drain4<double>(lane_base + (uint32_t)(hw >> 2) * kWdBufCols<double> + (uint32_t)(8 * (hw & 3) + i), ea,
                              w.exB + 8 * hw + i, x);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[i + e] = fma(P.sign, x[e], acc[i + e]);
        }
      }
      // the exponents and slabs have been read before the next ones are written
      if (!wd_round_end<double>(w, cols2, ok)) return false;
    }
  }
  return true;
}

// v_k = Rinv_k z_k, w_k = Qinv_k zeta_k (one step per CTA).
__device__ __forceinline__ void kalman_vectors(const KalmanArgs &a, long long k) {
  const int n = a.n, m = a.m;
  const double *Rk = a.Rinv + (size_t)k * (a.rinv_diag ? (size_t)m : (size_t)m * m), *zk = a.z + k * m;
  const double *Qk = a.Qinv + (size_t)k * n * n, *ek = a.zeta ? a.zeta + k * n : nullptr;
  for (int i = threadIdx.x; i < n + m; i += blockDim.x) {
    double s = 0.0;
    if (i < n) {
      if (ek)
        for (int j = 0; j < n; ++j) s = fma(Qk[(size_t)i * n + j], ek[j], s);
      a.w[k * n + i] = s;
    } else if (a.rinv_diag) {
      a.v[k * m + i - n] = Rk[i - n] * zk[i - n];
    } else {
      const double *r = Rk + (size_t)(i - n) * m;
      for (int j = 0; j < m; ++j) s = fma(r[j], zk[j], s);
      a.v[k * m + i - n] = s;
    }
  }
}

// Exponents for one step, a CTA: EQ and ER from the diagonals, zero beyond n or m.
// A diagonal entry that is not positive (or not a normal number) gives way to the
// largest of its row and column; where these are zero, the operand on the other
// side, on which the product does not depend, is scaled below anything that counts.
// EG scales Qinv G, whose entries are results: EQ, or nothing where the row
// maxima of Qinv and column maxima of G are smaller together without it (precisions
// that differ by orders of magnitude with a G that does not follow them).
constexpr short kKmDrop = -600;
constexpr int kKmSpread = 3;
__device__ short km_half_exp(const double *A, int n, int i) {
  double x = ldcg(A + (size_t)i * n + i);
  if (!(x > 0.0) || sl_exp(x) == 0) {
    x = 0.0;
    for (int j = 0; j < n; ++j) x = fmax(x, fmax(fabs(A[(size_t)i * n + j]), fabs(A[(size_t)j * n + i])));
    if (sl_exp(x) == 0) return kKmDrop;
  }
  return (short)sl_half_exp(x);
}
// Exponents of a finite v as it is and scaled by 2^e, into running maxima.
__device__ __forceinline__ void km_maxima(double v, int e, int &m0, int &m1) {
  const int x = sl_exp(v);
  if (x == 0 || x == 0x7FF) return;
  m0 = max(m0, x);
  m1 = max(m1, x + e);
}
__global__ void __launch_bounds__(256) k_kalman_prepare(const __grid_constant__ KalmanArgs a) {
  __shared__ int s_lo[2], s_hi[2], s_gain;
  const int n = a.n, m = a.m, pn = (int)kalman_pad(n), pm = (int)kalman_pad(m), tid = threadIdx.x;
  const long long k = blockIdx.x;
  const double *Q = a.Qinv + (size_t)k * n * n, *R = a.Rinv + (size_t)k * (a.rinv_diag ? (size_t)m : (size_t)m * m);
  short *EQ = a.EQ + k * pn, *EG = a.EG + k * pn, *ER = a.ER + k * pm;
  if (tid < 2) {
    s_lo[tid] = 1 << 20;
    s_hi[tid] = -(1 << 20);
  }
  if (tid == 0) s_gain = 0;
  __syncthreads();
  for (int i = tid; i < pn + pm; i += blockDim.x) {  // a warp's entries are one matrix's
    const int which = i >= pn, j = which ? i - pn : i;
    const bool in = j < (which ? m : n);
    short e = 0;
    if (in) {
      if (!which) {
        e = km_half_exp(Q, n, j);
      } else if (a.rinv_diag) {
        const double x = fabs(R[j]);
        e = sl_exp(x) == 0 ? kKmDrop : (short)sl_half_exp(x);
      } else {
        e = km_half_exp(R, m, j);
      }
    }
    const int lo = __reduce_min_sync(0xffffffffu, in ? (int)e : 1 << 20);
    const int hi = __reduce_max_sync(0xffffffffu, in ? (int)e : -(1 << 20));
    if ((tid & 31) == 0) {
      atomicMin(s_lo + which, lo);
      atomicMax(s_hi + which, hi);
    }
    if (which) ER[j] = e;
    else EQ[j] = EG[j] = e;
  }
  __syncthreads();
  const bool q = s_hi[0] - s_lo[0] > kKmSpread;
  if (tid == 0 && (q || s_hi[1] - s_lo[1] > kKmSpread)) atomicExch(a.scaled, 1);
  if (a.B) kalman_vectors(a, k);
  if (!q || k == 0) return;
  const double *G = a.G + (size_t)k * n * n;
  int gain = 0;  // sum of the maxima's exponents, scaled less unscaled
  for (int r = tid >> 5; r < n; r += blockDim.x >> 5) {
    int m0 = -(1 << 20), m1 = m0;
    for (int c = tid & 31; c < n; c += 32) km_maxima(ldcg(Q + (size_t)r * n + c), -EQ[c], m0, m1);
    m0 = __reduce_max_sync(0xffffffffu, m0);
    m1 = __reduce_max_sync(0xffffffffu, m1);
    if ((tid & 31) == 0) gain += m1 - m0;
  }
  for (int c = tid; c < n; c += blockDim.x) {
    int m0 = -(1 << 20), m1 = m0;
    for (int r = 0; r < n; ++r) km_maxima(ldcg(G + (size_t)r * n + c), EQ[r], m0, m1);
    gain += m1 - m0;
  }
  atomicAdd(&s_gain, gain);
  __syncthreads();
  if (s_gain > 0)
    for (int i = tid; i < pn; i += blockDim.x) EG[i] = 0;
}

// kDiag = 0: the products A_{k+1,k} and U_k; 1: the diagonal blocks.
template <int kDiag, bool kPair, bool kScaled>
__device__ __forceinline__ void kalman_tiles(const KalmanArgs &a, DevStatus *st, WdCta<double> &w, int *s_exK) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hw = warp >> 2, row0 = 32 * (warp & 3), row = row0 + lane;
  const uint32_t lane_base = w.tmem + ((uint32_t)row0 << 16);
  const int n = a.n, m = a.m;
  const size_t nn = (size_t)n * n, mn = (size_t)m * n, mm = a.rinv_diag ? (size_t)m : (size_t)m * m;
  const long long groups = kalman_groups(a.N, n);
  const int tr = kalman_row_tiles(n), tn = (n + 63) / 64, tm = kDiag || a.rinv_diag ? 0 : (m + 63) / 64;
  const int tiles = tr * (tn + tm);
  bool ok = true;
  for (long long t = blockIdx.x; t < groups * tiles && ok; t += gridDim.x) {
    const long long grp = t / tiles;
    const int u = (int)(t - grp * tiles), ct = u / tr, c0 = kPair ? 0 : 128 * (u - ct * tr);
    const bool isU = ct >= tn;
    const int r0 = 64 * (isU ? ct - tn : ct), R = isU ? m : n, ncols = min(64, R - r0);
    // slot b: step k_b, result columns c_b .. (rows of TMEM)
    double acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0.0;
    KmProduct P;
    P.lda = n;
    for (int part = kDiag && m > 0 ? 0 : 1; part < 2 && ok; ++part) {
      // kDiag: part 0: H^T U, part 1: -G^T A_sub; else one product
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const long long k = kPair ? 2 * grp + b : grp;
        const int cb = kPair ? 0 : c0 + 64 * b;
        const bool next = k + 1 < a.N, live = k < a.N && cb < n;
        KmSlot sa{nullptr, nullptr, 0}, sb{nullptr, nullptr, 0};
        if (kDiag && part == 0 && live) {
          sa = {(a.rinv_diag ? a.H : a.U) + (size_t)k * mn + cb, a.rinv_diag ? a.Rinv + (size_t)k * mm : nullptr,
                min(64, n - cb)};
          sb = {a.H + (size_t)k * mn + r0, nullptr, ncols};
        } else if (kDiag && live && next) {
          sa = {a.A_sub + (size_t)k * nn + cb, nullptr, min(64, n - cb)};
          sb = {a.G + (size_t)(k + 1) * nn + r0, nullptr, ncols};
        } else if (!kDiag && isU && live) {
          sa = {a.H + (size_t)k * mn + cb, nullptr, min(64, n - cb)};
          sb = {a.Rinv + (size_t)k * mm + (size_t)r0 * m, nullptr, ncols};
        } else if (!kDiag && !isU && live && next) {
          sa = {a.G + (size_t)(k + 1) * nn + cb, nullptr, min(64, n - cb)};
          sb = {a.Qinv + (size_t)(k + 1) * nn + (size_t)r0 * n, nullptr, ncols};
        }
        P.a[b] = sa;
        P.b[b] = sb;
        // (a slot without a step: any step's)
        const bool meas = kDiag ? part == 0 : isU;
        if (kScaled)
          P.e[b] = meas ? a.ER + min(k, a.N - 1) * kalman_pad(m)
                        : (kDiag ? a.EQ : a.EG) + min(k + 1, a.N - 1) * kalman_pad(n);
      }
      if (!kPair) P.b[1] = P.b[0];
      P.brows = !kDiag;
      P.K = (kDiag ? part == 0 : isU) ? m : n;
      P.ldb = kDiag ? n : isU ? m : n;
      P.sign = kDiag ? (part == 0 ? 1.0 : -1.0) : isU ? 1.0 : -1.0;
      ok = km_product<kPair, !kScaled ? 0 : kDiag ? -1 : 1>(w, P, ncols, row, hw, lane_base, s_exK, acc);
    }
    if (!ok) {
      if (threadIdx.x == 0) set_status(st, kStTimeout, -1, -1);
      break;
    }
    const int b = row >> 6, c = (kPair ? 0 : c0 + 64 * b) + (row & 63);
    const long long k = kPair ? 2 * grp + b : grp;
    if (k >= a.N || c >= n || (!kDiag && !isU && k + 1 >= a.N)) continue;
    double *out = kDiag ? a.A_diag + (size_t)k * nn : isU ? a.U + (size_t)k * mn : a.A_sub + (size_t)k * nn;
    const double *add = kDiag ? a.Qinv + (size_t)k * nn : nullptr;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int r = kPair ? 32 * (i >> 2) + 4 * hw + (i & 3) : 8 * hw + i;
      if (r < ncols) {
        const size_t o = (size_t)(r0 + r) * n + c;
        out[o] = kDiag ? ldcg(add + o) + acc[i] : acc[i];
      }
    }
  }
}

template <int kDiag, bool kPair>
__global__ void __launch_bounds__(kWdThreads<double>, 1) k_kalman_tc(const __grid_constant__ KalmanArgs a, DevStatus *st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t s_bar[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_exA[kSlRows], s_exB[64], s_exK[kKmGroups * (kSlRows + 64)];
  WdCta<double> w;
  wd_begin(w, smem_raw, s_bar, &s_tmem, s_exA, s_exB, s_exK, kKalmanTimeoutNs);
  if (*a.scaled) kalman_tiles<kDiag, kPair, true>(a, st, w, s_exK);
  else kalman_tiles<kDiag, kPair, false>(a, st, w, s_exK);
  wd_end(w);
}

// b_k = H_k^T v_k + w_k - G_{k+1}^T w_{k+1}.
__device__ __forceinline__ void kalman_rhs(const KalmanArgs &a, long long k) {
  const int n = a.n, m = a.m;
  const double *Hk = a.H + (size_t)k * m * n, *vk = a.v + k * m, *wk = a.w + k * n;
  const bool next = k + 1 < a.N;
  const double *G1 = a.G + (size_t)(k + 1) * n * n, *w1 = a.w + (k + 1) * n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double s = 0.0;
    for (int j = 0; j < m; ++j) s = fma(Hk[(size_t)j * n + i], vk[j], s);
    double g = 0.0;
    if (next)
      for (int j = 0; j < n; ++j) g = fma(G1[(size_t)j * n + i], w1[j], g);
    a.B[k * n + i] = s + wk[i] - g;
  }
}
__global__ void __launch_bounds__(kThreads) k_kalman_rhs(const __grid_constant__ KalmanArgs a) {
  kalman_rhs(a, blockIdx.x);
}

// The same on the FP64 ALU, for small assemblies: a flat grid of (step, task) CTAs
// of 64 x 64 tiles, two launches, the vectors among the tasks.
//   products  A_{k+1,k} (-Qinv G), U_k = Rinv_k H_k (a row scaling when Rinv_k is
//             diagonal), v_k and w_k;
//   diagonal  A_kk = Qinv_k + H_k^T U_k - G_{k+1}^T A_{k+1,k}, and b_k.
__device__ void store_tile(double *out, long long ld, int rows, int cols, int r0, int c0, const double (&acc)[4][4],
                           double sign, const double *add) {
  const int tm = threadIdx.x >> 4, tn = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + 4 * tm + i;
    if (r >= rows) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + 4 * tn + j;
      if (c >= cols) continue;
      const long long o = (long long)r * ld + c;
      out[o] = (add ? add[o] : 0.0) + sign * acc[i][j];
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_kalman_products_alu(const __grid_constant__ KalmanArgs a) {
  __shared__ double sA[kKc * kTilePad], sB[kKc * kTilePad];
  const int n = a.n, m = a.m, nt = ntiles(n), mt = ntiles(m);
  const int tasks = nt * nt + mt * nt + 1;
  const long long k = (long long)blockIdx.x / tasks;
  const int t = (int)((long long)blockIdx.x - k * tasks);
  const long long nn = (long long)n * n, mn = (long long)m * n;
  const long long mm = a.rinv_diag ? (long long)m : (long long)m * m;  // Rinv stride per step
  double acc[4][4] = {};
  if (t < nt * nt) {
    if (k + 1 >= a.N) return;
    const int r0 = (t / nt) * kTile, c0 = (t % nt) * kTile;
    const View<double> Q{a.Qinv + (k + 1) * nn, n, 1, n, n};  // (r, j) -> Qinv_{k+1}[r][j]
    const View<double> Gt{a.G + (k + 1) * nn, 1, n, n, n};    // (c, j) -> G_{k+1}[j][c]
    gemm_nt_tile(acc, Q, r0, Gt, c0, n, sA, sB);
    store_tile(a.A_sub + k * nn, n, n, n, r0, c0, acc, -1.0, nullptr);
  } else if (t < nt * nt + mt * nt) {
    const int u = t - nt * nt, r0 = (u / nt) * kTile, c0 = (u % nt) * kTile;
    if (a.rinv_diag) {
      const double *rk = a.Rinv + k * mm, *Hk = a.H + k * mn;
      double *Uk = a.U + k * mn;
      for (int e = threadIdx.x; e < kTile * kTile; e += blockDim.x) {
        const int r = r0 + e / kTile, c = c0 + e % kTile;
        if (r < m && c < n) Uk[(long long)r * n + c] = rk[r] * Hk[(long long)r * n + c];
      }
      return;
    }
    const View<double> R{a.Rinv + k * mm, m, 1, m, m};  // (r, j) -> Rinv_k[r][j]
    const View<double> Ht{a.H + k * mn, 1, n, n, m};    // (c, j) -> H_k[j][c]
    gemm_nt_tile(acc, R, r0, Ht, c0, m, sA, sB);
    store_tile(a.U + k * mn, n, m, n, r0, c0, acc, 1.0, nullptr);
  } else if (a.B) {
    kalman_vectors(a, k);
  }
}

__global__ void __launch_bounds__(kThreads) k_kalman_diag_alu(const __grid_constant__ KalmanArgs a) {
  __shared__ double sA[kKc * kTilePad], sB[kKc * kTilePad];
  const int n = a.n, m = a.m, nt = ntiles(n);
  const int tasks = nt * nt + 1;
  const long long k = (long long)blockIdx.x / tasks;
  const int t = (int)((long long)blockIdx.x - k * tasks);
  const long long nn = (long long)n * n, mn = (long long)m * n;
  if (t < nt * nt) {
    const int r0 = (t / nt) * kTile, c0 = (t % nt) * kTile;
    double acc[4][4] = {};
    const View<double> Hc{a.H + k * mn, 1, n, n, m};  // (r, j) -> H_k[j][r]
    const View<double> Uc{a.U + k * mn, 1, n, n, m};  // (c, j) -> U_k[j][c]
    gemm_nt_tile(acc, Hc, r0, Uc, c0, m, sA, sB);
    if (k + 1 < a.N) {
      double acc2[4][4] = {};
      const View<double> Gc{a.G + (k + 1) * nn, 1, n, n, n};  // (r, j) -> G_{k+1}[j][r]
      const View<double> Sc{a.A_sub + k * nn, 1, n, n, n};    // (c, j) -> A_{k+1,k}[j][c]
      gemm_nt_tile(acc2, Gc, r0, Sc, c0, n, sA, sB);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] -= acc2[i][j];
    }
    store_tile(a.A_diag + k * nn, n, n, n, r0, c0, acc, 1.0, a.Qinv + k * nn);
  } else if (a.B) {
    kalman_rhs(a, k);
  }
}

}  // namespace

// Limit of the ALU tiles' grids, the entry point's for either path.
long long kalman_max_steps(int n, int m) {
  const int nt = ntiles(n), mt = ntiles(m);
  return 0x7fffffffLL / (nt * nt + mt * nt + 1);
}

// The tensor-core path takes four launches and 128-column tiles of 64 K entries
// whatever n and m: few steps, or small ones, are faster on the ALU.  Its time over
// the ALU's, measured on GB300 (full Rinv; diagonal ones cross 1 at the same sizes
// within two):
//   N          n + m:  2     5     8     10    14    20    32    48    64
//   4 .. 32           1.3   1.3   1.2   1.2   1.2   1.15  1.1   1.05  0.95
//   128               1.3   1.2   1.2   1.15  1.1   1.0   0.9   0.85
//   512               1.4   1.25  1.1   1.1   1.0   0.85  0.75
//   2048              1.7   1.3   1.1   1.0   0.85  0.65
//   100000            2.7   1.6   1.2   1.0   0.7   0.5
// One step has no coupling to form (n + m = 96: 1.0 .. 1.15).
bool kalman_on_alu(long long N, int n, int m) {
  if (N == 1) return n + m <= 96;
  return n + m <= 48 && n + m <= 10 + 1280 / N;
}

cudaError_t launch_kalman_assemble(const KalmanArgs &a, DevStatus *st, int sms, cudaStream_t s) {
  if (a.N > kalman_max_steps(a.n, a.m)) return cudaErrorInvalidValue;
  if (kalman_on_alu(a.N, a.n, a.m)) {
    const int nt = ntiles(a.n), mt = ntiles(a.m);
    k_kalman_products_alu<<<(unsigned)(a.N * (nt * nt + mt * nt + 1)), kThreads, 0, s>>>(a);
    k_kalman_diag_alu<<<(unsigned)(a.N * (nt * nt + 1)), kThreads, 0, s>>>(a);
    return cudaGetLastError();
  }
  const bool pair = a.n <= 64;
  const void *kernels[2] = {pair ? (const void *)k_kalman_tc<0, true> : (const void *)k_kalman_tc<0, false>,
                            pair ? (const void *)k_kalman_tc<1, true> : (const void *)k_kalman_tc<1, false>};
  cudaError_t e = cudaSuccess;
  for (const void *k : kernels)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kKmSmem);
  if (e == cudaSuccess) {
    k_kalman_prepare<<<(unsigned)a.N, kalman_pad(a.n) + kalman_pad(a.m) <= 128 ? 128 : 256, 0, s>>>(a);
    e = cudaGetLastError();
  }
  for (int i = 0; i < 2 && e == cudaSuccess; ++i) {
    const int tn = (a.n + 63) / 64, tm = i || a.rinv_diag ? 0 : (a.m + 63) / 64;
    const long long tasks = kalman_groups(a.N, a.n) * kalman_row_tiles(a.n) * (tn + tm);
    const unsigned grid = (unsigned)(tasks < sms ? tasks : sms);
    void *args[] = {(void *)&a, (void *)&st};
    e = cudaLaunchKernel(kernels[i], dim3(grid), dim3(kWdThreads<double>), args, kKmSmem, s);
  }
  if (e != cudaSuccess || !a.B) return e;
  k_kalman_rhs<<<(unsigned)a.N, kThreads, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace bdss
