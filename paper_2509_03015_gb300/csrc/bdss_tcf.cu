// Factorisation of one level for blocks up to n = 64 with the coupling
// solves and the Schur products (Algorithm 1's trsm, Algorithm 3) on the
// tensor cores, two launches per level:
//
//   k_tcf_diag   per position of the level: the updates that the previous
//                level's eliminations left pending on it are applied
//                (Assemble); an odd position is then factored on the FP64
//                (FP32) ALU: L = chol(D), y = L^{-1} b, X = L^{-1}.
//   k_tcf_schur  per eliminated block, on the tensor cores by digit products
//                (bdss_slice.cuh): P = [W_L^T; W_R^T] = [A_{j,j-1}^T; A_{j+1,j}] X^T
//                (both factors scaled along their common index by D's diagonal),
//                then the products of P with itself, which hold everything
//                the elimination leaves behind:
//                  W_L^T W_L -> left separator's D,  W_R^T W_R -> right one's,
//                  -W_R^T W_L = S_{s+2,s},           P y -> both b.
//
// A separator has two eliminated neighbours, in different CTAs: each leaves
// its update in a buffer of its own and the next launch adds the two in a
// fixed order, so results do not depend on scheduling.
//
// The factor storage is that of the persistent kernel: L in Ld (FP32: L^{-1}),
// W^T in Wb, the level's couplings in Wb before their W -- except that the
// couplings a next level reads by columns (even slots: A_{j,j-1} of its
// eliminated blocks) are left transposed, so that every row of the second
// kernel's operands is contiguous.
#include "bdss_launch.h"
#include "bdss_slice_cta.cuh"
#include "bdss_tcf.h"

namespace bdss {

namespace {

constexpr int kDiagThreads = 128;   // levels of many blocks: several CTAs share an SM
constexpr int kSchurThreads = 512;
template <typename T> constexpr uint32_t kBufCols = SliceFmt<T>::kDig * kSlCols;  // accumulators of one column tile
template <typename T> constexpr uint32_t kTmem = sizeof(T) == 8 ? 512 : 256;       // a power of two
template <typename T> constexpr int kSchurCtas = sizeof(T) == 8 ? 1 : 2;            // per SM

template <typename T>
__global__ void __launch_bounds__(256) k_tcf_diag(const __grid_constant__ Args<T> a, const TcfLevel<T> w, int l,
                                                  int fold_all) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flag, s_go, s_cnt[8];
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;
  __syncthreads();
  if (!s_go) return;
  const int n = a.p.n, d = a.d, np = (n + 7) & ~7, ld = ldstride(np);
  const size_t nn = (size_t)n * n, nd = (size_t)n * d;
  const long long Nl = a.p.Nl[l], nE = Nl / 2, t = blockIdx.x;
  const bool elim = !fold_all && t < nE;
  const long long j = fold_all ? t : elim ? 2 * t + 1 : 2 * (t - nE);
  const long long orig = j << l;
  T *s = reinterpret_cast<T *>(smem_raw), *sB = s + (size_t)np * ld, *cbuf = sB + (size_t)d * ld;
  // the eliminated neighbours at level l - 1 are its blocks m = j - 1 (this
  // position is its right separator) and m = j (its left one)
  const bool hasM = l > 0 && j >= 1, hasP = l > 0 && j < a.p.Nl[l > 0 ? l - 1 : 0] / 2;
  const T *CM = w.C + (size_t)(2 * (j - 1) + 1) * nn, *CP = w.C + (size_t)(2 * j) * nn;
  if (l <= 1) stage_sym_lower(s, ld, a.A_diag + (size_t)orig * nn, n);  // the separators of level 0 are still A
  else stage_lower(s, ld, a.Ld + (size_t)orig * nn, n);
  if (l > 0)
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      const int i = e / n, c = e - i * n;
      if (c <= i) {
        T v = s[i * ld + c];
        if (hasM) v -= ldcg(CM + e);
        if (hasP) v -= ldcg(CP + e);
        s[i * ld + c] = v;
      }
    }
  if (d > 0) {
    const size_t bo = (size_t)orig * nd;
    const T *bM = w.cb + (size_t)(2 * (j - 1) + 1) * nd, *bP = w.cb + (size_t)(2 * j) * nd;
    for (int e = threadIdx.x; e < n * d; e += blockDim.x) {
      const int i = e / d, c = e - i * d;
      T v;
      if (l <= 1 && a.B64) v = (T)ldcg(a.B64 + bo + e);
      else if (l <= 1 && a.Bt) v = ldcg(a.Bt + bo + e);
      else v = ldcg(a.Y + bo + e);
      if (hasM) v -= ldcg(bM + e);
      if (hasP) v -= ldcg(bP + e);
      sB[c * ld + i] = v;
    }
  }
  __syncthreads();
  T *Lg = a.Ld + (size_t)orig * nn;
  if ((elim || fold_all) && threadIdx.x < kMaxN) {  // before the factorisation's first barrier and writes
    const int i = threadIdx.x;
    w.E[orig * kMaxN + i] = i < n ? (short)sl_half_exp(s[i * ld + i]) : (short)0;
  }
  if (elim) {
    for (int e = threadIdx.x; e < (np - n) * np; e += blockDim.x) {
      const int i = n + e / np, c = e % np;
      if (c <= i) s[i * ld + c] = T(i == c);
    }
    if (chol_inverse(s, ld, np, cbuf, s_cnt, &s_flag)) {
      if (threadIdx.x == 0) set_status(a.st, kStNotSPD, l, orig);
      return;
    }
    T *Xg = w.X + (size_t)t * nn;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      const int i = e / n, c = e - i * n;
      const T x = c <= i ? s[c * ld + i] : T(0);  // X[i][c] is in the upper triangle
      Xg[e] = x;
      // FP64: L with X^T above it; FP32: X
      if (!kStoreInverse<T>) Lg[e] = s[i * ld + c];
      else if (c <= i) Lg[e] = x;
    }
  } else {
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      const int i = e / n, c = e - i * n;
      if (c <= i) Lg[e] = s[i * ld + c];
    }
  }
  for (int e = threadIdx.x; e < n * d; e += blockDim.x) {
    if (elim) {  // y = L^{-1} b, threads along the rows: X[i][q] is s[q ld + i]
      const int c = e / n, i = e - c * n;
      const T *b = sB + c * ld;
      T v = T(0);
      for (int q = 0; q <= i; ++q) v = fma(s[q * ld + i], b[q], v);
      a.Y[(size_t)orig * nd + (size_t)i * d + c] = v;
    } else {
      const int i = e / d, c = e - i * d;
      a.Y[(size_t)orig * nd + e] = sB[c * ld + i];
    }
  }
}

constexpr int kStageRow = 48;               // bytes of a staged output row: 32 and a pad
constexpr int kStageWarp = 32 * kStageRow;  // bytes of a warp's output stage
constexpr int kWarps = kSchurThreads / 32;
// the column tiles' space, which also holds P (128 x 64) between its rounds
template <typename T> constexpr size_t kBSpace =
    (size_t)SliceFmt<T>::kDig * 2 * kSlBSlab > 128 * 64 * sizeof(T) ? (size_t)SliceFmt<T>::kDig * 2 * kSlBSlab
                                                                    : 128 * 64 * sizeof(T);
template <typename T> constexpr size_t schur_smem() {
  return (size_t)SliceFmt<T>::kDig * kSlASlab + kBSpace<T> + kWarps * kStageWarp + 1024;
}

template <typename T> struct Pair { T x, y; };
template <> struct __align__(16) Pair<double> { double x, y; };
template <> struct __align__(8) Pair<float> { float x, y; };

__device__ __forceinline__ Pair<double> ldcg_pair(const double *p) {
  const double2 x = __ldcg(reinterpret_cast<const double2 *>(p));
  return {x.x, x.y};
}
__device__ __forceinline__ Pair<float> ldcg_pair(const float *p) {
  const float2 x = __ldcg(reinterpret_cast<const float2 *>(p));
  return {x.x, x.y};
}

// Entries k, k + 1 of a contiguous row of n (zero from n on).
template <typename T, typename S>
__device__ __forceinline__ Pair<T> load_pair(const S *p, int k, int n, bool pairs) {
  Pair<T> v{T(0), T(0)};
  if (k < n) {
    if (pairs) {
      const Pair<S> x = ldcg_pair(p + k);
      v.x = (T)x.x;
      v.y = (T)x.y;
    } else {
      v.x = (T)ldcg(p + k);
      if (k + 1 < n) v.y = (T)ldcg(p + k + 1);
    }
  }
  return v;
}

// kNP = 64: a tile of 128 rows is one eliminated block (its W_L^T rows, then
// its W_R^T rows); kNP = 32 (n <= 32): two blocks, 32 rows per coupling.
//
// A tile takes rounds of products, each waited for and drained before the
// next: 0: the couplings times X^T (P); 1: P times its W_L^T rows; 2: P times
// its W_R^T rows; then P times y, 16 right-hand sides a round.
//
// What bounds it: issue slots of the integer digit work, with sixteen warps
// in one CTA per SM (the digits of a 128 x 64 FP64 tile are 128 KB).  Two
// things decide its speed.  Every global access is by whole 32-byte sectors
// (a warp takes rows, results pass through a stage).  And the code is small:
// one loop each for cutting rows, for issuing and for draining serves all
// rounds -- with the loops unrolled into each round the kernel was 260 KB of
// instructions, every pass over a tile missed the instruction cache, and a
// tile took 117,000 cycles.  N = 16384, n = 64: 4.0 ms over all levels (the
// products alone took the FP64 ALU 15.6 ms).
template <typename T, int kNP>
__global__ void __launch_bounds__(kSchurThreads, kSchurCtas<T>)
    k_tcf_schur(const __grid_constant__ Args<T> a, const TcfLevel<T> w, int l) {
  constexpr int kDig = SliceFmt<T>::kDig;
  constexpr int G = 64 / kNP;             // blocks per tile
  constexpr int NC = kNP / 4;             // columns of a tile row per thread (four threads per row)
  constexpr int LPR = kNP / 2;            // lanes per row (two entries each) where a warp takes rows
  constexpr int RPW = 32 / LPR;           // rows a warp takes at once
  constexpr int kBBytes = kDig * kSlBSlab;
  constexpr int kLdRaw = kNP + 1;         // row stride of the raw couplings of level 0
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t s_bar;
  __shared__ uint32_t s_tmem;
  __shared__ int s_ok, s_go;
  __shared__ int ex_row[kSlRows + 64];    // exponents of the A rows, then of the X rows
  __shared__ int ex_y[2][16];
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;
  __syncthreads();
  if (!s_go) return;
  unsigned char *A = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char *B0 = A + (size_t)kDig * kSlASlab;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char *stage = B0 + kBSpace<T> + warp * kStageWarp;
  T *raw = reinterpret_cast<T *>(B0);
  const int n = a.p.n, d = a.d, KS = (n + 15) / 16;
  const size_t nn = (size_t)n * n, nd = (size_t)n * d;
  const long long Nl = a.p.Nl[l], nE = Nl / 2, tasks = (nE + G - 1) / G;
  const bool pairs = (n & 1) == 0;                     // pairs of a row are aligned
  const bool segs = ((n * (int)sizeof(T)) & 15) == 0;  // 16-byte pieces of a row are aligned
  const bool flip = l + 1 < a.p.L;                     // even couplings of the next level are left transposed
  if (tid == 0) {
    mbar_init(&s_bar, 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&s_tmem, kTmem<T>);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  uint32_t ph = 0;
  bool ok = true;
  T *W = a.Wb + (size_t)a.p.off[l] * nn;
  const T *E = W;  // the level's couplings (level 0: the caller's A_sub)
  // where a warp takes rows: its lane's row among RPW and its entries k, k + 1
  const int sub = lane / LPR, k = 2 * (lane % LPR);
  // draining: TMEM lane = tile row, hw = which quarter of the columns
  const int quarter = warp & 3, hw = warp >> 2, row0 = 32 * quarter, row = row0 + lane;
  const int rblk = kNP == 64 ? 0 : row >> 6, rside = kNP == 64 ? row >> 6 : (row >> 5) & 1, rc = row & (kNP - 1);
  const uint32_t lane_base = tmem + ((uint32_t)row0 << 16);
  const int ctile = kNP == 64 ? hw >> 1 : rblk, tcol = kNP == 64 ? 16 * (hw & 1) : 8 * hw;
  constexpr int kPiece = 16 / sizeof(T);  // entries per 16-byte piece
  constexpr int kPieces = 64 / kPiece;    // pieces of a row of 64
  // row r of P in the column tiles' space, its pieces permuted by r (free of
  // bank conflicts by rows and by columns)
  auto p_piece = [&](int r, int pc) { return B0 + (size_t)r * (64 * sizeof(T)) + ((pc ^ (r & (kPieces - 1))) << 4); };
  // largest exponent of a row from its lanes' entries
  auto row_max = [&](int ex) {
    if constexpr (LPR == 32) {
      ex = __reduce_max_sync(0xffffffffu, ex);
    } else {
#pragma unroll
      for (int o = 1; o < LPR; o <<= 1) ex = max(ex, __shfl_xor_sync(0xffffffffu, ex, o));
    }
    return ex;
  };
  auto row_exp = [&](Pair<T> v, int *ex_at) {
    const int ex = row_max(max(sl_exp(v.x), sl_exp(v.y)));
    if (k == 0) *ex_at = sl_row_exp<T>(ex);
    return ex;
  };

  for (long long t = blockIdx.x; t < tasks && ok; t += gridDim.x) {
    const long long m0 = t * G;
    const bool anyR = 2 * m0 + 2 < Nl;
    if (l == 0) {
      // the caller's A_{j,j-1} row by row into the column tiles' space: their
      // columns are the W_L rows
      for (int e = tid; e < G * n * n; e += kSchurThreads) {
        const int blk = e / (n * n), f = e - blk * n * n, i = f / n, c = f - i * n;
        if (m0 + blk < nE) raw[(blk * kNP + i) * kLdRaw + c] = (T)ldcg(a.A_sub + (size_t)(2 * (m0 + blk)) * nn + f);
      }
      __syncthreads();
    }
    // scaling of entries k, k + 1: the couplings' down, X's up
    short2 ke[G];
#pragma unroll
    for (int b = 0; b < G; ++b)
      ke[b] = m0 + b < nE ? __ldcg(reinterpret_cast<const short2 *>(w.E + ((2 * (m0 + b) + 1) << l) * kMaxN + k))
                          : make_short2(0, 0);
    // ---- rows 0 .. 127: the couplings; 128 .. 191: X ---------------------------------
    // (level 0: X in a second pass, its digits take the place of the raw couplings)
    for (int r0 = 0; r0 < kSlRows + 64; r0 += 4 * kWarps * RPW) {
      if (l == 0 && r0 == kSlRows) __syncthreads();
      Pair<T> v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + (u * kWarps + warp) * RPW + sub;
        v[u].x = v[u].y = T(0);
        if (r < kSlRows) {
          const int blk = kNP == 64 ? 0 : r >> 6, side = kNP == 64 ? r >> 6 : (r >> 5) & 1, c = r & (kNP - 1);
          const long long m = m0 + blk;
          if (m < nE && c < n && (side == 0 || 2 * m + 2 < Nl)) {
            const size_t o = (size_t)(2 * m + side) * nn + (size_t)c * n;
            if (l > 0) {
              v[u] = load_pair<T>(E + o, k, n, pairs);
            } else if (side) {
              v[u] = load_pair<T>(a.A_sub + o, k, n, pairs);
            } else {
              if (k < n) v[u].x = raw[(blk * kNP + k) * kLdRaw + c];
              if (k + 1 < n) v[u].y = raw[(blk * kNP + k + 1) * kLdRaw + c];
            }
          }
        } else if (r < kSlRows + 64) {
          const int i = r - kSlRows, blk = kNP == 64 ? 0 : i >> 5, c = i & (kNP - 1);
          const long long m = m0 + blk;
          if (m < nE && c < n) v[u] = load_pair<T>(w.X + (size_t)m * nn + (size_t)c * n, k, n, pairs);
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = r0 + (u * kWarps + warp) * RPW + sub, i = r - kSlRows;
        if (r >= kSlRows + 64) continue;  // kNP = 32: the same for the whole warp
        unsigned char *at = r < kSlRows ? A + sl_off(r, k >> 3) : B0 + (i >> 5) * kBBytes + sl_off(i & 31, k >> 3);
        const short2 kb = ke[G > 1 && (r < kSlRows ? r >= 64 : i >= 32) ? G - 1 : 0];
        const int e0 = r < kSlRows ? -kb.x : kb.x, e1 = r < kSlRows ? -kb.y : kb.y;
        sl_prep(v[u].x, e0);
        sl_prep(v[u].y, e1);
        const int ex = row_max(max(sl_exp_at(v[u].x, e0), sl_exp_at(v[u].y, e1)));
        if (k == 0) ex_row[r] = ex;
        sl_store2<T>(v[u].x, v[u].y, ex, at + 2 * (k & 7), r < kSlRows ? kSlASlab : kSlBSlab, e0, e1);
      }
    }
    const long long m = m0 + rblk;
    const bool wlive = m < nE && (rside == 0 || 2 * m + 2 < Nl);  // the same for a warp's rows
    const int rounds = 3 + (d + 15) / 16;
#pragma unroll 1
    for (int rd = 0; rd < rounds; ++rd) {
      if (rd == 2 && !anyR) continue;
      const int d0 = 16 * (rd - 3);
      // ---- operands of the round ---------------------------------------------------------
      if (rd == 1) {
        // P stored (as W^T) and cut into digits
#pragma unroll 4
        for (int it = 0; it < kSlRows / (kWarps * RPW); ++it) {
          const int r = (it * kWarps + warp) * RPW + sub;
          const int blk = kNP == 64 ? 0 : r >> 6, side = kNP == 64 ? r >> 6 : (r >> 5) & 1, c = r & (kNP - 1);
          const long long mm = m0 + blk;
          const Pair<T> v = *reinterpret_cast<const Pair<T> *>(p_piece(r, k / kPiece) + (k % kPiece) * sizeof(T));
          if (mm < nE && c < n && k < n && (side == 0 || 2 * mm + 2 < Nl)) {
            T *Wr = W + (size_t)(2 * mm + side) * nn + (size_t)c * n + k;
            if (pairs) {
              *reinterpret_cast<Pair<T> *>(Wr) = v;
            } else {
              Wr[0] = v.x;
              if (k + 1 < n) Wr[1] = v.y;
            }
          }
          const int ex = row_exp(v, ex_row + r);
          sl_store2<T>(v.x, v.y, ex, A + sl_off(r, k >> 3) + 2 * (k & 7), kSlASlab);
        }
        __syncthreads();
      }
      if (rd == 1 || rd == 2) {
        // column tiles <- the 64 rows of one side (kNP = 32: 32 of each block)
        const int side = rd - 1;
#pragma unroll 4
        for (int e = tid; e < kDig * 64 * 8; e += kSchurThreads) {  // 16-byte groups
          const int p = e >> 9, rr = (e >> 3) & 63, g = e & 7;
          const int src = kNP == 64 ? 64 * side + rr : 64 * (rr >> 5) + 32 * side + (rr & 31);
          *reinterpret_cast<uint4 *>(B0 + (rr >> 5) * kBBytes + p * kSlBSlab + (rr & 31) * 128 + g * 16) =
              *reinterpret_cast<const uint4 *>(A + p * kSlASlab + src * 128 + g * 16);
        }
      }
      if (rd >= 3 && warp < 16 * G / RPW) {  // y: row r of 16 (of each block)
        const int rr = warp * RPW + sub, blk = rr >> 4, r = rr & 15;
        const long long mm = m0 + blk;
        Pair<T> v{T(0), T(0)};
        if (mm < nE && d0 + r < d) {
          const T *y = a.Y + (size_t)((2 * mm + 1) << l) * nd + d0 + r;
          if (k < n) v.x = ldcg(y + (size_t)k * d);
          if (k + 1 < n) v.y = ldcg(y + (size_t)(k + 1) * d);
        }
        const int ex = row_exp(v, &ex_y[blk][r]);
        sl_store2<T>(v.x, v.y, ex, B0 + blk * kBBytes + sl_off(r, k >> 3) + 2 * (k & 7), 16 * 128);
      }
      // every thread's operands before the MMAs that read them, its TMEM reads
      // before the MMAs that overwrite them
      fence_proxy_async_smem();
      tc_fence_before();
      __syncthreads();
      const int wu = __shfl_sync(0xffffffffu, warp, 0);
      if (wu < 2) {  // a warp per column tile
        tc_fence_after();
        if (sl_elect()) {
          const int cols = rd < 3 ? kSlCols : 16;
          // kNP = 64: rows 0 .. 31 of the lower triangular X have 32 entries
          if (wu == 0) sl_issue<T>(tmem, A, B0, cols, rd == 0 ? min(KS, 2) : KS);
          else if (rd < 3 || G > 1) sl_issue<T>(tmem + kBufCols<T>, A, B0 + kBBytes, cols, KS);
          tc_commit(&s_bar);
        }
        __syncwarp();
      }
      if (!mbar_wait_cta(&s_bar, ph, a.timeout_ns, &s_ok)) {
        if (tid == 0) set_status(a.st, kStTimeout, l, -1);
        // wait again (bounded) for the products in flight before TMEM is freed
        mbar_wait_cta(&s_bar, ph, a.timeout_ns, &s_ok);
        ok = false;
        break;
      }
      ph ^= 1;
      tc_fence_after();
      // ---- results of the round ------------------------------------------------------------
      //   0: P into the column tiles' space;
      //   1: left D (lower), the next level's coupling;  2: right D, the
      //      coupling if it is left transposed;  3 ..: right-hand sides
      const bool even = flip && (m & 1) == 0;
      T *dst = nullptr;
      bool lower = false, negate = false;
      int cols = NC;
      if (rd == 1 || rd == 2) {
        if (rside == rd - 1) {
          dst = w.C + (size_t)(2 * m + rside) * nn;
          lower = true;
        } else if (2 * m + 2 < Nl && even == (rd == 2)) {
          dst = a.Wb + ((size_t)a.p.off[l + 1] + (size_t)m) * nn;
          negate = true;
        }
        if (!dst || !wlive) cols = 0;
      } else if (rd >= 3) {
        dst = w.cb + (size_t)(2 * m + rside) * nd;
        cols = 4;
        if (!wlive || d0 + 4 * hw >= d) cols = 0;
      }
      const uint32_t acc_base = lane_base + (uint32_t)(rd < 3 ? ctile : rblk) * kBufCols<T> +
                                (uint32_t)(rd < 3 ? tcol : 4 * hw);
      const int tstep = rd < 3 ? kSlCols : 16;
      // exponents of the columns this thread drains
      const int *exc = rd == 0   ? ex_row + kSlRows + 32 * ctile + tcol
                       : rd < 3 ? ex_row + (kNP == 64 ? 64 * (rd - 1) : 64 * rblk + 32 * (rd - 1)) + hw * NC
                                : ex_y[rblk] + 4 * hw;
      const int ea = ex_row[row];
#pragma unroll 1
      for (int c = 0; c < cols; c += 4) {
        const int c0 = hw * NC + c;  // column of the n x n result (rounds 1, 2)
        if (rd > 0 && rd < 3 && (c0 >= n || (lower && c0 > (rc | 31)))) continue;  // warp-uniform
        uint32_t acc[kDig][4];
#pragma unroll
        for (int q = 0; q < kDig; ++q) tmem_ld4(acc_base + (uint32_t)(q * tstep + c), acc[q]);
        tmem_ld_wait();
        T v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float f[kDig];
#pragma unroll
          for (int q = 0; q < kDig; ++q) f[q] = __uint_as_float(acc[q][e]);
          v[e] = sl_value(f, ea, exc[c + e]);
        }
        if (rd == 0) {
#pragma unroll
          for (int e = 0; e < 4 / kPiece; ++e)
            *reinterpret_cast<uint4 *>(p_piece(row, c0 / kPiece + e)) = *reinterpret_cast<const uint4 *>(v + e * kPiece);
        } else if (rd < 3) {
          if (negate) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = -v[e];
          }
          // through the warp's stage, to memory in pieces of 16 bytes (a D update
          // with its upper triangle, which is never read)
          __syncwarp();
#pragma unroll
          for (int e = 0; e < 4 / kPiece; ++e)
            *reinterpret_cast<uint4 *>(stage + lane * kStageRow + 16 * e) = *reinterpret_cast<const uint4 *>(v + e * kPiece);
          __syncwarp();
          const int rb = row0 & (kNP - 1);
          if (segs) {
            constexpr int PR = 4 / kPiece;  // pieces per row
#pragma unroll
            for (int u = 0; u < PR; ++u) {
              const int rr = (32 / PR) * u + lane / PR, pc = lane % PR, c2 = c0 + pc * kPiece;
              const uint4 x = *reinterpret_cast<const uint4 *>(stage + rr * kStageRow + 16 * pc);
              if (rb + rr < n && c2 < n) *reinterpret_cast<uint4 *>(dst + (size_t)(rb + rr) * n + c2) = x;
            }
          } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int rr = 8 * u + (lane >> 2), c2 = c0 + (lane & 3);
              const T x = *reinterpret_cast<const T *>(stage + rr * kStageRow + (lane & 3) * sizeof(T));
              if (rb + rr < n && c2 < n) dst[(size_t)(rb + rr) * n + c2] = x;
            }
          }
        } else if (rc < n) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (d0 + 4 * hw + e < d) dst[(size_t)rc * d + d0 + 4 * hw + e] = v[e];
        }
      }
      // P complete before it is cut; the exponents and column tiles of the
      // round have been read before the next one's
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmem<T>);
}

// The top block (one block left at level L): the last level's pending update,
// its FP64 factor and inverse, x_0 = X^T (X b_0).
template <typename T>
__global__ void __launch_bounds__(256) k_tcf_top(const __grid_constant__ Args<T> a, const TcfLevel<T> w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flag, s_go, s_cnt[8];
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;
  __syncthreads();
  if (!s_go) return;
  const int n = a.p.n, d = a.d, np = (n + 7) & ~7, ld = ldstride(np), L = a.p.L;
  double *s = reinterpret_cast<double *>(smem_raw), *sB = s + (size_t)np * ld, *cbuf = sB + (size_t)2 * d * ld;
  for (int e = threadIdx.x; e < np * np; e += blockDim.x) {
    const int i = e / np, c = e - i * np;
    if (c > i) continue;
    double v = i == c;
    if (i < n) {
      T x = L > 1 ? ldcg(a.Ld + (size_t)i * n + c)
                  : T(0.5) * ((T)ldcg(a.A_diag + (size_t)i * n + c) + (T)ldcg(a.A_diag + (size_t)c * n + i));
      x -= ldcg(w.C + (size_t)i * n + c);
      v = (double)x;
    }
    s[i * ld + c] = v;
  }
  for (int e = threadIdx.x; e < n * d; e += blockDim.x) {
    const int i = e / d, c = e - i * d;
    T v = L > 1 ? ldcg(a.Y + e) : a.B64 ? (T)ldcg(a.B64 + e) : ldcg(a.Bt + e);
    v -= ldcg(w.cb + e);
    sB[c * ld + i] = (double)v;
  }
  __syncthreads();
  if (threadIdx.x < kMaxN) {
    const int i = threadIdx.x;
    w.E[i] = i < n ? (short)sl_half_exp(s[i * ld + i]) : (short)0;
  }
  if (chol_inverse(s, ld, np, cbuf, s_cnt, &s_flag)) {
    if (threadIdx.x == 0) set_status(a.st, kStNotSPD, L, 0);
    return;
  }
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int i = e / n, c = e - i * n;
    a.Ltop[e] = c <= i ? s[i * ld + c] : 0.0;
  }
  double *sY = sB + (size_t)d * ld;
  for (int e = threadIdx.x; e < n * d; e += blockDim.x) {  // X[i][q] is s[q ld + i]
    const int c = e / n, i = e - c * n;
    double v = 0.0;
    for (int q = 0; q <= i; ++q) v = fma(s[q * ld + i], sB[c * ld + q], v);
    sY[c * ld + i] = v;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n * d; e += blockDim.x) {
    const int c = e / n, i = e - c * n;
    double v = 0.0;
    for (int q = i; q < n; ++q) v = fma(s[i * ld + q], sY[c * ld + q], v);
    const size_t o = (size_t)i * d + c;
    a.Y[o] = (T)v;
    if (a.X64) a.X64[o] = a.x_accumulate ? a.X64[o] + v : v;
  }
}

// One level of a solve with the stored inverses.
//   kUp:   separator s: b_s -= Wt(s-1) y_{s-1} + Wt(s) y_{s+1}; if s is eliminated
//          at the next level (odd, and that level is not the blocks left for the
//          top sweep), y_s = X_s b_s.  first: no level before the first
//          elimination yet, y_j = X_j b_j of level 0.
//   down:  eliminated j: t = y_j - Wt(j-1)^T x_{j-1} - Wt(j)^T x_{j+1}, x_j = X_j^T t.
// Thread (i, g): row i of the result, a quarter of either sum; it loads all of
// its matrix entries at once, before any of them is used, and keeps them for
// every four columns of the right-hand sides.
//
// What bounds it: few blocks, two trips to memory and four barriers (a level of
// one 64 x 64 block: substitutions by one warp took 74 us); many, the FP64 pipe
// (5 n^2 d / 2 multiply-adds a block on the way down).
constexpr int kSolveCols = 4;
template <typename T, bool kUp>
__global__ void __launch_bounds__(256, 2) k_tcf_solve(const __grid_constant__ Args<T> a, int l, int first) {
  __shared__ T sV[2][kMaxN][kSolveCols], sR[4][kMaxN][kSolveCols], sT[kMaxN][kSolveCols];
  if (ld_relaxed_i32(&a.st->status) != 0) return;
  const int n = a.p.n, d = a.d, i = threadIdx.x & (kMaxN - 1), g = threadIdx.x / kMaxN;
  const size_t nn = (size_t)n * n, nd = (size_t)n * d;
  const long long m = blockIdx.x, Nl = a.p.Nl[l];
  const long long pos = kUp && !first ? 2 * m : 2 * m + 1, orig = pos << l;
  const bool hasM = !first && pos >= 1, hasP = !first && pos + 1 < Nl;
  // a triangular product follows, unless the next level is the serial top's
  const bool tri = !kUp || first || ((m & 1) && l + 1 < a.p.L);
  const bool raw = kUp && l == 0 && (a.B64 || a.Bt);
  // matrix entries: W of slot pos - 1 (g < 2) or pos (g >= 2), X of this block
  T wv[kMaxN / 2], xv[kMaxN / 4];
  const bool mine = i < n && (g < 2 ? hasM : hasP);
  const T *Wg = a.Wb + (size_t)(a.p.off[l] + pos - (g < 2 ? 1 : 0)) * nn;
#pragma unroll
  for (int u = 0; u < kMaxN / 2; ++u) {
    const int v = (g & 1) * (kMaxN / 2) + u;
    wv[u] = mine && v < n ? (kUp ? Wg[(size_t)i * n + v] : Wg[(size_t)v * n + i]) : T(0);
  }
  // FP64 keeps X^T above the diagonal of Ld (1 / L_ii on it), FP32 X below
  const T *Xg = a.Ld + (size_t)orig * nn;
#pragma unroll
  for (int u = 0; u < kMaxN / 4; ++u) {
    const int c = 4 * u + g;
    const bool in = tri && i < n && c < n && (kUp ? c <= i : c >= i);
    const int r0 = kUp ? i : c, c0 = kUp ? c : i;  // X[r0][c0]
    xv[u] = in ? (kStoreInverse<T> ? Xg[(size_t)r0 * n + c0] : Xg[(size_t)c0 * n + r0]) : T(0);
  }
  for (int d0 = 0; d0 < d; d0 += kSolveCols) {
    const int dc = min(kSolveCols, d - d0);
    for (int e = threadIdx.x; e < 2 * kMaxN * kSolveCols; e += 256) {
      const int side = e / (kMaxN * kSolveCols), v = (e / kSolveCols) % kMaxN, c = e % kSolveCols;
      const bool in = v < n && c < dc && (side ? hasP : hasM);
      sV[side][v][c] = in ? ldcg(a.Y + (size_t)((side ? pos + 1 : pos - 1) << l) * nd + (size_t)v * d + d0 + c) : T(0);
    }
    __syncthreads();
    T acc[kSolveCols] = {};
    if (hasM || hasP) {
#pragma unroll
      for (int u = 0; u < kMaxN / 2; ++u)
#pragma unroll
        for (int c = 0; c < kSolveCols; ++c)
          if (c < dc) acc[c] = fma(wv[u], sV[g >> 1][(g & 1) * (kMaxN / 2) + u][c], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < kSolveCols; ++c) sR[g][i][c] = acc[c];
    __syncthreads();
    if (i < n && g < dc) {  // thread (i, g): column g
      const size_t o = (size_t)orig * nd + (size_t)i * d + d0 + g;
      const T base = !raw ? ldcg(a.Y + o) : a.B64 ? (T)ldcg(a.B64 + o) : ldcg(a.Bt + o);
      const T t = base - ((sR[0][i][g] + sR[1][i][g]) + (sR[2][i][g] + sR[3][i][g]));
      sT[i][g] = t;
      if (!tri) a.Y[o] = t;
    } else {
      sT[i][g] = T(0);
    }
    __syncthreads();
    if (!tri) continue;
#pragma unroll
    for (int c = 0; c < kSolveCols; ++c) acc[c] = T(0);
#pragma unroll
    for (int u = 0; u < kMaxN / 4; ++u)
#pragma unroll
      for (int c = 0; c < kSolveCols; ++c)
        if (c < dc) acc[c] = fma(xv[u], sT[4 * u + g][c], acc[c]);
#pragma unroll
    for (int c = 0; c < kSolveCols; ++c) sR[g][i][c] = acc[c];
    __syncthreads();
    if (i < n && g < dc) {
      const size_t o = (size_t)orig * nd + (size_t)i * d + d0 + g;
      const T x = (sR[0][i][g] + sR[1][i][g]) + (sR[2][i][g] + sR[3][i][g]);
      a.Y[o] = x;
      if (!kUp && a.X64) a.X64[o] = a.x_accumulate ? a.X64[o] + (double)x : (double)x;
    }
    // sR and sT are next written after two barriers
  }
}

// k_tcf_solve for many right-hand sides (FP64): the products with W as digit
// products, 16 columns at a time, the triangular one on the ALU.  One block a
// tile: its 128 A rows are the rows (up) or columns (down) of its two W, each
// multiplied by its own neighbour's vectors (B tile 0 or 1), so the halves of
// the result are added.
//
// On the way down the common index of W x runs over the separators' states:
// both factors are scaled along it (E; bdss_slice.cuh).
//
// With 16 columns the FP64 ALU needs 2.5 n^2 d multiply-adds a block and way
// (82,000 cycles at n = 64); here cutting W (the same for any d) and 16k cycles
// of triangular product remain.
constexpr int kTcRhs = 16;
constexpr int kTcLdX = kMaxN + 1;
constexpr size_t kTcSolveSmem = 8 * kSlASlab + 2 * 8 * kTcRhs * 128 +
                                (size_t)(kSlRows * kTcRhs + kMaxN * kTcRhs + kMaxN * kTcLdX) * sizeof(double) + 1024;
template <bool kUp>
__global__ void __launch_bounds__(1024, 1) k_tcf_solve_tc(const __grid_constant__ Args<double> a, const short *E, int l,
                                                          int first) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t s_bar[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_go, s_exA[kSlRows], s_exB[2 * kTcRhs], s_exP[8 * kSlRows];
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;
  __syncthreads();
  if (!s_go) return;
  WdCta<double> w;
  wd_begin(w, smem_raw, s_bar, &s_tmem, s_exA, s_exB, s_exP, a.timeout_ns);
  constexpr int kTileB = 8 * kTcRhs * 128;  // bytes of a B tile's digits
  double *red = reinterpret_cast<double *>(w.B + 2 * kTileB), *sT = red + kSlRows * kTcRhs, *sX = sT + kMaxN * kTcRhs;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, hw = warp >> 2, row0 = 32 * (warp & 3), row = row0 + lane;
  const uint32_t lane_base = w.tmem + ((uint32_t)row0 << 16);
  const int n = a.p.n, d = a.d, ks = (n + 15) >> 4;
  const size_t nn = (size_t)n * n, nd = (size_t)n * d;
  const long long Nl = a.p.Nl[l], count = !kUp || first ? Nl / 2 : (Nl + 1) / 2;
  const bool pairs = (n & 1) == 0;
  bool ok = true;
  for (long long m = blockIdx.x; m < count && ok; m += gridDim.x) {
    const long long pos = kUp && !first ? 2 * m : 2 * m + 1, orig = pos << l;
    const bool hasM = !first && pos >= 1, hasP = !first && pos + 1 < Nl;
    const bool tri = !kUp || first || ((m & 1) && l + 1 < a.p.L), raw = kUp && l == 0 && (a.B64 || a.Bt);
    const double *W0 = a.Wb + (size_t)(a.p.off[l] + pos - 1) * nn, *W1 = W0 + nn;
    // X (FP64 keeps X^T above the diagonal of Ld): X[i][q] at sX[q kTcLdX + i], q <= i
    double xv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int q = (tid >> 6) + 16 * u, i = tid & 63;
      xv[u] = tri && i < n && q <= i ? ldcg(a.Ld + (size_t)orig * nn + (size_t)q * n + i) : 0.0;
    }
    if (hasM || hasP) {
      if constexpr (kUp) {  // rows of W^T, a warp per row
        double v[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int r = 32 * u + warp, k = 2 * lane, i = r & 63;
          const double *src = (r < 64 ? W0 : W1) + (size_t)i * n + k;
          v[u][0] = v[u][1] = 0.0;
          if ((r < 64 ? hasM : hasP) && i < n && k < n) {
            if (pairs) {
              const double2 x = __ldcg(reinterpret_cast<const double2 *>(src));
              v[u][0] = x.x;
              v[u][1] = x.y;
            } else {
              v[u][0] = ldcg(src);
              if (k + 1 < n) v[u][1] = ldcg(src + 1);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int r = 32 * u + warp, k = 2 * lane;
          const int ex = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(sl_exp(v[u][0]), sl_exp(v[u][1])));
          if (lane == 0) w.exA[r] = sl_row_exp<double>(ex);
          sl_store2<double>(v[u][0], v[u][1], ex, w.A + sl_off(r, k >> 3) + 2 * (k & 7), kSlASlab);
        }
      } else {  // columns of W^T: thread (column, eight K entries)
        const int c = tid & 63, g = (tid >> 6) & 7, half = tid >> 9;
        const double *src = half ? W1 : W0;
        const bool live = half ? hasP : hasM;
        SlScale8 sc = {};
        if (live) sc = sl_scale8(E + ((half ? pos + 1 : pos - 1) << l) * kMaxN + 8 * g);
        double v[8];
        int ex = kSlNoEx;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int p = 8 * g + i;
          v[i] = live && c < n && p < n ? ldcg(src + (size_t)p * n + c) : 0.0;
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) ex = max(ex, sl_exp_at(v[i], -sc.at(i)));
        w.exP[g * kSlRows + 64 * half + c] = ex;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 8; ++q) ex = max(ex, w.exP[q * kSlRows + 64 * half + c]);
        if (g == 0) w.exA[64 * half + c] = ex;
        store8<double, -1>(v, ex, w.A + sl_off(64 * half + c, g), kSlASlab, sc);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) sX[((tid >> 6) + 16 * u) * kTcLdX + (tid & 63)] = xv[u];
    for (int d0 = 0; d0 < d && ok; d0 += kTcRhs) {
      const int i = tid >> 4, c = tid & 15;  // the result entry this thread forms
      const bool in = i < n && d0 + c < d;
      const size_t o = (size_t)orig * nd + (size_t)i * d + d0 + c;
      double t = !in ? 0.0 : !raw ? ldcg(a.Y + o) : a.B64 ? ldcg(a.B64 + o) : ldcg(a.Bt + o);
      if (hasM || hasP) {
        // B row of this warp: column d0 + r of the neighbour's vectors
        const int r = warp & 15, side = warp >> 4, k = 2 * lane;
        const double *src = a.Y + (size_t)((side ? pos + 1 : pos - 1) << l) * nd + d0 + r;
        const bool live = (side ? hasP : hasM) && d0 + r < d;
        const double v0 = live && k < n ? src[(size_t)k * d] : 0.0, v1 = live && k + 1 < n ? src[(size_t)(k + 1) * d] : 0.0;
        short2 ke = make_short2(0, 0);
        if constexpr (!kUp) {
          if (live) ke = __ldcg(reinterpret_cast<const short2 *>(E + ((side ? pos + 1 : pos - 1) << l) * kMaxN + k));
        }
        const int ex = __reduce_max_sync(0xffffffffu, max(sl_exp_nz(v0, ke.x), sl_exp_nz(v1, ke.y)));
        if (lane == 0) w.exB[warp] = ex;
        sl_store2<double>(v0, v1, ex, w.B + side * kTileB + sl_off(r, k >> 3) + 2 * (k & 7), kTcRhs * 128, ke.x, ke.y);
        fence_proxy_async_smem();
        tc_fence_before();
        __syncthreads();
        const int wu = __shfl_sync(0xffffffffu, warp, 0);
        if (wu < 2) {
          tc_fence_after();
          if (sl_elect()) {
            sl_issue<double>(w.tmem + 256 * wu, w.A, w.B + wu * kTileB, kTcRhs, ks);
            tc_commit(w.bar + wu);
          }
          __syncwarp();
        }
        ok = wd_wait<double>(w, row >> 6);
        if (ok) {
          uint32_t acc[8][2];
#pragma unroll
          for (int q = 0; q < 8; ++q)
            tmem_ld2(lane_base + (uint32_t)((row >> 6) * 256 + q * kTcRhs + 2 * hw), acc[q]);
          tmem_ld_wait();
          const int ea = w.exA[row];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float f[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) f[q] = __uint_as_float(acc[q][e]);
            red[row * kTcRhs + 2 * hw + e] = sl_value(f, ea, w.exB[(row >> 6) * kTcRhs + 2 * hw + e]);
          }
        }
        ok = wd_round_end<double>(w, true, ok);
        if (!ok) {
          if (tid == 0) set_status(a.st, kStTimeout, l, -1);
          break;
        }
        t -= red[i * kTcRhs + c] + red[(64 + i) * kTcRhs + c];
      }
      if (!tri) {
        if (in) a.Y[o] = t;
      } else {
        sT[i * kTcRhs + c] = in ? t : 0.0;
        __syncthreads();
        if (in) {
          double x = 0.0;
          if constexpr (kUp) {
            for (int q = 0; q <= i; ++q) x = fma(sX[q * kTcLdX + i], sT[q * kTcRhs + c], x);
          } else {
            for (int q = i; q < n; ++q) x = fma(sX[i * kTcLdX + q], sT[q * kTcRhs + c], x);
          }
          a.Y[o] = x;
          if (!kUp && a.X64) a.X64[o] = a.x_accumulate ? a.X64[o] + x : x;
        }
      }
      __syncthreads();
    }
  }
  wd_end(w);
}

size_t diag_smem(int n, int d, size_t esz) { const int np = (n + 7) & ~7;
  return ((size_t)(np + d) * ldstride(np) + 17 * kMaxN) * esz; }

}  // namespace

template <typename T>
cudaError_t tcf_configure(int n, int d) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const void *kernels[] = {(const void *)k_tcf_diag<T>, (const void *)k_tcf_top<T>, (const void *)k_tcf_schur<T, 32>,
                           (const void *)k_tcf_schur<T, 64>};
  for (const void *k : kernels) {
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e == cudaSuccess && k != kernels[0] && k != kernels[1] && schur_smem<T>() > (size_t)optin - fa.sharedSizeBytes)
      e = cudaErrorInvalidConfiguration;
  }
  if (sizeof(T) == 8) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute((const void *)k_tcf_solve_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kTcSolveSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute((const void *)k_tcf_solve_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)kTcSolveSmem);
  }
  if (e == cudaSuccess && diag_smem(n, d, sizeof(T)) > (size_t)optin - 64) e = cudaErrorInvalidConfiguration;
  return e;
}

template <typename T>
cudaError_t launch_tcf_diag(const Args<T> &a, const TcfLevel<T> &c, int l, int fold_all, int sms, cudaStream_t s) {
  const long long Nl = a.p.Nl[l], nE = Nl / 2;
  const long long tasks = fold_all ? Nl : nE + (l > 0 ? Nl - nE : 0);
  // with few blocks the pivot chain of one block is the level's time: more
  // threads per block shorten its updates
  const int threads = nE <= 2 * sms ? 256 : kDiagThreads;
  k_tcf_diag<T><<<(unsigned)tasks, threads, diag_smem(a.p.n, a.d, sizeof(T)), s>>>(a, c, l, fold_all);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_tcf_schur(const Args<T> &a, const TcfLevel<T> &c, int l, int sms, cudaStream_t s) {
  const long long nE = a.p.Nl[l] / 2;
  const int G = a.p.n <= 32 ? 2 : 1;
  const long long tasks = (nE + G - 1) / G;
  const long long most = (long long)kSchurCtas<T> * sms;
  const unsigned grid = (unsigned)(tasks < most ? tasks : most);
  if (G == 2) k_tcf_schur<T, 32><<<grid, kSchurThreads, schur_smem<T>(), s>>>(a, c, l);
  else k_tcf_schur<T, 64><<<grid, kSchurThreads, schur_smem<T>(), s>>>(a, c, l);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_tcf_top(const Args<T> &a, const TcfLevel<T> &c, cudaStream_t s) {
  const int np = (a.p.n + 7) & ~7;
  const size_t smem = ((size_t)(np + 2 * a.d) * ldstride(np) + 17 * kMaxN) * sizeof(double);
  k_tcf_top<T><<<1, 256, smem, s>>>(a, c);
  return cudaGetLastError();
}

template <bool kUp>
static cudaError_t launch_solve_tc(const Args<double> &a, const short *E, int l, int first, long long count, int sms,
                                   cudaStream_t s) {
  const unsigned grid = (unsigned)(count < sms ? count : sms);
  k_tcf_solve_tc<kUp><<<grid, 1024, kTcSolveSmem, s>>>(a, E, l, first);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_tcf_up(const Args<T> &a, int l, int first, int sms, cudaStream_t s) {
  const long long count = first ? a.p.Nl[l] / 2 : (a.p.Nl[l] + 1) / 2;
  if constexpr (sizeof(T) == 8) {
    if (a.d > kTcfMinRhsTc) return launch_solve_tc<true>(a, nullptr, l, first, count, sms, s);
  }
  k_tcf_solve<T, true><<<(unsigned)count, 256, 0, s>>>(a, l, first);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_tcf_down(const Args<T> &a, const short *E, int l, int sms, cudaStream_t s) {
  const long long count = a.p.Nl[l] / 2;
  if constexpr (sizeof(T) == 8) {
    if (a.d > kTcfMinRhsTc) return launch_solve_tc<false>(a, E, l, 0, count, sms, s);
  }
  k_tcf_solve<T, false><<<(unsigned)count, 256, 0, s>>>(a, l, 0);
  return cudaGetLastError();
}

#define BDSS_TCF_INSTANTIATE(T)                                                                       \
  template cudaError_t tcf_configure<T>(int, int);                                                    \
  template cudaError_t launch_tcf_diag<T>(const Args<T> &, const TcfLevel<T> &, int, int, int, cudaStream_t); \
  template cudaError_t launch_tcf_schur<T>(const Args<T> &, const TcfLevel<T> &, int, int, cudaStream_t);        \
  template cudaError_t launch_tcf_top<T>(const Args<T> &, const TcfLevel<T> &, cudaStream_t);                     \
  template cudaError_t launch_tcf_up<T>(const Args<T> &, int, int, int, cudaStream_t);                                 \
  template cudaError_t launch_tcf_down<T>(const Args<T> &, const short *, int, int, cudaStream_t);
BDSS_TCF_INSTANTIATE(double)
BDSS_TCF_INSTANTIATE(float)

}  // namespace bdss
