// Factorisation of one level for blocks 64 < n <= 256 with its products on
// the tensor cores (digit products, bdss_slice.cuh).
//
// An eliminated block j is factored panel by panel (nb <= 64 columns, the
// same width for all but the last).  With its couplings and right-hand sides
// as further rows, the block is the matrix
//   [ D ; A_{j,j-1}^T ; A_{j+1,j} ; b^T ]   (n, n, n and d rows of n columns)
// and eliminating D turns it into [ L ; W_L^T ; W_R^T ; y^T ] = [...] L^{-T}.
// Per panel k two launches:
//   k_wide_diag   the diagonal tile on the FP64 (FP32) ALU: L_kk = chol, X_kk
//                 = L_kk^{-1};
//   k_wide_panel  every other row v: P_vk = (S_vk - sum_{p<k} P_vp L_kp^T) X_kk^T,
//                 and for rows of D their own diagonal tile, updated by P P^T.
// Then one launch forms what the separators receive (k_wide_schur): D, the
// next level's couplings, b.
//
// Every n x n operand is read along contiguous rows: couplings are stored as
// the rows the elimination needs (the even slots of a level, its eliminated
// blocks' left couplings, transposed), from the level-0 ingest on.  Couplings
// and their W^T share a slot of Wb, D and its L a slot of Ld (reciprocal
// diagonal), where a diagonal tile keeps X_kk^T above its diagonal for the
// downward pass.
#include "bdss_launch.h"
#include "bdss_slice.cuh"
#include "bdss_wide.h"

namespace bdss {

namespace {

constexpr int kWdThreads = 512;
constexpr int kWdWarps = kWdThreads / 32;
constexpr int kWdTile = 64;  // rows of a slot, columns of an output tile
template <typename T> constexpr int kWdStageRow = sizeof(T) == 8 ? 48 : 16;  // bytes of a staged output row
template <typename T> constexpr uint32_t kWdBufCols = SliceFmt<T>::kDig * kSlCols;  // accumulators of 32 columns
template <typename T> constexpr uint32_t kWdTmem = 2 * kWdBufCols<T>;
template <typename T> constexpr int kWdBBytes = SliceFmt<T>::kDig * kSlBSlab;
template <typename T> constexpr size_t wd_smem() {
  return (size_t)SliceFmt<T>::kDig * (kSlASlab + 2 * kSlBSlab) + (size_t)kWdWarps * 32 * kWdStageRow<T> + 1024;
}

// Panels: equal widths rounded up to 8 columns, so that the diagonal tiles'
// pivot chains, which are the critical path, are equally long.
__host__ __device__ inline WidePanels panels_of(int n) {
  const int nt = (n + kWdTile - 1) / kWdTile;
  return {nt, ((n + nt - 1) / nt + 7) / 8 * 8};
}

// 64 rows of an operand or result: entry (r, c) at p[r rs + c cs], c counted
// from the chunk's first column; rows from `rows` on are zero.
template <typename T>
struct Slot {
  T *p;
  long long rs, cs;
  int rows;
};

template <typename T>
__device__ __forceinline__ Slot<T> no_slot() {
  return {nullptr, 0, 0, 0};
}

template <typename T>
struct WdCta {
  unsigned char *A, *B, *stage;  // digit slabs, this warp's output stage
  uint32_t tmem;
  uint64_t *bar;
  int *exA, *exB, *exP, *s_ok;   // row exponents: A (128), B (64), partial (4 x 128)
  uint32_t ph;
  long long timeout_ns;
};

template <typename T>
__device__ __forceinline__ void load2(const T *p, T &x, T &y);
template <>
__device__ __forceinline__ void load2<double>(const double *p, double &x, double &y) {
  const double2 v = __ldcg(reinterpret_cast<const double2 *>(p));
  x = v.x;
  y = v.y;
}
template <>
__device__ __forceinline__ void load2<float>(const float *p, float &x, float &y) {
  const float2 v = __ldcg(reinterpret_cast<const float2 *>(p));
  x = v.x;
  y = v.y;
}

// Digits of the K columns [0, kc) of the slots a0, a1 (A rows 0 .. 63, 64 ..
// 127; skipped unless do_a) and b (B rows), a warp per row: all loads of the
// 192 rows first, then the cutting.
template <typename T>
__device__ __forceinline__ void wd_cut(const WdCta<T> &w, const Slot<T> &a0, const Slot<T> &a1, const Slot<T> &b,
                                       bool do_a, bool do_b, int kc, bool pairs) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = 2 * lane;
  T v[12][2];
#pragma unroll
  for (int u = 0; u < 12; ++u) {
    const Slot<T> &s = u < 4 ? a0 : u < 8 ? a1 : b;
    const int r = (u & 3) * kWdWarps + warp;
    v[u][0] = v[u][1] = T(0);
    if ((u < 8 ? do_a : do_b) && r < s.rows && k < kc) {
      const T *p = s.p + (long long)r * s.rs + (long long)k * s.cs;
      if (pairs && s.cs == 1) {
        load2(p, v[u][0], v[u][1]);
      } else {
        v[u][0] = ldcg(p);
        if (k + 1 < kc) v[u][1] = ldcg(p + s.cs);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 12; ++u) {
    if (!(u < 8 ? do_a : do_b)) continue;
    const int r = (u & 3) * kWdWarps + warp;
    const int ex = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(sl_exp(v[u][0]), sl_exp(v[u][1])));
    if (u < 8) {
      const int ra = 64 * (u >> 2) + r;
      if (lane == 0) w.exA[ra] = ex;
      sl_store2<T>(v[u][0], v[u][1], ex, w.A + sl_off(ra, k >> 3) + 2 * (k & 7), kSlASlab);
    } else {
      if (lane == 0) w.exB[r] = ex;
      sl_store2<T>(v[u][0], v[u][1], ex, w.B + (r >> 5) * kWdBBytes<T> + sl_off(r & 31, k >> 3) + 2 * (k & 7),
                   kSlBSlab);
    }
  }
}

// Eight consecutive K entries of one row -> 16 bytes of every digit slab.
template <typename T>
__device__ __forceinline__ void store8(const T *v, int ex, unsigned char *dst, int stride);
template <>
__device__ __forceinline__ void store8<double>(const double *v, int ex, unsigned char *dst, int stride) {
  unsigned w[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned long long u0 = sl_biased(v[2 * i], ex), u1 = sl_biased(v[2 * i + 1], ex);
    const unsigned h0 = (unsigned)(u0 >> 32), h1 = (unsigned)(u1 >> 32), l0 = (unsigned)u0, l1 = (unsigned)u1;
    sl_half_pairs(__byte_perm(h0, h1, 0x7632), w[i][1], w[i][0]);
    sl_half_pairs(__byte_perm(h0, h1, 0x5410), w[i][3], w[i][2]);
    sl_half_pairs(__byte_perm(l0, l1, 0x7632), w[i][5], w[i][4]);
    sl_half_pairs(__byte_perm(l0, l1, 0x5410), w[i][7], w[i][6]);
  }
#pragma unroll
  for (int p = 0; p < 8; ++p)
    *reinterpret_cast<uint4 *>(dst + p * stride) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
}
template <>
__device__ __forceinline__ void store8<float>(const float *v, int ex, unsigned char *dst, int stride) {
  unsigned w[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned u0 = sl_biased(v[2 * i], ex), u1 = sl_biased(v[2 * i + 1], ex);
    sl_half_pairs(__byte_perm(u0, u1, 0x7632), w[i][1], w[i][0]);
    sl_half_pairs(__byte_perm(u0, u1, 0x5410), w[i][3], w[i][2]);
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
    *reinterpret_cast<uint4 *>(dst + p * stride) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
}

// The A rows from registers: this thread's 16 columns of its row.  Contains
// CTA barriers.
template <typename T>
__device__ __forceinline__ void wd_cut_regs(const WdCta<T> &w, const T (&v)[16], int row, int hw) {
  int ex = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) ex = max(ex, sl_exp(v[i]));
  w.exP[hw * kSlRows + row] = ex;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 4; ++q) ex = max(ex, w.exP[q * kSlRows + row]);
  if (hw == 0) w.exA[row] = ex;
#pragma unroll
  for (int i = 0; i < 2; ++i) store8<T>(v + 8 * i, ex, w.A + sl_off(row, 2 * hw + i), kSlASlab);
}

// The product of the cut operands, waited for.  cols2: the second 32 columns
// as well; ks0 / ks1: K steps of either column tile.  False after a timeout.
template <typename T>
__device__ __forceinline__ bool wd_product(WdCta<T> &w, bool cols2, int ks0, int ks1) {
  // every thread's operands before the products that read them, its TMEM
  // reads before the products that overwrite them
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    tc_fence_after();
    sl_issue<T>(w.tmem, w.A, w.B, kSlCols, ks0);
    if (cols2) sl_issue<T>(w.tmem + kWdBufCols<T>, w.A, w.B + kWdBBytes<T>, kSlCols, ks1);
    tc_commit(w.bar);
  }
  if (!mbar_wait_cta(w.bar, w.ph, w.timeout_ns, w.s_ok)) {
    // wait again (bounded) for the products in flight before TMEM is freed
    mbar_wait_cta(w.bar, w.ph, w.timeout_ns, w.s_ok);
    return false;
  }
  w.ph ^= 1;
  tc_fence_after();
  return true;
}

// Four columns of the product from TMEM address `at`, as values.
template <typename T>
__device__ __forceinline__ void wd_drain4(uint32_t at, int ea, const int *exb, T (&v)[4]) {
  constexpr int kDig = SliceFmt<T>::kDig;
  uint32_t acc[kDig][4];
#pragma unroll
  for (int q = 0; q < kDig; ++q) tmem_ld4(at + (uint32_t)(q * kSlCols), acc[q]);
  tmem_ld_wait();
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float f[kDig];
#pragma unroll
    for (int q = 0; q < kDig; ++q) f[q] = __uint_as_float(acc[q][e]);
    v[e] = sl_value(f, ea, exb[e]);
  }
}

// Four columns of a warp's 32 rows to memory through the warp's stage, in
// 16-byte pieces where rows allow it.  dst: the warp's first row, first
// column; rows / cols: how many of them exist.  sub: subtract from what is
// there instead.
template <typename T>
__device__ __forceinline__ void wd_store4(unsigned char *stage, const T (&v)[4], T *dst, long long ld, int rows,
                                          int cols, bool segs, bool sub) {
  constexpr int kPiece = 16 / sizeof(T), PR = 4 / kPiece;
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int e = 0; e < PR; ++e)
    *reinterpret_cast<uint4 *>(stage + lane * kWdStageRow<T> + 16 * e) = *reinterpret_cast<const uint4 *>(v + e * kPiece);
  __syncwarp();
  if (segs) {
#pragma unroll
    for (int u = 0; u < PR; ++u) {
      const int rr = (32 / PR) * u + lane / PR, pc = lane % PR;
      uint4 x = *reinterpret_cast<const uint4 *>(stage + rr * kWdStageRow<T> + 16 * pc);
      if (rr < rows && pc * kPiece < cols) {
        uint4 *at = reinterpret_cast<uint4 *>(dst + rr * ld + pc * kPiece);
        if (sub) {
          uint4 o = __ldcg(at);
          T *ov = reinterpret_cast<T *>(&o);
          const T *xv = reinterpret_cast<const T *>(&x);
#pragma unroll
          for (int i = 0; i < kPiece; ++i) ov[i] -= xv[i];
          x = o;
        }
        *at = x;
      }
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int rr = 8 * u + (lane >> 2), c = lane & 3;
      const T x = *reinterpret_cast<const T *>(stage + rr * kWdStageRow<T> + c * sizeof(T));
      if (rr < rows && c < cols) {
        T *at = dst + rr * ld + c;
        *at = sub ? ldcg(at) - x : x;
      }
    }
  }
}

// Set up and release of the CTA's tensor-core state.  All threads call.
template <typename T>
__device__ __forceinline__ void wd_begin(WdCta<T> &w, unsigned char *smem_raw, uint64_t *bar, uint32_t *s_tmem,
                                         int *exA, int *exB, int *exP, int *s_ok, long long timeout_ns) {
  w.A = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  w.B = w.A + (size_t)SliceFmt<T>::kDig * kSlASlab;
  w.stage = w.B + 2 * kWdBBytes<T> + (threadIdx.x >> 5) * 32 * kWdStageRow<T>;
  w.bar = bar;
  w.exA = exA;
  w.exB = exB;
  w.exP = exP;
  w.s_ok = s_ok;
  w.ph = 0;
  w.timeout_ns = timeout_ns;
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 32) tmem_alloc(s_tmem, kWdTmem<T>);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  w.tmem = *s_tmem;
}
template <typename T>
__device__ __forceinline__ void wd_end(const WdCta<T> &w) {
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) tmem_dealloc(w.tmem, kWdTmem<T>);
}

#define WD_CTA_SETUP(T)                                                                                   \
  extern __shared__ __align__(16) unsigned char smem_raw[];                                               \
  __shared__ uint64_t s_bar;                                                                              \
  __shared__ uint32_t s_tmem;                                                                             \
  __shared__ int s_ok, s_go, s_exA[kSlRows], s_exB[kWdTile], s_exP[4 * kSlRows];                          \
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;                                        \
  __syncthreads();                                                                                        \
  if (!s_go) return;                                                                                      \
  WdCta<T> w;                                                                                             \
  wd_begin(w, smem_raw, &s_bar, &s_tmem, s_exA, s_exB, s_exP, &s_ok, a.timeout_ns);                       \
  /* this thread drains row `row` (slot row >> 6), 16 columns from 16 hw */                               \
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hw = warp >> 2, row0 = 32 * (warp & 3),     \
            row = row0 + lane;                                                                            \
  const uint32_t lane_base = w.tmem + ((uint32_t)row0 << 16);                                             \
  const uint32_t acc16 = lane_base + (uint32_t)(hw >> 1) * kWdBufCols<T> + (uint32_t)(16 * (hw & 1));

// Slot i of the rows below panel k of block j: block rows k + 1 .. of D, then
// W_L, W_R and the right-hand sides.
template <typename T>
__device__ __forceinline__ Slot<T> panel_slot(const Args<T> &a, const WidePanels &P, int l, long long j, int k, int i) {
  const int n = a.p.n;
  const size_t nn = (size_t)n * n;
  const long long orig = j << l;
  const int nD = P.nt - 1 - k, nW = l < a.p.L ? P.nt : 0;
  if (i < nD) {
    const int ib = k + 1 + i;
    return {a.Ld + (size_t)orig * nn + (size_t)ib * P.nb * n, n, 1, min(P.nb, n - ib * P.nb)};
  }
  i -= nD;
  if (i < 2 * nW) {
    const int side = i >= nW, q = i - side * nW;
    if (side && j + 1 >= a.p.Nl[l]) return no_slot<T>();
    return {a.Wb + (size_t)(a.p.off[l] + j - 1 + side) * nn + (size_t)q * P.nb * n, n, 1, min(P.nb, n - q * P.nb)};
  }
  if (i == 2 * nW && a.d > 0) return {a.Y + (size_t)orig * n * a.d, 1, a.d, a.d};
  return no_slot<T>();
}
// Slots of a panel: the D rows alone are the last panel's ones without couplings.
__host__ __device__ inline int panel_slots(const WidePanels &P, bool couplings, int k, int d) {
  return P.nt - 1 - k + (couplings ? 2 * P.nt : 0) + (d > 0 ? 1 : 0);
}

template <typename T>
__global__ void __launch_bounds__(kWdThreads, sizeof(T) == 8 ? 1 : 2)
    k_wide_panel(const __grid_constant__ Args<T> a, const WideBuf<T> wb, int l, int k) {
  WD_CTA_SETUP(T)
  const int n = a.p.n;
  const WidePanels P = panels_of(n);
  const bool top = l == a.p.L;
  const long long nE = top ? 1 : a.p.Nl[l] / 2;
  const int tiles = (panel_slots(P, !top, k, a.d) + 1) / 2;
  const bool pairs = (n & 1) == 0, segs = ((n * (int)sizeof(T)) & 15) == 0;
  const int kb = min(P.nb, n - k * P.nb);  // columns of this panel
  bool ok = true;
  for (long long t = blockIdx.x; t < nE * tiles && ok; t += gridDim.x) {
    const long long m = t / tiles, j = top ? 0 : 2 * m + 1;
    const int i0 = 2 * (int)(t - m * tiles);
    const Slot<T> s0 = panel_slot(a, P, l, j, k, i0), s1 = panel_slot(a, P, l, j, k, i0 + 1);
    if (s0.rows == 0 && s1.rows == 0) continue;
    const int nD = P.nt - 1 - k - i0;  // this tile's slots of D
    const T *Lk = a.Ld + ((size_t)(j << l) * n + (size_t)k * P.nb) * n;
    const Slot<T> mine = row < 64 ? s0 : s1;
    const int r = row & 63, wrows = mine.rows - (row0 & 63);  // rows of this warp
    T acc[16];
#pragma unroll 1
    for (int rd = 0; rd < k + (nD > 0 ? 3 : 1); ++rd) {
      const int c0 = rd < k ? rd * P.nb : k * P.nb;  // the chunk's first column
      if (rd <= k) {
        Slot<T> c_0 = s0, c_1 = s1;
        c_0.p += (long long)c0 * s0.cs;
        c_1.p += (long long)c0 * s1.cs;
        Slot<T> b = rd < k ? Slot<T>{const_cast<T *>(Lk) + c0, n, 1, kb}
                           : Slot<T>{wb.X + (size_t)m * kWdTile * kWdTile, kWdTile, 1, kWdTile};
        wd_cut<T>(w, c_0, c_1, b, rd < k || k == 0, true, rd < k ? P.nb : kb, pairs);
      }
      if ((rd == k && k > 0) || rd == k + 1) {
        if (rd == k) {  // S - sum of the products
          const T *src = mine.p + (long long)r * mine.rs + (long long)(k * P.nb + 16 * hw) * mine.cs;
#pragma unroll
          for (int i = 0; i < 16; ++i)
            acc[i] = (r < mine.rows && 16 * hw + i < kb) ? ldcg(src + i * mine.cs) - acc[i] : T(0);
        }
        wd_cut_regs<T>(w, acc, row, hw);
        if (rd == k + 1) __syncthreads();
      }
      if (rd > k) {
        // B tiles: rows 32 h .. 32 h + 31 of either slot
        const int h = rd - k - 1;
#pragma unroll 4
        for (int e = threadIdx.x; e < SliceFmt<T>::kDig * 64 * 8; e += kWdThreads) {
          const int p = e >> 9, rr = (e >> 3) & 63, g = e & 7;
          const int src = 64 * (rr >> 5) + 32 * h + (rr & 31);
          *reinterpret_cast<uint4 *>(w.B + (rr >> 5) * kWdBBytes<T> + p * kSlBSlab + (rr & 31) * 128 + g * 16) =
              *reinterpret_cast<const uint4 *>(w.A + p * kSlASlab + src * 128 + g * 16);
        }
      }
      const int ks = ((rd < k ? P.nb : kb) + 15) >> 4;
      // X is lower triangular: its first 32 rows have 32 columns
      if (!wd_product<T>(w, rd <= k ? kb > 32 : nD > 1, rd == k ? min(ks, 2) : ks, ks)) {
        if (threadIdx.x == 0) set_status(a.st, kStTimeout, l, -1);
        ok = false;
        break;
      }
      const int ea = w.exA[row];
      if (rd <= k) {
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
          if (16 * hw + c < kb && wrows > 0) {  // the same for a warp
            T v[4];
            wd_drain4<T>(acc16 + c, ea, w.exB + 16 * hw + c, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c + e] = rd > 0 && rd < k ? acc[c + e] + v[e] : v[e];
            if (rd == k) {
              const int col = k * P.nb + 16 * hw + c;
              if (mine.cs == 1) {
                wd_store4<T>(w.stage, v, mine.p + (long long)(row0 & 63) * mine.rs + col, mine.rs, wrows,
                             kb - 16 * hw - c, segs, false);
              } else if (r < mine.rows) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                  if (16 * hw + c + e < kb) mine.p[(long long)(col + e) * mine.cs + r * mine.rs] = v[e];
              }
            }
          } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c + e] = T(0);
          }
        }
      } else if ((row >> 6) < nD) {
        // columns 32 h .. of the diagonal tile of each slot of D, lower part
        const int h = rd - k - 1;
#pragma unroll
        for (int c = 0; c < 8; c += 4) {
          const int col = 32 * h + 8 * hw + c;
          if (col < mine.rows && wrows > 0 && col <= (r | 31)) {
            T v[4];
            wd_drain4<T>(lane_base + (uint32_t)(row >> 6) * kWdBufCols<T> + (uint32_t)(8 * hw + c), ea,
                         w.exA + (row & 64) + col, v);
            const int ib = k + 1 + i0 + (row >> 6);
            wd_store4<T>(w.stage, v, mine.p + (long long)(row0 & 63) * mine.rs + ib * P.nb + col, mine.rs, wrows,
                         mine.rows - col, segs, true);
          }
        }
      }
      // the exponents and slabs of the round have been read before the next one's
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
    }
  }
  wd_end(w);
}

// Tasks of one separator: D tiles (pairs of block rows by a block column, up
// to the diagonal), right-hand sides, next coupling's tiles.
__host__ __device__ inline int schur_tiles_d(int nt) {
  int c = 0;
  for (int t = 0; t < (nt + 1) / 2; ++t) c += min(2 * t + 2, nt);
  return c;
}
__host__ __device__ inline int schur_tiles(int nt, int d) {
  const int tr = (nt + 1) / 2;
  return schur_tiles_d(nt) + (d > 0 ? tr : 0) + tr * nt;
}

template <typename T>
__global__ void __launch_bounds__(kWdThreads, sizeof(T) == 8 ? 1 : 2)
    k_wide_schur(const __grid_constant__ Args<T> a, int l) {
  WD_CTA_SETUP(T)
  const int n = a.p.n, d = a.d;
  const size_t nn = (size_t)n * n;
  const WidePanels P = panels_of(n);
  const int nt = P.nt, nb = P.nb, tr = (nt + 1) / 2;
  const long long Nl = a.p.Nl[l], nS = (Nl + 1) / 2;
  const int tD = schur_tiles_d(nt), tR = d > 0 ? tr : 0, tiles = schur_tiles(nt, d);
  const bool pairs = (n & 1) == 0, segs = ((n * (int)sizeof(T)) & 15) == 0;
  const T *W = a.Wb + (size_t)a.p.off[l] * nn;
  bool ok = true;
  for (long long t = blockIdx.x; t < nS * tiles && ok; t += gridDim.x) {
    const long long q = t / tiles, s = 2 * q, orig = s << l;
    const bool hasM = s >= 2, hasP = s + 1 < Nl, hasE = s + 2 < Nl;
    int u = (int)(t - q * tiles), ti = 0, jb = 0;
    const bool isD = u < tD, isR = !isD && u < tD + tR, isE = !isD && !isR;
    if (isD) {
      while (u >= min(2 * ti + 2, nt)) {
        u -= min(2 * ti + 2, nt);
        ++ti;
      }
      jb = u;
    } else if (isR) {
      ti = u - tD;
    } else {
      u -= tD + tR;
      ti = u / nt;
      jb = u - ti * nt;
    }
    if ((isE && !hasE) || (!isE && !hasM && !hasP)) continue;
    // the next level's even couplings are left transposed: W_L^T W_R instead of W_R^T W_L
    const bool flip = (q & 1) == 0;
    const T *A0 = isE ? W + (size_t)(flip ? s : s + 1) * nn : W + (size_t)(s - 1) * nn;
    const T *A1 = W + (size_t)s * nn;  // not isE: the right neighbour
    const T *BE = W + (size_t)(flip ? s + 1 : s) * nn;
    const int ra = 2 * ti * nb, rows0 = min(nb, n - ra), rows1 = max(0, min(nb, n - ra - nb));
    const int bcols = isR ? d : min(nb, n - jb * nb);  // output columns
    const int first = (isE || hasM) ? 0 : nt, last = (isE || !hasP) ? nt : 2 * nt;
    const int r = row & 63, rows = row < 64 ? rows0 : rows1, wrows = rows - (row0 & 63);
    T acc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[i] = T(0);
#pragma unroll 1
    for (int rd = first; rd < last; ++rd) {
      const int second = rd >= nt, p = rd - second * nt, c0 = p * nb, kc = min(nb, n - c0);
      const T *As = (second ? A1 : A0) + (size_t)ra * n + c0;
      const Slot<T> s0{const_cast<T *>(As), n, 1, rows0}, s1{const_cast<T *>(As) + (size_t)nb * n, n, 1, rows1};
      Slot<T> b;
      if (isR) {
        const long long jn = second ? s + 1 : s - 1;
        b = {a.Y + ((size_t)(jn << l) * n + c0) * d, 1, d, d};
      } else {
        const T *Bs = isE ? BE : second ? A1 : A0;
        b = {const_cast<T *>(Bs) + (size_t)jb * nb * n + c0, n, 1, bcols};
      }
      wd_cut<T>(w, s0, s1, b, true, true, kc, pairs);
      const int ks = (kc + 15) >> 4;
      if (!wd_product<T>(w, bcols > 32, ks, ks)) {
        if (threadIdx.x == 0) set_status(a.st, kStTimeout, l, -1);
        ok = false;
        break;
      }
      const int ea = w.exA[row];
#pragma unroll
      for (int c = 0; c < 16; c += 4)
        if (16 * hw + c < bcols && wrows > 0) {
          T v[4];
          wd_drain4<T>(acc16 + c, ea, w.exB + 16 * hw + c, v);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[c + e] += v[e];
        }
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
    }
    if (!ok) break;
    if (isR) {
      if (r < rows) {
        T *y = a.Y + ((size_t)orig * n + ra + (row & 64 ? nb : 0) + r) * d + 16 * hw;
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if (16 * hw + i < d) y[i] = ldcg(y + i) - acc[i];
      }
      continue;
    }
    T *dst = isE ? a.Wb + ((size_t)a.p.off[l + 1] + (size_t)q) * nn : a.Ld + (size_t)orig * nn;
    const int rw = ra + (row & 64 ? nb : 0) + (row0 & 63);  // the warp's first row
#pragma unroll
    for (int c = 0; c < 16; c += 4) {
      const int col = jb * nb + 16 * hw + c;
      if (16 * hw + c >= bcols || wrows <= 0 || (isD && col > rw + 31)) continue;  // the same for a warp
      T v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = isE ? -acc[c + e] : acc[c + e];
      wd_store4<T>(w.stage, v, dst + (size_t)rw * n + col, n, wrows, bcols - 16 * hw - c, segs, isD);
    }
  }
  wd_end(w);
}

// Cholesky factor and inverse of the diagonal tiles of panel k.
constexpr int kDiagThreads = 256;
template <typename T>
__global__ void __launch_bounds__(kDiagThreads) k_wide_diag(const __grid_constant__ Args<T> a, const WideBuf<T> wb,
                                                           int l, int k) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flag, s_go;
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;
  __syncthreads();
  if (!s_go) return;
  const int n = a.p.n;
  const WidePanels P = panels_of(n);
  const int kb = min(P.nb, n - k * P.nb), ld = ldstride(kb);
  const long long m = blockIdx.x, orig = (l == a.p.L ? 0 : 2 * m + 1) << l;
  T *s = reinterpret_cast<T *>(smem_raw);
  T *Lg = a.Ld + (size_t)orig * n * n + ((size_t)k * P.nb) * n + k * P.nb;
  for (int e = threadIdx.x; e < kb * kb; e += blockDim.x) {
    const int i = e / kb, c = e - i * kb;
    if (c <= i) s[i * ld + c] = ldcg(Lg + (size_t)i * n + c);
  }
  __syncthreads();
  if (chol_fused(s, ld, kb, s, 0, s, 0, &s_flag)) {
    if (threadIdx.x == 0) set_status(a.st, kStNotSPD, l, orig);
    return;
  }
  tri_inverse_upper(s, ld, kb);
  T *Xg = wb.X + (size_t)m * kWdTile * kWdTile;
  for (int e = threadIdx.x; e < kWdTile * kWdTile; e += blockDim.x) {
    const int i = e / kWdTile, c = e - i * kWdTile;
    Xg[e] = (c <= i && i < kb) ? s[c * ld + i] : T(0);  // X[i][c] is in the upper triangle
  }
  for (int e = threadIdx.x; e < kb * kb; e += blockDim.x) {
    const int i = e / kb, c = e - i * kb;
    Lg[(size_t)i * n + c] = s[i * ld + c];
  }
}

// Level 0.  Tasks per block: the lower 32 x 32 tiles of sym(A_ii), the tiles
// of the coupling below it, its right-hand sides.
template <typename T>
__global__ void __launch_bounds__(256) k_wide_ingest(const __grid_constant__ Args<T> a) {
  __shared__ double t0[32][33], t1[32][33];
  const int n = a.p.n, d = a.d, nt = (n + 31) / 32, lower = nt * (nt + 1) / 2, per = lower + nt * nt + (d > 0);
  const size_t nn = (size_t)n * n;
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  for (long long t = blockIdx.x; t < a.p.N * per; t += gridDim.x) {
    const long long i = t / per;
    int u = (int)(t - i * per);
    if (u < lower) {
      int ti = 0;
      while ((ti + 1) * (ti + 2) / 2 <= u) ++ti;
      const int tj = u - ti * (ti + 1) / 2;
      const double *g = a.A_diag + (size_t)i * nn;
#pragma unroll
      for (int q = 0; q < 32; q += 8) {
        const int r = q + y;
        if (32 * ti + r < n && 32 * tj + x < n) t0[r][x] = __ldcg(g + (size_t)(32 * ti + r) * n + 32 * tj + x);
        if (32 * tj + r < n && 32 * ti + x < n) t1[r][x] = __ldcg(g + (size_t)(32 * tj + r) * n + 32 * ti + x);
      }
      __syncthreads();
      T *o = a.Ld + (size_t)i * nn;
#pragma unroll
      for (int q = 0; q < 32; q += 8) {
        const int r = q + y;
        if (32 * ti + r < n && 32 * tj + x < n)
          o[(size_t)(32 * ti + r) * n + 32 * tj + x] = T(0.5) * ((T)t0[r][x] + (T)t1[x][r]);
      }
      __syncthreads();
    } else if (u < lower + nt * nt) {
      if (i + 1 >= a.p.N) continue;
      u -= lower;
      const int ti = u / nt, tj = u - ti * nt;
      const double *g = a.A_sub + (size_t)i * nn;
      T *o = a.Wb + (size_t)i * nn;
      if (i & 1) {
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
          const int r = 32 * ti + q + y, c = 32 * tj + x;
          if (r < n && c < n) o[(size_t)r * n + c] = (T)__ldcg(g + (size_t)r * n + c);
        }
      } else {  // the left coupling of block i + 1
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
          const int r = 32 * ti + q + y, c = 32 * tj + x;
          if (r < n && c < n) t0[q + y][x] = __ldcg(g + (size_t)r * n + c);
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 32; q += 8) {
          const int r = 32 * tj + q + y, c = 32 * ti + x;
          if (r < n && c < n) o[(size_t)r * n + c] = (T)t0[x][q + y];
        }
        __syncthreads();
      }
    } else {
      const size_t o = (size_t)i * n * d;
      for (int e = threadIdx.x; e < n * d; e += blockDim.x)
        a.Y[o + e] = a.B64 ? (T)__ldcg(a.B64 + o + e) : ldcg(a.Bt + o + e);
    }
  }
}

// Downward pass (Algorithms 6, 2), first half: t_j = y_j - W_L x_{j-1} - W_R x_{j+1}
// for 64 rows of an eliminated block, (W x)[q] = sum_p Wt[p][q] x[p]: a thread
// per row and quarter of the sum, four columns of x at a time.
constexpr int kDownCols = 4;
template <typename T>
__global__ void __launch_bounds__(256) k_wide_down1(const __grid_constant__ Args<T> a, int l) {
  __shared__ T sX[2 * kMaxNLarge * kDownCols], sR[4][64][kDownCols];
  if (ld_relaxed_i32(&a.st->status) != 0) return;
  const int n = a.p.n, d = a.d, parts = (n + 63) / 64;
  const size_t nn = (size_t)n * n, nd = (size_t)n * d;
  const long long m = blockIdx.x / parts, j = 2 * m + 1;
  const int q0 = 64 * (int)(blockIdx.x - m * parts), qi = threadIdx.x & 63, g = threadIdx.x >> 6, q = q0 + qi;
  const bool hasR = j + 1 < a.p.Nl[l];
  const T *Wt = a.Wb + (size_t)(a.p.off[l] + j - 1) * nn;  // W_L^T rows, then W_R^T rows
  const int np = hasR ? 2 * n : n, p0 = g * np / 4, p1 = (g + 1) * np / 4;
  const T *xm = a.Y + (size_t)((j - 1) << l) * nd, *xp = a.Y + (size_t)((j + 1) << l) * nd;
  T *y = a.Y + (size_t)(j << l) * nd;
  for (int c0 = 0; c0 < d; c0 += kDownCols) {
    for (int e = threadIdx.x; e < np * kDownCols; e += 256) {
      const int p = e / kDownCols, c = c0 + e % kDownCols;
      sX[e] = c >= d ? T(0) : p < n ? ldcg(xm + (size_t)p * d + c) : ldcg(xp + (size_t)(p - n) * d + c);
    }
    __syncthreads();
    T acc[kDownCols] = {};
    if (q < n) {
#pragma unroll 8
      for (int p = p0; p < p1; ++p) {
        const T wv = ldcg(Wt + (size_t)p * n + q);
#pragma unroll
        for (int c = 0; c < kDownCols; ++c)
          if (c0 + c < d) acc[c] = fma(wv, sX[p * kDownCols + c], acc[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < kDownCols; ++c) sR[g][qi][c] = acc[c];
    __syncthreads();
    if (q < n && c0 + g < d) {
      const T v = (sR[0][qi][g] + sR[1][qi][g]) + (sR[2][qi][g] + sR[3][qi][g]);
      T *o = y + (size_t)q * d + c0 + g;
      *o = ldcg(o) - v;
    }
    __syncthreads();
  }
}

// Second half: x_j = L_j^{-T} t_j from the last panel up,
//   x_k = X_kk^T (t_k - sum_{p>k} L_pk^T x_p),
// eight groups of 64 threads, one per eighth of the rows p; X_kk^T is the
// upper triangle of the diagonal tile.  l == L: the top block.
template <typename T>
__global__ void __launch_bounds__(512) k_wide_down2(const __grid_constant__ Args<T> a, int l) {
  __shared__ T sV[kMaxNLarge * kDownCols], sR[8][64][kDownCols];
  if (ld_relaxed_i32(&a.st->status) != 0) return;
  const int n = a.p.n, d = a.d;
  const WidePanels P = panels_of(n);
  const size_t nd = (size_t)n * d;
  const long long m = blockIdx.x, orig = (l == a.p.L ? 0 : 2 * m + 1) << l;
  const T *Lg = a.Ld + (size_t)orig * n * n;
  T *y = a.Y + (size_t)orig * nd;
  const int i = threadIdx.x & 63, g = threadIdx.x >> 6;
  for (int c0 = 0; c0 < d; c0 += kDownCols) {
    for (int e = threadIdx.x; e < n * kDownCols; e += 512) {
      const int p = e / kDownCols, c = c0 + e % kDownCols;
      sV[e] = c < d ? ldcg(y + (size_t)p * d + c) : T(0);
    }
    __syncthreads();
    for (int k = P.nt - 1; k >= 0; --k) {
      const int k0 = k * P.nb, kb = min(P.nb, n - k0), below = n - k0 - kb;
      for (int half = 0; half < 2; ++half) {
        // half 0: the rows below the panel; half 1: the triangle of the tile
        if (half == 0 && below == 0) continue;
        T acc[kDownCols] = {};
        if (i < kb) {
          if (half == 0) {
            const int p1 = k0 + kb + (g + 1) * below / 8;
#pragma unroll 8
            for (int p = k0 + kb + g * below / 8; p < p1; ++p) {
              const T lv = ldcg(Lg + (size_t)p * n + k0 + i);
#pragma unroll
              for (int c = 0; c < kDownCols; ++c)
                if (c0 + c < d) acc[c] = fma(lv, sV[p * kDownCols + c], acc[c]);
            }
          } else {
            const T *xr = Lg + (size_t)(k0 + i) * n + k0;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int p = 8 * u + g;
              if (p >= i && p < kb) {
                const T xv = ldcg(xr + p);
#pragma unroll
                for (int c = 0; c < kDownCols; ++c)
                  if (c0 + c < d) acc[c] = fma(xv, sV[(k0 + p) * kDownCols + c], acc[c]);
              }
            }
          }
        }
#pragma unroll
        for (int c = 0; c < kDownCols; ++c) sR[g][i][c] = acc[c];
        __syncthreads();
        if (g < kDownCols && i < kb && c0 + g < d) {
          T v = sR[0][i][g];
#pragma unroll
          for (int u = 1; u < 8; ++u) v += sR[u][i][g];
          T *o = sV + (k0 + i) * kDownCols + g;
          *o = half == 0 ? *o - v : v;
        }
        __syncthreads();
      }
    }
    for (int e = threadIdx.x; e < n * kDownCols; e += 512) {
      const int p = e / kDownCols, c = c0 + e % kDownCols;
      if (c < d) y[(size_t)p * d + c] = sV[e];
    }
    __syncthreads();
  }
}

}  // namespace

WidePanels wide_panels(int n) { return panels_of(n); }

template <typename T>
size_t wide_x_bytes(long long N) {
  return (size_t)(N / 2 > 1 ? N / 2 : 1) * kWdTile * kWdTile * sizeof(T);
}

template <typename T>
cudaError_t wide_configure() {
  cudaError_t e = cudaFuncSetAttribute((const void *)k_wide_panel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)wd_smem<T>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute((const void *)k_wide_schur<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)wd_smem<T>());
  return e;
}

static unsigned wd_grid(long long tasks, long long most) { return (unsigned)(tasks < most ? tasks : most); }

template <typename T>
cudaError_t launch_wide_ingest(const Args<T> &a, int sms, cudaStream_t s) {
  k_wide_ingest<T><<<wd_grid(a.p.N * 16, 8LL * sms), 256, 0, s>>>(a);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_diag(const Args<T> &a, const WideBuf<T> &w, int l, int k, cudaStream_t s) {
  const long long nE = l == a.p.L ? 1 : a.p.Nl[l] / 2;
  const size_t smem = (size_t)kWdTile * ldstride(kWdTile) * sizeof(T);
  k_wide_diag<T><<<(unsigned)nE, kDiagThreads, smem, s>>>(a, w, l, k);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_panel(const Args<T> &a, const WideBuf<T> &w, int l, int k, int sms, cudaStream_t s) {
  const WidePanels P = panels_of(a.p.n);
  const bool top = l == a.p.L;
  const long long tasks = (top ? 1 : a.p.Nl[l] / 2) * ((panel_slots(P, !top, k, a.d) + 1) / 2);
  if (tasks == 0) return cudaSuccess;  // the last panel of the top block without right-hand sides
  k_wide_panel<T><<<wd_grid(tasks, sizeof(T) == 8 ? sms : 2 * sms), kWdThreads, wd_smem<T>(), s>>>(a, w, l, k);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_schur(const Args<T> &a, int l, int sms, cudaStream_t s) {
  const long long tasks = (a.p.Nl[l] + 1) / 2 * schur_tiles(panels_of(a.p.n).nt, a.d);
  k_wide_schur<T><<<wd_grid(tasks, sizeof(T) == 8 ? sms : 2 * sms), kWdThreads, wd_smem<T>(), s>>>(a, l);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_down(const Args<T> &a, int l, cudaStream_t s) {
  const long long nE = l == a.p.L ? 1 : a.p.Nl[l] / 2;
  if (l < a.p.L) k_wide_down1<T><<<(unsigned)(nE * ((a.p.n + 63) / 64)), 256, 0, s>>>(a, l);
  k_wide_down2<T><<<(unsigned)nE, 512, 0, s>>>(a, l);
  return cudaGetLastError();
}

#define BDSS_WIDE_INSTANTIATE(T)                                                                                   \
  template size_t wide_x_bytes<T>(long long);                                                                     \
  template cudaError_t wide_configure<T>();                                                                       \
  template cudaError_t launch_wide_ingest<T>(const Args<T> &, int, cudaStream_t);                                 \
  template cudaError_t launch_wide_diag<T>(const Args<T> &, const WideBuf<T> &, int, int, cudaStream_t);          \
  template cudaError_t launch_wide_panel<T>(const Args<T> &, const WideBuf<T> &, int, int, int, cudaStream_t);    \
  template cudaError_t launch_wide_schur<T>(const Args<T> &, int, int, cudaStream_t);                             \
  template cudaError_t launch_wide_down<T>(const Args<T> &, int, cudaStream_t);
BDSS_WIDE_INSTANTIATE(double)

}  // namespace bdss
