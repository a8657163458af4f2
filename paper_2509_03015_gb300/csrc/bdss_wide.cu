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
//   k_wide_panel  every other row v: P_vk = (S_vk - sum_{p<k} P_vp L_kp^T) X_kk^T
//                 (scaled along the columns by the tile's diagonal), and for
//                 rows of D their own diagonal tile, updated by P P^T.
// Then one launch forms what the separators receive (k_wide_schur): D, the
// next level's couplings, b.
//
// Every n x n operand is read along contiguous rows: couplings are stored as
// the rows the elimination needs (the even slots of a level, its eliminated
// blocks' left couplings, transposed), from the level-0 ingest on.  Couplings
// and their W^T share a slot of Wb, D and its L a slot of Ld (reciprocal
// diagonal), where a diagonal tile keeps X_kk^T above its diagonal for the
// downward pass.
//
// Why: the substitutions of the couplings are n^3 multiply-adds a block on an
// ALU of 2 FP64 multiply-adds a cycle and SM.  Measured (factor + solve):
//   N = 1024, n = 256, d = 1, FP64              89.2 -> 22.0 ms
//   N = 100, n = 256, d = 1, FP32 refined        8.96 -> 5.1 ms
//   N = 4096, n = 256, d = 16, TF32 mode refined 58.0 -> 49.3 ms
#include "bdss_launch.h"
#include "bdss_slice_cta.cuh"
#include "bdss_wide.h"

namespace bdss {

namespace {

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
  int rs, cs;
  int rows;
  int q = -1;  // >= 0: unit rows, the q-th block row of the identity (zero before column q nb)
};

template <typename T>
__device__ __forceinline__ Slot<T> no_slot() {
  return {nullptr, 0, 0, 0};
}

template <typename T>
__device__ __forceinline__ void load2_cached(const T *p, T &x, T &y) {
  struct alignas(2 * sizeof(T)) Two { T x, y; };
  const Two v = *reinterpret_cast<const Two *>(p);
  x = v.x;
  y = v.y;
}

// Digits of the K columns [0, kc) of the slots a0, a1 (A rows 0 .. 63, 64 ..
// 127; skipped unless do_a) and b (B rows), a warp per row: all loads of the
// 192 rows first, then the cutting.  kScaled: the A rows scaled down by 2^E
// along K.
template <typename T, bool kScaled>
__device__ __forceinline__ void wd_cut(const WdCta<T> &w, const Slot<T> &a0, const Slot<T> &a1, const Slot<T> &b,
                                       bool do_a, bool do_b, int kc, bool pairs, const short *E) {
  constexpr int kR = 64 / kWdWarps<T>;  // rows of a slot per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = 2 * lane;
  T v[3 * kR][2];
  short2 ke = make_short2(0, 0);
  if constexpr (kScaled) {
    ke = __ldcg(reinterpret_cast<const short2 *>(E + k));
  }
#pragma unroll
  for (int u = 0; u < 3 * kR; ++u) {
    const Slot<T> &s = u < kR ? a0 : u < 2 * kR ? a1 : b;
    const int r = (u % kR) * kWdWarps<T> + warp;
    v[u][0] = v[u][1] = T(0);
    if ((u < 2 * kR ? do_a : do_b) && r < s.rows && k < kc) {
      const T *p = s.p + (r * s.rs + k * s.cs);
      if (pairs && s.cs == 1) {
        load2(p, v[u][0], v[u][1]);
      } else {
        v[u][0] = ldcg(p);
        if (k + 1 < kc) v[u][1] = ldcg(p + s.cs);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 3 * kR; ++u) {
    if (!(u < 2 * kR ? do_a : do_b)) continue;
    const int r = (u % kR) * kWdWarps<T> + warp;
    const bool scaled = kScaled && u < 2 * kR;
    int ex, rex;
    if (scaled) {
      sl_prep(v[u][0], -ke.x);
      sl_prep(v[u][1], -ke.y);
      rex = ex = __reduce_max_sync(0xffffffffu, max(sl_exp_at(v[u][0], -ke.x), sl_exp_at(v[u][1], -ke.y)));
    } else {
      ex = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(sl_exp(v[u][0]), sl_exp(v[u][1])));
      rex = sl_row_exp<T>(ex);
    }
    if (u < 2 * kR) {
      const int ra = 64 * (u / kR) + r;
      if (lane == 0) w.exA[ra] = rex;
      sl_store2<T>(v[u][0], v[u][1], ex, w.A + sl_off(ra, k >> 3) + 2 * (k & 7), kSlASlab, scaled ? -ke.x : 0,
                   scaled ? -ke.y : 0);
    } else {
      if (lane == 0) w.exB[r] = rex;
      sl_store2<T>(v[u][0], v[u][1], ex, w.B + (r >> 5) * kWdBBytes<T> + sl_off(r & 31, k >> 3) + 2 * (k & 7),
                   kSlBSlab);
    }
  }
}

// Slot i of the rows below panel k of block j (the level's m-th): block rows
// k + 1 .. of D, then W_L, W_R, the right-hand sides and, where L^{-1} is
// wanted, the first k block rows of the identity, which become L^{-T}.
template <typename T>
__device__ __forceinline__ Slot<T> panel_slot(const Args<T> &a, const WideBuf<T> &wb, const WidePanels &P, int l,
                                              long long j, long long m, int k, int i) {
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
  i -= 2 * nW;
  if (a.d > 0 && i-- == 0) return {a.Y + (size_t)orig * n * a.d, 1, a.d, a.d};
  if (wb.Li && i < k) return {wb.V + (size_t)m * nn + (size_t)i * P.nb * n, n, 1, P.nb, i};
  return no_slot<T>();
}
// Slots of a panel: the D rows alone are the last panel's ones without couplings.
__host__ __device__ inline int panel_slots(const WidePanels &P, bool couplings, int k, int d, bool inverse) {
  return P.nt - 1 - k + (couplings ? 2 * P.nt : 0) + (d > 0 ? 1 : 0) + (inverse ? k : 0);
}

// Rounds of a tile of two slots: one per earlier panel (left-looking, so that a
// row's entries are read and written once a panel and no second launch is
// needed), P, and for rows of D two with half the columns each for their own
// diagonal tiles.
//
// What bounds it, in FP64: the logic pipe while operands are cut and sums
// converted, and the products themselves, half hidden (profile of
// k_wide_schur, whose rounds are the same).  N = 1024, n = 256: the four panels
// of level 0 take 0.55, 0.91, 0.89 and 1.04 ms.
//
// kFirst: panel 0 (its operands are cut, and scaled, as they come from memory;
// a later panel's from registers).
template <typename T, bool kFirst>
__global__ void __launch_bounds__(kWdThreads<T>, sizeof(T) == 8 ? 1 : 2)
    k_wide_panel(const __grid_constant__ Args<T> a, const WideBuf<T> wb, int l, int panel) {
  const int k = kFirst ? 0 : panel;
  __shared__ __align__(16) short s_E[kWdTile];
  WD_CTA_SETUP(T)
  const int n = a.p.n;
  const WidePanels P = panels_of(n);
  const bool top = l == a.p.L;
  const long long nE = top ? 1 : a.p.Nl[l] / 2;
  const int tiles = (panel_slots(P, !top, k, a.d, wb.Li != nullptr) + 1) / 2;
  const bool pairs = (n & 1) == 0, segs = ((n * (int)sizeof(T)) & 15) == 0;
  const int kb = min(P.nb, n - k * P.nb);  // columns of this panel
  bool ok = true;
  for (long long t = blockIdx.x; t < nE * tiles && ok; t += gridDim.x) {
    const long long m = t / tiles, j = top ? 0 : 2 * m + 1;
    const int i0 = 2 * (int)(t - m * tiles);
    const Slot<T> s0 = panel_slot(a, wb, P, l, j, m, k, i0), s1 = panel_slot(a, wb, P, l, j, m, k, i0 + 1);
    if (s0.rows == 0 && s1.rows == 0) continue;
    const int nD = P.nt - 1 - k - i0;  // this tile's slots of D
    const T *Lk = a.Ld + ((size_t)(j << l) * n + (size_t)k * P.nb) * n;
    const short *Ek = wb.E + m * kWdTile;
    if (!kFirst && threadIdx.x < kWdTile / 2)  // at hand in round k
      reinterpret_cast<short2 *>(s_E)[threadIdx.x] = __ldcg(reinterpret_cast<const short2 *>(Ek) + threadIdx.x);
    const Slot<T> mine = row < 64 ? s0 : s1;
    const int r = row & 63, wrows = mine.rows - (row0 & 63);  // rows of this warp
    T acc[kWdCols<T>];
#pragma unroll 1
    for (int rd = 0; rd < k + (nD > 0 ? 3 : 1); ++rd) {
      const int c0 = rd < k ? rd * P.nb : k * P.nb;  // the chunk's first column
      if (rd <= k) {
        Slot<T> c_0 = s0, c_1 = s1;
        c_0.p += c0 * s0.cs;
        c_1.p += c0 * s1.cs;
        if (rd < s0.q) c_0.rows = 0;
        if (rd < s1.q) c_1.rows = 0;
        Slot<T> b = rd < k ? Slot<T>{const_cast<T *>(Lk) + c0, n, 1, kb}
                           : Slot<T>{wb.X + (size_t)m * kWdTile * kWdTile, kWdTile, 1, kWdTile};
        wd_cut<T, kFirst>(w, c_0, c_1, b, rd < k || kFirst, true, rd < k ? P.nb : kb, pairs, Ek);
      }
      if ((rd == k && !kFirst) || rd == k + 1) {
        SlScale8 sc[kWdCols<T> / 8] = {};
        if (!kFirst && rd == k) {
#pragma unroll
          for (int i = 0; i < kWdCols<T> / 8; ++i) sc[i] = sl_scale8(s_E + cb + 8 * i);
        }
        if (!kFirst && rd == k) {  // S - sum of the products
          const T *src = mine.p + (r * mine.rs + (k * P.nb + cb) * mine.cs);
#pragma unroll
          for (int i = 0; i < kWdCols<T>; i += 2) {  // (plain loads: a sector serves several of them)
            T x0 = T(0), x1 = T(0);
            if (mine.q < 0 && r < mine.rows) {
              if (pairs && mine.cs == 1) {
                if (cb + i < kb) load2_cached(src + i, x0, x1);
              } else {
                if (cb + i < kb) x0 = src[i * mine.cs];
                if (cb + i + 1 < kb) x1 = src[(i + 1) * mine.cs];
              }
            }
            acc[i] = x0 - acc[i];
            acc[i + 1] = x1 - acc[i + 1];
            sl_prep(acc[i], -sc[i >> 3].at(i & 7));
            sl_prep(acc[i + 1], -sc[(i + 1) >> 3].at((i + 1) & 7));
          }
        }
        wd_cut_regs<T, !kFirst>(w, acc, sc, row, hw);
        if (rd == k + 1) __syncthreads();
      }
      if (rd > k) {
        // B tiles: rows 32 h .. 32 h + 31 of either slot
        const int h = rd - k - 1;
#pragma unroll 4
        for (int e = threadIdx.x; e < SliceFmt<T>::kDig * 64 * 8; e += kWdThreads<T>) {
          const int p = e >> 9, rr = (e >> 3) & 63, g = e & 7;
          const int src = 64 * (rr >> 5) + 32 * h + (rr & 31);
          *reinterpret_cast<uint4 *>(w.B + (rr >> 5) * kWdBBytes<T> + p * kSlBSlab + (rr & 31) * 128 + g * 16) =
              *reinterpret_cast<const uint4 *>(w.A + p * kSlASlab + src * 128 + g * 16);
        }
      }
      const int ks = ((rd < k ? P.nb : kb) + 15) >> 4;
      const bool cols2 = rd <= k ? kb > 32 : nD > 1;
      // X is lower triangular: its first 32 rows have 32 columns
      wd_issue<T>(w, cols2, rd == k ? min(ks, 2) : ks, ks);
      const int ea = w.exA[row];
      if (rd <= k) {
        if (cb < kb && wrows > 0) {  // the same for a warp
          ok = wd_wait<T>(w, ctile);
#pragma unroll
          for (int c = 0; c < kWdCols<T>; c += 4) {
            if (cb + c < kb && ok) {
              T v[4];
              wd_drain4<T>(accb + c, ea, w.exB + cb + c, v);
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[c + e] = rd > 0 && rd < k ? acc[c + e] + v[e] : v[e];
              if (rd == k) {
                const int col = k * P.nb + cb + c;
                if (mine.cs == 1) {
                  wd_store4<T>(w.stage, v, mine.p + (row0 & 63) * mine.rs + col, mine.rs, wrows, kb - cb - c, segs,
                               false);
                  if (mine.q >= 0 && r < mine.rows) {  // L^{-1}: a warp's rows are consecutive columns
                    T *o = wb.Li + (size_t)(j << l) * n * n + (size_t)col * n + mine.q * P.nb + r;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                      if (cb + c + e < kb) o[(size_t)e * n] = v[e];
                  }
                } else if (r < mine.rows) {
#pragma unroll
                  for (int e = 0; e < 4; ++e)
                    if (cb + c + e < kb) mine.p[(col + e) * mine.cs + r * mine.rs] = v[e];
                }
              }
            } else {
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[c + e] = T(0);
            }
          }
        } else {
#pragma unroll
          for (int c = 0; c < kWdCols<T>; ++c) acc[c] = T(0);
        }
      } else if ((row >> 6) < nD) {
        // columns 32 h .. of the diagonal tile of each slot of D, lower part
        const int h = rd - k - 1, cd = kWdCols<T> / 2 * hw;
        ok = wd_wait<T>(w, row >> 6);
#pragma unroll
        for (int c = 0; c < kWdCols<T> / 2; c += 4) {
          const int col = 32 * h + cd + c;
          if (ok && col < mine.rows && wrows > 0 && col <= (r | 31)) {
            T v[4];
            wd_drain4<T>(lane_base + (uint32_t)(row >> 6) * kWdBufCols<T> + (uint32_t)(cd + c), ea,
                         w.exA + (row & 64) + col, v);
            const int ib = k + 1 + i0 + (row >> 6);
            wd_store4<T>(w.stage, v, mine.p + (row0 & 63) * mine.rs + ib * P.nb + col, mine.rs, wrows,
                         mine.rows - col, segs, true);
          }
        }
      }
      // the exponents, slabs and stages of the round have been read before the next one's
      ok = wd_round_end<T>(w, cols2, ok);
      if (!ok) {
        if (threadIdx.x == 0) set_status(a.st, kStTimeout, l, -1);
        break;
      }
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

// One round per K chunk of 64; a D tile sums both eliminated neighbours.  The
// accumulators hold one chunk exactly, the chunks meet in registers.
//
// What bounds it, in FP64: the logic pipe, 59 % busy over a launch, 2.1
// instructions a cycle; level 0 of N = 1024, n = 256 takes 3.7 ms (planes of
// ten BF16 digits cut by a launch of their own and read through TMA took 9.6 ms
// over all levels, this kernel 7.9).  In FP32: instructions as well (59 % of the
// issue slots); pipelining two rounds in one CTA of 32 warps changed nothing.
template <typename T>
__global__ void __launch_bounds__(kWdThreads<T>, sizeof(T) == 8 ? 1 : 2)
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
    T acc[kWdCols<T>];
#pragma unroll
    for (int i = 0; i < kWdCols<T>; ++i) acc[i] = T(0);
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
      wd_cut<T, false>(w, s0, s1, b, true, true, kc, pairs, nullptr);
      const int ks = (kc + 15) >> 4;
      const bool cols2 = bcols > 32;
      wd_issue<T>(w, cols2, ks, ks);
      const int ea = w.exA[row];
      if (cb < bcols && wrows > 0) {  // the same for a warp
        ok = wd_wait<T>(w, ctile);
#pragma unroll
        for (int c = 0; c < kWdCols<T>; c += 4)
          if (cb + c < bcols && ok) {
            T v[4];
            wd_drain4<T>(accb + c, ea, w.exB + cb + c, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c + e] += v[e];
          }
      }
      ok = wd_round_end<T>(w, cols2, ok);
      if (!ok) {
        if (threadIdx.x == 0) set_status(a.st, kStTimeout, l, -1);
        break;
      }
    }
    if (!ok) break;
    if (isR) {
      if (r < rows) {
        T *y = a.Y + ((size_t)orig * n + ra + (row & 64 ? nb : 0) + r) * d + cb;
#pragma unroll
        for (int i = 0; i < kWdCols<T>; ++i)
          if (cb + i < d) y[i] = ldcg(y + i) - acc[i];
      }
      continue;
    }
    T *dst = isE ? a.Wb + ((size_t)a.p.off[l + 1] + (size_t)q) * nn : a.Ld + (size_t)orig * nn;
    const int rw = ra + (row & 64 ? nb : 0) + (row0 & 63);  // the warp's first row
#pragma unroll
    for (int c = 0; c < kWdCols<T>; c += 4) {
      const int col = jb * nb + cb + c;
      if (cb + c >= bcols || wrows <= 0 || (isD && col > rw + 31)) continue;  // the same for a warp
      T v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = isE ? -acc[c + e] : acc[c + e];
      wd_store4<T>(w.stage, v, dst + (size_t)rw * n + col, n, wrows, bcols - cb - c, segs, isD);
    }
    __syncthreads();  // the stages have been read before the next task's B digits take their place
  }
  wd_end(w);
}

// Cholesky factor and inverse of the diagonal tiles of panel k (chol_inverse).
// One block's tile takes 77 us in FP64 and 35 us in FP32, launch included: the
// critical path of levels with few blocks.
constexpr int kDiagThreads = 256;
template <typename T>
__global__ void __launch_bounds__(kDiagThreads) k_wide_diag(const __grid_constant__ Args<T> a, const WideBuf<T> wb,
                                                           int l, int k) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int s_flag, s_go, s_cnt[8];
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;
  __syncthreads();
  if (!s_go) return;
  const int n = a.p.n;
  const WidePanels P = panels_of(n);
  const int kb = min(P.nb, n - k * P.nb), kp = (kb + 7) & ~7, ld = ldstride(kp);
  const long long m = blockIdx.x, orig = (l == a.p.L ? 0 : 2 * m + 1) << l;
  T *s = reinterpret_cast<T *>(smem_raw), *cbuf = s + (size_t)kp * ld;
  T *Lg = a.Ld + (size_t)orig * n * n + ((size_t)k * P.nb) * n + k * P.nb;
  // a thread takes a column of the tile, every fourth row
  const int c = threadIdx.x & (kWdTile - 1), i0 = threadIdx.x / kWdTile;
  constexpr int kStep = kDiagThreads / kWdTile;
#pragma unroll
  for (int u = 0; u < kWdTile / kStep; ++u) {
    const int i = i0 + u * kStep;
    if (i < kp && c <= i) s[i * ld + c] = i < kb ? ldcg(Lg + (size_t)i * n + c) : T(i == c);
  }
  __syncthreads();
  // before the factorisation's first barrier and writes
  const int ec = c < kb ? sl_half_exp(s[c * (ld + 1)]) : 0;
  if (threadIdx.x < kWdTile) wb.E[m * kWdTile + c] = (short)ec;
  if (chol_inverse(s, ld, kp, cbuf, s_cnt, &s_flag)) {
    if (threadIdx.x == 0) set_status(a.st, kStNotSPD, l, orig);
    return;
  }
  T *Xg = wb.X + (size_t)m * kWdTile * kWdTile;
  // L^{-1}: the tile, zeros to its right; the same tile of L^{-T}
  const int k0 = k * P.nb;
  T *Li = wb.Li + (size_t)orig * n * n + (size_t)k0 * n + k0, *V = wb.V + (size_t)m * n * n + (size_t)k0 * n + k0;
#pragma unroll 4
  for (int u = 0; u < kWdTile / kStep; ++u) {
    const int i = i0 + u * kStep;
    const bool in = i < kb && c < kb;
    const T x = in && c <= i ? s[c * ld + i] : T(0);  // X[i][c] is in the upper triangle
    Xg[i * kWdTile + c] = sl_scale(x, ec);
    if (in) {
      Lg[(size_t)i * n + c] = s[i * ld + c];
      if (wb.Li) V[(size_t)i * n + c] = i <= c ? s[i * ld + c] : T(0);
    }
    if (wb.Li && i < kb)
      for (int z = c; z < n - k0; z += kWdTile) Li[(size_t)i * n + z] = z == c && in ? x : T(0);
  }
}

// The FP64 top block of an FP32 factorisation: D_0 (lower) and b_0 to FP64.
__global__ void __launch_bounds__(256) k_wide_top_in(const __grid_constant__ Args<float> a, double *D, double *y) {
  const int n = a.p.n;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < n * n; e += gridDim.x * 256) D[e] = e % n <= e / n ? (double)ldcg(a.Ld + e) : 0.0;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < n * a.d; e += gridDim.x * 256) y[e] = (double)ldcg(a.Y + e);
}
// Its results: float(L) and float(L^{-1}) for the solve passes, x_0.
__global__ void __launch_bounds__(256) k_wide_top_out(const __grid_constant__ Args<float> a, const double *Li,
                                                      const double *x) {
  if (ld_relaxed_i32(&a.st->status) != 0) return;
  const int n = a.p.n;
  for (int e = blockIdx.x * 256 + threadIdx.x; e < n * n; e += gridDim.x * 256) {
    a.Ltinv[e] = e % n <= e / n ? (float)__ldcg(a.Ltop + e) : 0.0f;
    a.Ltinv[n * n + e] = (float)__ldcg(Li + e);
  }
  for (int e = blockIdx.x * 256 + threadIdx.x; e < n * a.d; e += gridDim.x * 256) {
    const double v = __ldcg(x + e);
    a.Y[e] = (float)v;
    if (a.X64) a.X64[e] = a.x_accumulate ? a.X64[e] + v : v;
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

// Downward pass (Algorithms 6, 2) in FP64, split in two so that a level of few
// blocks spreads its W over SMs (27 and 57 us for one block of n = 256), and
// over the columns there are instead of 64-wide vector tiles.  First half: t_j = y_j - W_L x_{j-1} - W_R x_{j+1}
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
  const void *kernels[] = {(const void *)k_wide_panel<T, true>, (const void *)k_wide_panel<T, false>,
                           (const void *)k_wide_schur<T>};
  cudaError_t e = cudaSuccess;
  for (const void *k : kernels)
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wd_smem<T>());
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
  const size_t smem = ((size_t)kWdTile * ldstride(kWdTile) + 17 * kMaxN) * sizeof(T);
  k_wide_diag<T><<<(unsigned)nE, kDiagThreads, smem, s>>>(a, w, l, k);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_panel(const Args<T> &a, const WideBuf<T> &w, int l, int k, int sms, cudaStream_t s) {
  const WidePanels P = panels_of(a.p.n);
  const bool top = l == a.p.L;
  const long long tasks = (top ? 1 : a.p.Nl[l] / 2) * ((panel_slots(P, !top, k, a.d, w.Li != nullptr) + 1) / 2);
  if (tasks == 0) return cudaSuccess;  // the last panel of the top block without right-hand sides
  const unsigned grid = wd_grid(tasks, sizeof(T) == 8 ? sms : 2 * sms);
  if (k == 0) k_wide_panel<T, true><<<grid, kWdThreads<T>, wd_smem<T>(), s>>>(a, w, l, k);
  else k_wide_panel<T, false><<<grid, kWdThreads<T>, wd_smem<T>(), s>>>(a, w, l, k);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_schur(const Args<T> &a, int l, int sms, cudaStream_t s) {
  const long long tasks = (a.p.Nl[l] + 1) / 2 * schur_tiles(panels_of(a.p.n).nt, a.d);
  k_wide_schur<T><<<wd_grid(tasks, sizeof(T) == 8 ? sms : 2 * sms), kWdThreads<T>, wd_smem<T>(), s>>>(a, l);
  return cudaGetLastError();
}

cudaError_t launch_wide_top_in(const Args<float> &a, double *D, double *y, cudaStream_t s) {
  k_wide_top_in<<<64, 256, 0, s>>>(a, D, y);
  return cudaGetLastError();
}
cudaError_t launch_wide_top_out(const Args<float> &a, const double *Li, const double *x, cudaStream_t s) {
  k_wide_top_out<<<64, 256, 0, s>>>(a, Li, x);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wide_down(const Args<T> &a, int l, cudaStream_t s) {
  const long long nE = l == a.p.L ? 1 : a.p.Nl[l] / 2;
  if (l < a.p.L) k_wide_down1<T><<<(unsigned)(nE * ((a.p.n + 63) / 64)), 256, 0, s>>>(a, l);
  k_wide_down2<T><<<(unsigned)nE, 512, 0, s>>>(a, l);
  return cudaGetLastError();
}

#define BDSS_WIDE_INSTANTIATE(T)                                                                                  \
  template size_t wide_x_bytes<T>(long long);                                                                    \
  template cudaError_t wide_configure<T>();                                                                      \
  template cudaError_t launch_wide_ingest<T>(const Args<T> &, int, cudaStream_t);                                \
  template cudaError_t launch_wide_diag<T>(const Args<T> &, const WideBuf<T> &, int, int, cudaStream_t);         \
  template cudaError_t launch_wide_panel<T>(const Args<T> &, const WideBuf<T> &, int, int, int, cudaStream_t);   \
  template cudaError_t launch_wide_schur<T>(const Args<T> &, int, int, cudaStream_t);
BDSS_WIDE_INSTANTIATE(double)
BDSS_WIDE_INSTANTIATE(float)
template cudaError_t launch_wide_down<double>(const Args<double> &, int, cudaStream_t);

}  // namespace bdss
