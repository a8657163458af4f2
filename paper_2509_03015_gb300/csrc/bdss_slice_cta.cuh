// One CTA's share of the digit products (bdss_slice.cuh): 128 A rows by 64 B
// rows by a K chunk of 64, cut by 16 warps into shared memory, multiplied by
// one thread's tcgen05.mma and drained by the same warps.
#pragma once
#include "bdss_slice.cuh"

namespace bdss {

// FP64: one CTA of 32 warps per SM (its digit slabs fill the shared memory);
// FP32: two of 16.
template <typename T> constexpr int kWdThreads = sizeof(T) == 8 ? 1024 : 512;
template <typename T> constexpr int kWdWarps = kWdThreads<T> / 32;
template <typename T> constexpr int kWdCols = 8192 / kWdThreads<T>;  // columns of an output row per thread
constexpr int kWdTile = 64;  // rows of a slot, columns of an output tile
template <typename T> constexpr uint32_t kWdBufCols = SliceFmt<T>::kDig * kSlCols;  // accumulators of 32 columns
template <typename T> constexpr uint32_t kWdTmem = sizeof(T) == 8 ? 512 : 256;  // a power of two
template <typename T> constexpr int kWdBBytes = SliceFmt<T>::kDig * kSlBSlab;
constexpr int kWdStage = 32 * 4;  // entries of a warp's output stage: 32 rows of four
template <typename T> constexpr size_t wd_smem() {
  return (size_t)SliceFmt<T>::kDig * (kSlASlab + 2 * kSlBSlab) + 1024;
}

template <typename T>
struct WdCta {
  // digit slabs; this warp's output stage, in the first B tile's place, whose
  // products are complete whenever there is something to put out
  unsigned char *A, *B, *stage;
  uint32_t tmem;
  uint64_t *bar;               // one per column tile
  int *exA, *exB, *exP;        // row exponents: A (128), B (64), partial (64 / kWdCols x 128)
  uint32_t ph0, ph1;
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

// Eight consecutive K entries of one row -> 16 bytes of every digit slab.
// kSign = 1 or -1: entry i counts as v[i] 2^(kSign e_i) (FP32: scaled already).
struct SlScale8 {  // the exponents e of eight K indices
  unsigned w[4];
  __device__ __forceinline__ int at(int i) const { return (int)(short)(w[i >> 1] >> (16 * (i & 1))); }
};
__device__ __forceinline__ SlScale8 sl_scale8(const short *p) {  // 16-byte aligned
  const uint4 x = *reinterpret_cast<const uint4 *>(p);
  return {{x.x, x.y, x.z, x.w}};
}
template <int kSign>
__device__ __forceinline__ void store8_of(const double *v, int ex, unsigned char *dst, int stride, SlScale8 sc) {
  unsigned w[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const unsigned long long u0 = sl_biased(v[2 * i], ex - kSign * sc.at(2 * i)),
                             u1 = sl_biased(v[2 * i + 1], ex - kSign * sc.at(2 * i + 1));
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
template <int kSign>
__device__ __forceinline__ void store8_of(const float *v, int ex, unsigned char *dst, int stride, SlScale8) {
  unsigned w[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i) sl_parts(v[2 * i], v[2 * i + 1], ex, w[i]);
#pragma unroll
  for (int p = 0; p < 3; ++p)
    *reinterpret_cast<uint4 *>(dst + p * stride) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
}
template <typename T, int kSign = 0>
__device__ __forceinline__ void store8(const T *v, int ex, unsigned char *dst, int stride, SlScale8 sc = {}) {
  store8_of<kSign>(v, ex, dst, stride, sc);
}

// The A rows from registers: this thread's kWdCols columns of its row, scaled
// down by sc if kScaled.  Contains a CTA barrier.
template <typename T, bool kScaled>
__device__ __forceinline__ void wd_cut_regs(const WdCta<T> &w, const T (&v)[kWdCols<T>],
                                            const SlScale8 (&sc)[kWdCols<T> / 8], int row, int hw) {
  constexpr int kGroups = kWdCols<T> / 8;
  int ex = 0;
#pragma unroll
  for (int i = 0; i < kWdCols<T>; ++i) ex = max(ex, kScaled ? sl_exp_at(v[i], -sc[i >> 3].at(i & 7)) : sl_exp(v[i]));
  w.exP[hw * kSlRows + row] = ex;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 64 / kWdCols<T>; ++q) ex = max(ex, w.exP[q * kSlRows + row]);
  if (hw == 0) w.exA[row] = kScaled ? ex : sl_row_exp<T>(ex);
#pragma unroll
  for (int i = 0; i < kGroups; ++i)
    store8<T, kScaled ? -1 : 0>(v + 8 * i, ex, w.A + sl_off(row, kGroups * hw + i), kSlASlab, sc[i]);
}

// Issue the product of the cut operands.  cols2: the second 32 columns as
// well; ks0 / ks1: K steps of either column tile.
template <typename T>
__device__ __forceinline__ void wd_issue(WdCta<T> &w, bool cols2, int ks0, int ks1) {
  // every thread's operands before the products that read them, its TMEM
  // reads before the products that overwrite them
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  // the second tile's commit covers the first's products as well
  if (__shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0) == 0) {
    tc_fence_after();
    if (sl_elect()) {
      sl_issue<T>(w.tmem, w.A, w.B, kSlCols, ks0);
      tc_commit(w.bar);
      if (cols2) {
        sl_issue<T>(w.tmem + kWdBufCols<T>, w.A, w.B + kWdBBytes<T>, kSlCols, ks1);
        tc_commit(w.bar + 1);
      }
    }
    __syncwarp();
  }
}
// Wait (bounded) for a column tile's product, a warp at a time: the warps of
// the first tile drain it while the second is multiplied.  False after a
// timeout; wd_round_end makes that the whole CTA's.
template <typename T>
__device__ __forceinline__ bool wd_wait(const WdCta<T> &w, int tile) {
  const bool ok = mbar_wait(w.bar + tile, tile ? w.ph1 : w.ph0, w.timeout_ns);
  tc_fence_after();
  return __all_sync(0xffffffffu, ok);
}
// End of a round: what it left in shared memory and TMEM has been read.
template <typename T>
__device__ __forceinline__ bool wd_round_end(WdCta<T> &w, bool cols2, bool ok) {
  tc_fence_before();
  ok = __syncthreads_and(ok);
  tc_fence_after();
  if (!ok) {  // once more (bounded), so that no product is in flight when TMEM is freed
    mbar_wait(w.bar, w.ph0, w.timeout_ns);
    if (cols2) mbar_wait(w.bar + 1, w.ph1, w.timeout_ns);
  }
  w.ph0 ^= 1;
  w.ph1 ^= cols2 ? 1u : 0u;
  return ok;
}

// Four columns of the product from TMEM address `at`, as values.
__device__ __forceinline__ void tmem_ld2(uint32_t taddr, uint32_t (&r)[2]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr) : "memory");
}
template <typename T>
__device__ __forceinline__ void wd_drain4(uint32_t at, int ea, const int *exb, T (&v)[4]) {
  constexpr int kDig = SliceFmt<T>::kDig;
#pragma unroll
  for (int c = 0; c < 4; c += 2) {  // two at a time: registers
    uint32_t acc[kDig][2];
#pragma unroll
    for (int q = 0; q < kDig; ++q) tmem_ld2(at + (uint32_t)(q * kSlCols + c), acc[q]);
    tmem_ld_wait();
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float f[kDig];
#pragma unroll
      for (int q = 0; q < kDig; ++q) f[q] = __uint_as_float(acc[q][e]);
      v[c + e] = sl_value(f, ea, exb[c + e]);
    }
  }
}

// Four columns of a warp's 32 rows to memory through the warp's stage, in
// 16-byte pieces where rows allow it.  dst: the warp's first row, first
// column; rows / cols: how many of them exist.  sub: subtract from what is
// there instead.
template <typename T>
__device__ __forceinline__ void wd_store4(unsigned char *stage, const T (&v)[4], T *dst, int ld, int rows,
                                          int cols, bool segs, bool sub) {
  constexpr int kPiece = 16 / sizeof(T), PR = 4 / kPiece;
  const int lane = threadIdx.x & 31;
  // row r, piece pc: neighbouring groups of four rows swap their pieces, so
  // that eight lanes meet eight different bank groups
  auto at = [&](int r, int pc) { return stage + (r * PR + (PR == 2 ? pc ^ ((r >> 2) & 1) : pc)) * 16; };
  __syncwarp();
#pragma unroll
  for (int e = 0; e < PR; ++e) *reinterpret_cast<uint4 *>(at(lane, e)) = *reinterpret_cast<const uint4 *>(v + e * kPiece);
  __syncwarp();
  if (segs) {
#pragma unroll
    for (int u = 0; u < PR; ++u) {
      const int rr = (32 / PR) * u + lane / PR, pc = lane % PR;
      uint4 x = *reinterpret_cast<const uint4 *>(at(rr, pc));
      if (rr < rows && pc * kPiece < cols) {
        uint4 *o4 = reinterpret_cast<uint4 *>(dst + rr * ld + pc * kPiece);
        if (sub) {
          uint4 o = __ldcg(o4);
          T *ov = reinterpret_cast<T *>(&o);
          const T *xv = reinterpret_cast<const T *>(&x);
#pragma unroll
          for (int i = 0; i < kPiece; ++i) ov[i] -= xv[i];
          x = o;
        }
        *o4 = x;
      }
    }
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int rr = 8 * u + (lane >> 2), c = lane & 3;
      const T x = *reinterpret_cast<const T *>(at(rr, c / kPiece) + (c % kPiece) * sizeof(T));
      if (rr < rows && c < cols) {
        T *o = dst + rr * ld + c;
        *o = sub ? ldcg(o) - x : x;
      }
    }
  }
}

// Set up and release of the CTA's tensor-core state.  All threads call.
template <typename T>
__device__ __forceinline__ void wd_begin(WdCta<T> &w, unsigned char *smem_raw, uint64_t *bar, uint32_t *s_tmem,
                                         int *exA, int *exB, int *exP, long long timeout_ns) {
  w.A = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  w.B = w.A + (size_t)SliceFmt<T>::kDig * kSlASlab;
  w.stage = w.B + (threadIdx.x >> 5) * kWdStage * sizeof(T);
  static_assert(kWdWarps<T> * kWdStage * sizeof(T) <= (size_t)kWdBBytes<T>, "the stages fit the first B tile");
  w.bar = bar;
  w.exA = exA;
  w.exB = exB;
  w.exP = exP;
  w.ph0 = w.ph1 = 0;
  w.timeout_ns = timeout_ns;
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
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
  __shared__ uint64_t s_bar[2];                                                                           \
  __shared__ uint32_t s_tmem;                                                                             \
  __shared__ int s_go, s_exA[kSlRows], s_exB[kWdTile], s_exP[64 / kWdCols<T> * kSlRows];                  \
  if (threadIdx.x == 0) s_go = ld_relaxed_i32(&a.st->status) == 0;                                        \
  __syncthreads();                                                                                        \
  if (!s_go) return;                                                                                      \
  WdCta<T> w;                                                                                             \
  wd_begin(w, smem_raw, s_bar, &s_tmem, s_exA, s_exB, s_exP, a.timeout_ns);                               \
  /* this thread drains row `row` (slot row >> 6), kWdCols columns from column cb */                      \
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, hw = warp >> 2, row0 = 32 * (warp & 3),     \
            row = row0 + lane, cb = kWdCols<T> * hw, ctile = cb >> 5;                                     \
  const uint32_t lane_base = w.tmem + ((uint32_t)row0 << 16);                                             \
  const uint32_t accb = lane_base + (uint32_t)ctile * kWdBufCols<T> + (uint32_t)(cb & 31);

}  // namespace bdss
