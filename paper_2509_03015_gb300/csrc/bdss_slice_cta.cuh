// One CTA's share of the digit products (bdss_slice.cuh): 128 A rows by 64 B
// rows by a K chunk of 64, cut by 16 warps into shared memory, multiplied by
// one thread's tcgen05.mma and drained by the same warps.
#pragma once
#include "bdss_slice.cuh"

namespace bdss {

constexpr int kWdThreads = 512;
constexpr int kWdWarps = kWdThreads / 32;
constexpr int kWdTile = 64;  // rows of a slot, columns of an output tile
template <typename T> constexpr int kWdStageRow = sizeof(T) == 8 ? 48 : 16;  // bytes of a staged output row
template <typename T> constexpr uint32_t kWdBufCols = SliceFmt<T>::kDig * kSlCols;  // accumulators of 32 columns
template <typename T> constexpr uint32_t kWdTmem = sizeof(T) == 8 ? 512 : 256;  // a power of two
template <typename T> constexpr int kWdBBytes = SliceFmt<T>::kDig * kSlBSlab;
template <typename T> constexpr size_t wd_smem() {
  return (size_t)SliceFmt<T>::kDig * (kSlASlab + 2 * kSlBSlab) + (size_t)kWdWarps * 32 * kWdStageRow<T> + 1024;
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
  unsigned w[4][3];
#pragma unroll
  for (int i = 0; i < 4; ++i) sl_parts(v[2 * i], v[2 * i + 1], ex, w[i]);
#pragma unroll
  for (int p = 0; p < 3; ++p)
    *reinterpret_cast<uint4 *>(dst + p * stride) = make_uint4(w[0][p], w[1][p], w[2][p], w[3][p]);
}

// The A rows from registers: this thread's 16 columns of its row.  Contains a
// CTA barrier.
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
__device__ __forceinline__ void wd_store4(unsigned char *stage, const T (&v)[4], T *dst, int ld, int rows,
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

}  // namespace bdss
