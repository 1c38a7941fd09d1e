// Device parts shared by the single and the grouped split products
// (split_gemm.cu, split_grouped.cu): pair-wide tcgen05 operations, the split of
// FP32 values into BF16 parts and the copies of FP32 tiles of A.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace rqlp {
namespace sp {

constexpr int BM = 128;               // rows per CTA (TMEM lanes)
constexpr int BK = 32;                // K per unit
constexpr int CG = 2;                 // CTAs per tile (cta_group::2)
constexpr int kThreads = 640;         // 4 + 8 + 8 warps
constexpr int kGroups = 7;            // 16-column groups of a drain warp: N <= 224
constexpr int kMaxStages = 8;
constexpr int kMaxASlots = 8;
constexpr uint32_t kABytes = BM * BK * 4;        // FP32 stage of A by TMA
constexpr int kRowFloats = BK + 4;               // a row of a stage copied by the split warps: nine 16-byte chunks
constexpr uint32_t kCopyBytes = BM * kRowFloats * 4;   // such a stage (18 KB)
constexpr int kCopyStages = 6;
constexpr int kPrefetch = 12;         // units between the L2 prefetch and the copy
constexpr long long kWaitLimit = 4000000000LL;   // cycles (~2 s)
// Parts hold a value exactly when its magnitude lies in [2^-96, 2^127) (or is
// zero): below, the last part would be subnormal; above, the first may round
// to infinity.
constexpr uint32_t kRangeHi = 0x7F000000u, kRangeLo = 0x0F800000u;

__device__ inline void post_timeout(int* info) {
  if (info != nullptr && atomicCAS(info, 0, RQLP_ERR_TIMEOUT) == 0) info[1] = 0;
}

// Tile and unit of K at a position of a range.
struct Cursor {
  int t, k;
  __device__ Cursor(int u, int kb) : t(u / kb), k(u % kb) {}
  __device__ void next(int kb) {
    if (++k == kb) {
      k = 0;
      ++t;
    }
  }
};
// Stage of a ring and the parity of its current round.
struct Ring {
  int s = 0;
  uint32_t ph = 0;
  __device__ void next(int n) {
    if (++s == n) {
      s = 0;
      ph ^= 1u;
    }
  }
};

// D[tmem] (+)= A[tmem] B[shared memory] over the CTA pair, issued by its leader.
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
               " tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d), "r"(a), "l"(b),
               "r"(idesc), "r"(acc) : "memory");
}
// Arrive on `bar` of both CTAs of the pair once the MMAs issued so far are done.
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(tc::smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// Arrive on the pair leader's barrier. Relaxed: what the arrival hands over
// lies in tensor memory and is ordered by the tcgen05 waits and fences around
// it; a releasing arrive at cluster scope takes most of a microsecond (a unit
// of 256 x 32 took 1.5 us with it and 0.7 us without).
__device__ __forceinline__ void arrive_leader(uint64_t* bar) {
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(tc::smem_u32(bar)));
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
__device__ __forceinline__ bool try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.relaxed.cta.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok) : "r"(tc::smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Wait for MMAs, tensor-memory hand-overs or free stages; data that was copied
// to shared memory is waited for with tc::mbar_wait (acquire).
__device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity) {
  if (try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!try_wait(bar, parity))
    if (clock64() - t0 > kWaitLimit) return false;
  return true;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// True in one lane of a converged warp. The loops that issue copies and MMAs run
// in the whole warp with the issue itself under elect: their operands then stay
// in uniform registers (under a divergent branch an MMA took ~75 clocks to
// issue).
__device__ __forceinline__ bool elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   tc::smem_u32(dst)), "l"(src), "r"(bytes), "r"(tc::smem_u32(bar)) : "memory");
}
// Eight 32-bit columns of this lane's row.
__device__ __forceinline__ void st_row8(uint32_t t, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(t), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}
// Sixteen columns of this lane's row; the values are there after ld_wait().
__device__ __forceinline__ void ld16(uint32_t t, float* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]), "=f"(v[8]),
        "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15])
      : "r"(t));
}
__device__ __forceinline__ void ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Keeps the uses of v behind the wait above (no instruction).
__device__ __forceinline__ void ld_done(float* v) {
  asm volatile("" : "+f"(v[0]), "+f"(v[1]), "+f"(v[2]), "+f"(v[3]), "+f"(v[4]), "+f"(v[5]), "+f"(v[6]), "+f"(v[7]),
                    "+f"(v[8]), "+f"(v[9]), "+f"(v[10]), "+f"(v[11]), "+f"(v[12]), "+f"(v[13]), "+f"(v[14]),
                    "+f"(v[15]));
}
__device__ __forceinline__ void st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// (x0, x1) -> packed parts; the differences are exact in FP32.
template <int PARTS>
__device__ __forceinline__ void split2(float x0, float x1, uint32_t* p) {
  p[0] = pack(x0, x1);
  const float r0 = x0 - __uint_as_float(p[0] << 16), r1 = x1 - __uint_as_float(p[0] & 0xFFFF0000u);
  p[1] = pack(r0, r1);
  if (PARTS == 3) p[2] = pack(r0 - __uint_as_float(p[1] << 16), r1 - __uint_as_float(p[1] & 0xFFFF0000u));
}

// The products of one unit: d the main accumulator, dc the corrections', t0 the
// A slot, x the descriptors of X's parts (16 of K are 32 bytes on).
template <int PARTS>
__device__ __forceinline__ void issue_products(uint32_t d, uint32_t dc, uint32_t t0, const uint64_t* x, uint32_t idesc,
                                               int nx, bool corr_first, uint32_t acc, uint32_t cacc) {
  if (PARTS == 3 && corr_first) {   // a chain of one unit: the small products, then the main ones
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      const uint32_t t = t0 + ks * 8;
      mma_ts(d, t + 32, x[0] + 2 * ks, idesc, ks);
      if (nx > 1) {
        mma_ts(d, t + 16, x[1] + 2 * ks, idesc, 1u);
        mma_ts(d, t, x[PARTS - 1] + 2 * ks, idesc, 1u);
        mma_ts(d, t, x[1] + 2 * ks, idesc, 1u);
      }
      mma_ts(d, t + 16, x[0] + 2 * ks, idesc, 1u);
    }
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) mma_ts(d, t0 + ks * 8, x[0] + 2 * ks, idesc, 1u);
  } else {
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
      const uint32_t t = t0 + ks * 8;
      mma_ts(d, t, x[0] + 2 * ks, idesc, ks ? 1u : acc);
      mma_ts(dc, t + 16, x[0] + 2 * ks, idesc, ks ? 1u : cacc);
      if (nx > 1) mma_ts(dc, t, x[1] + 2 * ks, idesc, 1u);
      if (PARTS == 3) {
        mma_ts(dc, t + 32, x[0] + 2 * ks, idesc, 1u);
        if (nx > 1) {
          mma_ts(dc, t + 16, x[1] + 2 * ks, idesc, 1u);
          mma_ts(dc, t, x[PARTS - 1] + 2 * ks, idesc, 1u);
        }
      }
    }
  }
}

// What the split warps collect beside the parts: the extremes of |A| (zero
// counts as large) and the sum of squares, Kahan-compensated per unit.
struct Checks {
  uint32_t umax = 0, umin = 0xFFFFFFFFu;
  float ss = 0.f, comp = 0.f, part = 0.f;
  __device__ void fold() {
    const float y = part - comp, t = ss + y;
    comp = (t - ss) - y;
    ss = t;
    part = 0.f;
  }
  __device__ void report(int* bad, int lane) const {
    if (__any_sync(0xffffffffu, umax >= kRangeHi || umin < kRangeLo - 1u) && lane == 0) atomicOr(bad, 1);
  }
  __device__ void add(double* sumsq, int lane) const {
    double v = (double)ss - (double)comp;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) atomicAdd(sumsq, v);
  }
};
// Sixteen values along K -> eight packed columns per part.
template <int PARTS>
__device__ __forceinline__ void split_half(const float* v, uint32_t (&o)[PARTS][8], bool check, bool sq, Checks& ck) {
  if (check) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const uint32_t x = __float_as_uint(v[j]) & 0x7FFFFFFFu;
      ck.umax = max(ck.umax, x);
      ck.umin = min(ck.umin, x - 1u);   // zero wraps to the largest value
    }
  }
  if (sq) {
#pragma unroll
    for (int j = 0; j < 16; ++j) ck.part = fmaf(v[j], v[j], ck.part);
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint32_t p[PARTS];
    split2<PARTS>(v[2 * j], v[2 * j + 1], p);
#pragma unroll
    for (int q = 0; q < PARTS; ++q) o[q][j] = p[q];
  }
}

// ---------------------------------------------------------------- drain warps
template <int NG>
__device__ __forceinline__ void clear_sums(float (&s)[NG][16]) {
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int j = 0; j < 16; ++j) s[g][j] = 0.f;
}
// s += ng groups of 16 accumulator columns of this lane's row; all lanes.
template <int NG>
__device__ __forceinline__ void drain_columns(float (&s)[NG][16], uint32_t ta, int ng) {
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    if (g < ng) {
      float v[16];
      ld16(ta + 16 * g, v);
      ld_wait();
      ld_done(v);
#pragma unroll
      for (int j = 0; j < 16; ++j) s[g][j] += v[j];
    }
  }
  tc::tc_fence_before();
  __syncwarp();
}
// s -> ncols columns of the lane's row at dst (float4 q of it at q qstep; vec:
// 16-byte aligned), added to what an earlier flush left there.
template <int NG>
__device__ __forceinline__ void store_sums(float (&s)[NG][16], float* dst, int qstep, int g0, int ng, int ncols,
                                           bool vec, bool flushed) {
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    const int c0 = 16 * (g0 + g);
    if (g < ng) {
      if (flushed) {
        if (vec && c0 + 16 <= ncols) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float4 o = *reinterpret_cast<const float4*>(dst + (c0 / 4 + q) * qstep);
            s[g][4 * q] += o.x; s[g][4 * q + 1] += o.y; s[g][4 * q + 2] += o.z; s[g][4 * q + 3] += o.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (c0 + j < ncols) s[g][j] += dst[c0 + j];
        }
      }
      if (vec && c0 + 16 <= ncols) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float4*>(dst + (c0 / 4 + q) * qstep) =
              make_float4(s[g][4 * q], s[g][4 * q + 1], s[g][4 * q + 2], s[g][4 * q + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          if (c0 + j < ncols) dst[c0 + j] = s[g][j];
      }
    }
  }
}

// ---------------------------------------------------------------- X
// X (K x N FP32) -> stage images: for every unit of 32 of K, CTA of a group,
// and part, npad / CG rows (columns of X) of 32 K entries, 16-byte chunks
// swizzled over 64-byte rows; zeros past K and N. A block of 256 threads takes
// 64 of K and 32 columns through shared memory; a thread writes one 16-byte
// chunk (8 of K) of each part.
__device__ __forceinline__ void split_x_tile(const float* __restrict__ X, long long K, int N, long long ldx,
                                             uint16_t* __restrict__ img, int npad, int parts, int kb, long long k0,
                                             int n0, int* xlo, int* bad) {
  __shared__ float tile[64][33];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int kk = (threadIdx.x >> 5) + 8 * i, nn = threadIdx.x & 31;
    const long long k = k0 + kk;
    tile[kk][nn] = (k < K && n0 + nn < N) ? X[k * ldx + n0 + nn] : 0.f;
  }
  __syncthreads();
  const int nn = threadIdx.x >> 3, ch = threadIdx.x & 7;   // column, chunk of 8 of K
  const int n = n0 + nn;
  const long long unit = (k0 >> 5) + (ch >> 2);
  bool any = false, out_of_range = false;
  if (n < npad && unit < kb) {
    uint32_t p[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t q[3];
      const float x0 = tile[ch * 8 + 2 * j][nn], x1 = tile[ch * 8 + 2 * j + 1][nn];
      split2<3>(x0, x1, q);
      p[0][j] = q[0]; p[1][j] = q[1]; p[2][j] = q[2];
      any |= (q[1] & 0x7FFF7FFFu) != 0;
      const uint32_t m0 = __float_as_uint(x0) & 0x7FFFFFFFu, m1 = __float_as_uint(x1) & 0x7FFFFFFFu;
      out_of_range |= max(m0, m1) >= kRangeHi || min(m0 - 1u, m1 - 1u) < kRangeLo - 1u;
    }
    const int nh = npad / CG, r = n % nh;
    const size_t stage = ((size_t)unit * CG + n / nh) * parts * nh * 32;
    const size_t at = stage + (size_t)r * 32 + (size_t)(((ch & 3) ^ ((r >> 1) & 3)) * 8);
    for (int q = 0; q < parts; ++q)
      *reinterpret_cast<uint4*>(img + at + (size_t)q * nh * 32) = make_uint4(p[q][0], p[q][1], p[q][2], p[q][3]);
  }
  if (__syncthreads_or(any) && threadIdx.x == 0 && *(volatile int*)xlo == 0) atomicOr(xlo, 1);
  if (bad != nullptr && __syncthreads_or(out_of_range) && threadIdx.x == 0) atomicOr(bad, 1);
}

// ---------------------------------------------------------------- copies of A by the split warps
// Without TMA (rows of A that are not 16-byte aligned, or many problems): a
// warp copies its 32 rows of a stage by 16-byte asynchronous copies. The 32
// values of a row start at any 4-byte address, so nine aligned chunks cover
// them, shift() words ahead of the first. (By 4-byte copies, 32 instead of nine
// instructions a unit, a unit took twice as long.) TRANS: stage rows are rows of
// memory, this warp's 32 columns each; else this warp's rows, 32 of K each.
struct ARef {
  const float* A;
  long long lda;
  int M, K;                // op(A) is M x K
};
// Byte offsets of this lane's nine chunks (chunk lane + 32 i: row r = e / 9) from
// a warp's first value in a unit. They are the same for every unit, as first
// rows and columns are multiples of 32. False when a row stride is too long
// for them.
__device__ __forceinline__ bool chunk_offsets(const ARef& a, int lane, int (&off)[9]) {
  const int b = (int)(reinterpret_cast<uintptr_t>(a.A) & 15);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int e = lane + 32 * i, r = e / 9, c = e - 9 * r;
    off[i] = (int)((((long long)r * a.lda * 4 + b) & ~15LL) + 16 * c - b);
  }
  return a.lda < (1 << 24);
}
// The same copy as copy_rows for a unit whose chunks all lie inside A.
__device__ __forceinline__ void copy_interior(const ARef& a, long long i0, long long j0, const int (&off)[9], float* dst,
                                              int lane) {
  const char* p = reinterpret_cast<const char*>(a.A + i0 * a.lda + j0);
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst) + 16 * lane;   // chunk e at 16 e: rows are nine chunks
#pragma unroll
  for (int i = 0; i < 9; ++i)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 512 * i), "l"(p + off[i]) : "memory");
}
__device__ __forceinline__ bool interior(const ARef& a, bool trans, long long i0, long long j0) {
  return i0 + 32 <= (trans ? a.K : a.M) && j0 + kRowFloats <= (trans ? a.M : a.K) &&
         (i0 > 0 || j0 > 0 || (reinterpret_cast<uintptr_t>(a.A) & 15) == 0);
}
// Copies rows r = 0 .. 31 of this warp (first row / column of memory: i0, j0)
// to dst; rows past the end of memory are zeros, chunks outside A are clipped.
__device__ __forceinline__ void copy_rows(const ARef& a, bool trans, long long i0, long long j0, float* dst, int lane) {
  const long long rows = trans ? a.K : a.M, cols = trans ? a.M : a.K;
  const char* lo = reinterpret_cast<const char*>(a.A);
  const char* hi = reinterpret_cast<const char*>(a.A + (rows - 1) * a.lda + cols);   // end of A
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int e = lane + 32 * i, r = e / 9, c = e - 9 * r;
    const char* p = reinterpret_cast<const char*>(a.A + (i0 + r) * a.lda + j0);
    p = reinterpret_cast<const char*>(reinterpret_cast<uintptr_t>(p) & ~uintptr_t(15)) + 16 * c;
    float* d = dst + r * kRowFloats + 4 * c;
    const long long left = hi - p;
    if (i0 + r >= rows || left <= 0) {
      cp_async16(d, reinterpret_cast<const void*>(reinterpret_cast<uintptr_t>(lo) & ~uintptr_t(15)), 0);
    } else if (p < lo) {   // the chunk that A's first value lies in
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const char* q = p + 4 * u;
        cp_async4(d + u, q >= lo && q < hi ? q : lo, q >= lo && q < hi ? 4 : 0);
      }
    } else {
      cp_async16(d, p, left < 16 ? (int)left : 16);
    }
  }
}
__device__ __forceinline__ int shift(const float* p) { return (int)((reinterpret_cast<uintptr_t>(p) >> 2) & 3); }

// v[j] = op(A)(this lane's row, k0 + 16 half + j) from such a stage (this
// warp's part of it), zero past M and K (what lies there in memory is not A's).
template <bool TRANS>
__device__ __forceinline__ void read_copied(const ARef& a, int k0, int r0, const float* f, int half, int lane, float* v) {
  if (TRANS) {
    // row k of the stage is shifted by (s + k lda) % 4
    const int s = shift(a.A + (long long)k0 * a.lda + r0), l3 = (int)(a.lda & 3);
    const float* p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = f + (16 * half + j) * kRowFloats + ((s + j * l3) & 3) + lane;
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = p[j & 3][(j & ~3) * kRowFloats];
  } else {
    const int s = shift(a.A + (long long)(r0 + lane) * a.lda + k0);
    const float* p = f + lane * kRowFloats + 16 * half;
    float w[20];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const float4 q = *reinterpret_cast<const float4*>(p + 4 * i);
      w[4 * i] = q.x; w[4 * i + 1] = q.y; w[4 * i + 2] = q.z; w[4 * i + 3] = q.w;
    }
#pragma unroll
    for (int i = 0; i < 18; ++i) w[i] = s & 1 ? w[i + 1] : w[i];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = s & 2 ? w[i + 2] : w[i];
  }
  if (k0 + 16 * half + 16 > a.K || r0 + 32 > a.M) {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (k0 + 16 * half + j >= a.K || r0 + lane >= a.M) v[j] = 0.f;
  }
}
// One line of A per lane into L2.
__device__ __forceinline__ void prefetch_rows(const ARef& a, bool trans, long long i0, long long j0, int lane) {
  const long long rows = trans ? a.K : a.M, cols = trans ? a.M : a.K;
  if (i0 + lane < rows && j0 < cols)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a.A + (i0 + lane) * a.lda + j0));
}

}  // namespace sp
}  // namespace rqlp
