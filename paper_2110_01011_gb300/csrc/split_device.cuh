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
// Units per accumulation chain of the BF16x3 form: the loss of a chain grows with
// its length. Three parts, against 64 bits: K = 4096, 2560, 2048, 1024 leave L of 15
// factorisations 1.48e-6, 1.28e-6, 1.26e-6, 9.0e-7 off on average (P 5.5e-6, 4.5e-6,
// 4.4e-6, 2.9e-6); 8192^2, k = 128 took 1204 us at 2048 and 1222 us at 1024, where the
// single main accumulator waits for every drain. Batches keep 4096 with three parts
// as well (24 problems: L 2.8e-6 off, 2.3e-6 at 2048): with other chains single entries of
// ill-conditioned problems move by up to 1.6e-3 of their size.
constexpr int kChainTwo = 4096 / BK, kChainThree = 2048 / BK, kChainBatch = 4096 / BK;
constexpr uint32_t kABytes = BM * BK * 4;        // FP32 stage of A by TMA
constexpr long long kWaitLimit = 4000000000LL;   // cycles (~2 s)
// The FP32 form splits 2^24 A and 2^24 X: no FP32 value has a bit below 2^-149, so
// every nonzero part is then a normal BF16 number and three of them hold the value,
// however small it is. (Without the factor one nonzero value below 2^-96, of which a
// kernel matrix or a localised basis has many, sent the whole product to the FMA
// units: 16384 x 12288, q = 1 with such entries 11.9 ms, now 3.24 as without them.)
// The drain warps take the sums back by 2^-48 in the multiply-add that was an add,
// so ordinary results are the same bits. What overflows on the way, values of 2^104 and sums of
// 2^80 upward, gives sums that are not finite, which the drain warps look for.
constexpr float kScaleUp = 16777216.f, kScaleDown = 1.f / (kScaleUp * kScaleUp);

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
// Arrive on the pair leader's barrier. Relaxed: what these arrivals hand over lies
// in tensor memory and is ordered by the tcgen05 waits and fences around them; a
// releasing arrive at cluster scope takes most of a microsecond (a unit of 256 x
// 32 took 1.5 us with it and 0.7 us without). Shared memory is never handed over
// this way.
__device__ __forceinline__ uint32_t leader_addr(const void* p) {   // p's place in the leader's shared memory
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(tc::smem_u32(p)));
  return remote;
}
__device__ __forceinline__ void arrive_remote(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void arrive_leader(uint64_t* bar) { arrive_remote(leader_addr(bar)); }
// Hands back a stage that the warp's lanes have read, for a copy to refill: every
// lane's reads are over before the copy may write (proxy fence), and the arrive
// releases. Without the fence the arrive overtook reads that waited behind the
// drain warps' stores, and a tile's values came from eight units of K later.
__device__ __forceinline__ void arrive_read(uint64_t* bar, int lane) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0) tc::mbar_arrive(bar);
}
// Acquires at CTA scope.
__device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity) { return tc::mbar_wait(bar, parity, kWaitLimit); }
// The same by a whole warp, with one answer for all lanes: a limit that runs out
// in some of them must not part the warp in front of an elect or a barrier.
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, wait(bar, parity));
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
// A box of X's image into this CTA's shared memory, counted by a barrier of the
// pair's leader (both CTAs' halves of a stage complete on it, so the MMAs, which
// read both, wait for one barrier that the copies themselves signal).
__device__ __forceinline__ void load_image(void* dst, const CUtensorMap* map, uint32_t leader_bar, int row) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(tc::smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(leader_bar)
      : "memory");
}
constexpr int kImgRow = 256;   // BF16 entries of an image row: 8 columns of X by 32 of K
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

// The split warps' sum of squares of A, Kahan-compensated per unit.
struct Squares {
  float ss = 0.f, comp = 0.f, part = 0.f;
  __device__ void fold() {
    const float y = part - comp, t = ss + y;
    comp = (t - ss) - y;
    ss = t;
    part = 0.f;
  }
  __device__ void add(double* sumsq, int lane) const {
    double v = (double)ss - (double)comp;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) atomicAdd(sumsq, v);
  }
};
// Sixteen values along K -> eight packed columns per part.
template <int PARTS>
__device__ __forceinline__ void split_half(float* v, uint32_t (&o)[PARTS][8], bool scaled, bool sq, Squares& sum) {
  if (sq) {
#pragma unroll
    for (int j = 0; j < 16; ++j) sum.part = fmaf(v[j], v[j], sum.part);
  }
  if (scaled) {
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] *= kScaleUp;
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
// Sums that a drain warp could not read (its wait ran out): NaN, which no result
// hides and which check_sums reports.
template <int NG>
__device__ __forceinline__ void lose_sums(float (&s)[NG][16]) {
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int j = 0; j < 16; ++j) s[g][j] = __int_as_float(0x7fffffff);
}
// s += f times ng groups of 16 accumulator columns of this lane's row; all lanes.
template <int NG>
__device__ __forceinline__ void drain_columns(float (&s)[NG][16], uint32_t ta, int ng, float f) {
#pragma unroll
  for (int g = 0; g < NG; ++g) {
    if (g < ng) {
      float v[16];
      ld16(ta + 16 * g, v);
      ld_wait();
      ld_done(v);
#pragma unroll
      for (int j = 0; j < 16; ++j) s[g][j] = fmaf(v[j], f, s[g][j]);
    }
  }
  tc::tc_fence_before();
  __syncwarp();
}
// Raises *bad where one of the ncols sums of the lane's row is not finite.
template <int NG>
__device__ __forceinline__ void check_sums(const float (&s)[NG][16], int g0, int ng, int ncols, int* bad) {
  bool fine = true;
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (g < ng && 16 * (g0 + g) + j < ncols) fine = fine && fabsf(s[g][j]) <= 3.402823466e38f;
  if (!fine) atomicOr(bad, 1);
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
// X (K x N FP32) -> stage images (read back as boxes of 512-byte rows): for every unit of 32 of K, CTA of a group,
// and part, npad / CG rows (columns of X) of 32 K entries, 16-byte chunks
// swizzled over 64-byte rows; zeros past K and N. A block of 256 threads takes
// 64 of K and 32 columns through shared memory; a thread writes one 16-byte
// chunk (8 of K) of each part.
__device__ __forceinline__ void split_x_tile(const float* __restrict__ X, long long K, int N, long long ldx,
                                             uint16_t* __restrict__ img, int npad, int parts, int kb, long long k0,
                                             int n0, int* xlo, bool scaled) {
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
  const float up = scaled ? kScaleUp : 1.f;
  bool any = false;
  if (n < npad && unit < kb) {
    uint32_t p[3][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t q[3];
      split2<3>(up * tile[ch * 8 + 2 * j][nn], up * tile[ch * 8 + 2 * j + 1][nn], q);
      p[0][j] = q[0]; p[1][j] = q[1]; p[2][j] = q[2];
      any |= (q[1] & 0x7FFF7FFFu) != 0;
    }
    const int nh = npad / CG, r = n % nh;
    const size_t stage = ((size_t)unit * CG + n / nh) * parts * nh * 32;
    const size_t at = stage + (size_t)r * 32 + (size_t)(((ch & 3) ^ ((r >> 1) & 3)) * 8);
    for (int q = 0; q < parts; ++q)
      *reinterpret_cast<uint4*>(img + at + (size_t)q * nh * 32) = make_uint4(p[q][0], p[q][1], p[q][2], p[q][3]);
  }
  if (__syncthreads_or(any) && threadIdx.x == 0 && *(volatile int*)xlo == 0) atomicOr(xlo, 1);
}

// ---------------------------------------------------------------- A with rows at any 4-byte address
// TMA wants 16-byte aligned rows. Four rows apart, rows of any FP32 matrix have
// the same alignment and a stride that is a multiple of 16 bytes: so one map
// takes the rows of one class r % 4, from the aligned address at or before the
// class's first value, and the values lie `shift` floats behind where the map
// puts them. A stage is four boxes, four floats wider than the tile; what lies
// past A is zero. op(A) = A: box c holds 32 rows (4 i + c) of 36 floats, read by
// split warp c, so that TMEM lane 32 c + i is row 4 i + c of the tile. op(A) =
// A^T: box c holds 8 rows (K = 4 i + c) of 132 floats. (Copies by the split
// warps themselves, nine 16-byte chunks per row, took 1.3 to 1.7 times as long
// per unit.)
constexpr uint32_t kBoxN = 32 * 36 * 4, kBoxT = 8 * 132 * 4;   // bytes of a box
constexpr uint32_t kClassBytes = 4 * kBoxN;                    // a stage
struct Classes {
  int shift[4];
  int past[4];             // 1: no row in the class (its box starts past the map's end)
};
// The map of X's image for products of kb units, boxes of one part of a stage;
// the four maps of A (rows x cols, row stride lda). False when the encoder is missing.
bool image_map(CUtensorMap* m, const uint16_t* img, int kb, int npad, int parts);
bool class_maps(CUtensorMap* m, Classes* cl, const float* A, int64_t rows, int64_t cols, int64_t lda, bool trans);
template <bool TRANS>
__device__ __forceinline__ void load_classes(unsigned char* f, const CUtensorMap* m0, const CUtensorMap* m1,
                                             const CUtensorMap* m2, const CUtensorMap* m3, const Classes& cl,
                                             uint64_t* bar, int k, int row) {
  const CUtensorMap* m[4] = {m0, m1, m2, m3};
  tc::mbar_expect_tx(bar, 4 * (TRANS ? kBoxT : kBoxN));
#pragma unroll
  for (int c = 0; c < 4; ++c)   // first columns are multiples of 32 floats
    tc::tma_load_2d(f + c * (TRANS ? kBoxT : kBoxN), m[c], bar, TRANS ? row : k, (TRANS ? k : row) / 4 + cl.past[c]);
}
// v[j] = op(A)(this lane's row, 16 half + j) of split warp w.
template <bool TRANS>
__device__ __forceinline__ void read_classes(const unsigned char* f, const Classes& cl, int w, int half, int lane,
                                             float* v) {
  if (TRANS) {
    const float* p[4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
      p[c] = reinterpret_cast<const float*>(f + c * kBoxT) + 4 * half * 132 + cl.shift[c] + 32 * w + lane;
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = p[j & 3][(j >> 2) * 132];
  } else {
    const int s = w < 2 ? (w == 0 ? cl.shift[0] : cl.shift[1]) : (w == 2 ? cl.shift[2] : cl.shift[3]);
    const float* p = reinterpret_cast<const float*>(f + w * kBoxN) + lane * 36 + 16 * half;
    float x[20];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const float4 q = *reinterpret_cast<const float4*>(p + 4 * i);
      x[4 * i] = q.x; x[4 * i + 1] = q.y; x[4 * i + 2] = q.z; x[4 * i + 3] = q.w;
    }
#pragma unroll
    for (int i = 0; i < 18; ++i) x[i] = s & 1 ? x[i + 1] : x[i];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = s & 2 ? x[i + 2] : x[i];
  }
}

}  // namespace sp
}  // namespace rqlp
