// Products of the first CholeskyQR pass in the BF16x3 form (tcgen05 / TMEM / TMA):
// the Gram X^T X of a tall X and X R^{-1}, X split into BF16 parts in memory once
// for both.
//
// The Gram takes two parts, X = X_hi + X_lo, and the products hi hi + hi lo + lo hi
// (its factor only preconditions). X R^{-1} takes three of each operand and
// every product above 2^-27, A_hi X_hi + A_hi X_lo + A_lo X_hi + A_lo2 X_hi + A_hi
// X_lo2 + A_lo X_lo (six): R^{-1} spreads its entries over orders of magnitude, so
// the two-part form's error, relative to |X| |R^{-1}|, would be kappa(X) times
// larger relative to the result.
//
// split_a_kernel writes the parts in 64-column panels: panel c / 64 holds rows 0
// .. m - 1 of those 64 columns, 128 bytes per row, so that 128 rows of one panel are
// one TMA box; prep_x_kernel writes the other operand's parts transposed
// (d x K, K-major). tc_pass_kernel is persistent, a CTA taking whole 128-row
// tiles: warps 0-3 drain the accumulator from TMEM (each warp its 32 lanes),
// warp 4 issues TMA loads, warp 5 allocates TMEM and issues the MMAs. Every wait
// is bounded; a timeout is reported in the status word and the kernel drains what
// it started and frees its TMEM before returning.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace rqlp {
namespace {

using bf16 = __nv_bfloat16;

constexpr int BM = 128;              // MMA M: output rows per tile (TMEM lanes)
constexpr int BK = 32;               // K per pipeline stage of the Gram kernel (64 bytes of BF16)
constexpr int kThreads = 192;        // 6 warps
constexpr int kMaxStages = 8;
constexpr long long kWaitLimit = 4000000000LL;   // cycles (~2 s) before a wait gives up
// K per pipeline stage of a product: 64 (128-byte rows, 128B swizzle) where at least
// three such stages fit in shared memory, else 32 (64-byte rows, 64B swizzle).
// Larger TMA boxes stream faster, but the pipeline needs stages in flight.

struct TcArgs {
  int M, d, npad, kblocks, tiles, stages;
  int tpc;                   // whole tiles per CTA
  int vec_out;               // out rows are 16-byte aligned (float4 stores)
  float* out;
  long long ldo;
  int nbuf;                  // pairs of accumulators (2: the epilogue overlaps the next tile)
  int* info;                 // status word (may be null)
  uint32_t idesc, stage_bytes, tmem_cols;
};

__device__ void post_timeout(int* info) {
  if (info != nullptr && atomicCAS(info, 0, RQLP_ERR_TIMEOUT) == 0) info[1] = 0;
}

// out = A X with A and X in three parts. A tile's products go to two accumulators, the
// main product's and the corrections': these are ~2^-8 of it or smaller, and added to
// the same FP32 sum they would lose bits to its magnitude at every MMA. The epilogue
// adds the two with round-to-nearest. K = d <= 256: one chain per tile.
template <int BKP>
__global__ void __launch_bounds__(kThreads, 1)
tc_pass_kernel(const __grid_constant__ CUtensorMap tmAhi, const __grid_constant__ CUtensorMap tmAlo,
               const __grid_constant__ CUtensorMap tmXhi, const __grid_constant__ CUtensorMap tmXlo,
               const __grid_constant__ CUtensorMap tmAlo2, const __grid_constant__ CUtensorMap tmXlo2,
               const TcArgs a) {
  grid_wait();
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)S * a.stage_bytes);
  uint64_t* empty = full + S;
  uint64_t* accf = empty + S;
  uint64_t* acce = accf + 2;
  uint64_t* done = acce + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int* epi_ok = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t0 = (int)blockIdx.x * a.tpc, t1 = min(t0 + a.tpc, a.tiles);   // this CTA's tiles (at least one)
  const int KB = a.kblocks;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&accf[b], 1);
      tc::mbar_init(&acce[b], 4 * 32);
    }
    tc::mbar_init(done, 1);
    tc::fence_barrier_init();
  }
  if (warp == 5) {
    tc::tmem_alloc(tmem_slot, a.tmem_cols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Stage layout: A_hi, A_lo, A_lo2, X_hi, X_lo, X_lo2.
  constexpr uint32_t kAP = BM * BKP * 2;    // one BF16 A tile
  constexpr uint32_t kRow = BKP * 2;        // bytes of a K-major row: the swizzle span
  constexpr uint32_t kSbo = 8 * kRow;       // 8-row swizzle atom of the K-major operands
  constexpr uint32_t kSw = BKP == 64 ? tc::kSwizzle128 : tc::kSwizzle64;
  const uint32_t xbytes = (uint32_t)a.npad * BKP * 2;
  constexpr uint32_t xoff = 3 * kAP;

  if (warp == 4 && lane == 0) {
    // ------------------------------------------------ TMA producer
    tc::prefetch_tmap(&tmAhi);
    tc::prefetch_tmap(&tmAlo);
    tc::prefetch_tmap(&tmAlo2);
    tc::prefetch_tmap(&tmXhi);
    tc::prefetch_tmap(&tmXlo);
    tc::prefetch_tmap(&tmXlo2);
    const int n = (t1 - t0) * KB;
    int issued = 0;
    bool ok = true;
    for (; issued < n; ++issued) {
      const int stage = issued % S;
      if (!tc::mbar_wait(&empty[stage], (uint32_t)((issued / S) & 1) ^ 1u, kWaitLimit)) { ok = false; break; }
      const int mr = (t0 + issued / KB) * BM, k = issued % KB * BKP;
      unsigned char* base = smem + (size_t)stage * a.stage_bytes;
      tc::mbar_expect_tx(&full[stage], xoff + 3 * xbytes);
      // A maps are 3-D over the panel layout, {column in panel, row, panel}:
      // 128 rows (M) x BKP columns (K) of panel k / 64
      tc::tma_load_3d(base, &tmAhi, &full[stage], k & 63, mr, k >> 6);
      tc::tma_load_3d(base + kAP, &tmAlo, &full[stage], k & 63, mr, k >> 6);
      tc::tma_load_3d(base + 2 * kAP, &tmAlo2, &full[stage], k & 63, mr, k >> 6);
      tc::tma_load_2d(base + xoff, &tmXhi, &full[stage], k, 0);
      tc::tma_load_2d(base + xoff + xbytes, &tmXlo, &full[stage], k, 0);
      tc::tma_load_2d(base + xoff + 2 * xbytes, &tmXlo2, &full[stage], k, 0);
    }
    if (!ok) post_timeout(a.info);
    // Drain: every load this thread started has landed before the CTA exits.
    for (int i = max(0, issued - S); i < issued; ++i)
      if (!tc::mbar_wait(&full[i % S], (uint32_t)((i / S) & 1), kWaitLimit)) post_timeout(a.info);
  } else if (warp == 5 && lane == 0) {
    // ------------------------------------------------ MMA issuer
    int consumed = 0;
    bool ok = true;
    for (int t = t0; t < t1 && ok; ++t) {
      const int seg = t - t0, ab = seg % a.nbuf;
      if (!tc::mbar_wait(&acce[ab], (uint32_t)(((seg / a.nbuf) & 1) ^ 1), kWaitLimit)) { ok = false; break; }
      tc::tc_fence_after();
      const uint32_t d_main = tmem_base + (uint32_t)(ab * 2 * a.npad), d_corr = d_main + (uint32_t)a.npad;
      for (int kb = 0; kb < KB; ++kb, ++consumed) {
        const int stage = consumed % S;
        if (!tc::mbar_wait(&full[stage], (uint32_t)((consumed / S) & 1), kWaitLimit)) { ok = false; break; }
        tc::tc_fence_after();
        const uint32_t ahi = tc::smem_u32(smem + (size_t)stage * a.stage_bytes), xhi = ahi + xoff;
#pragma unroll
        for (int ks = 0; ks < BKP / 16; ++ks) {
          // K-major: 16 k-columns = 32 bytes into the row
          uint64_t da[3], dx[3];
#pragma unroll
          for (int p = 0; p < 3; ++p) {
            da[p] = tc::smem_desc(ahi + p * kAP + ks * 32, 16, kSbo, kSw);
            dx[p] = tc::smem_desc(xhi + p * xbytes + ks * 32, 16, kSbo, kSw);
          }
          const uint32_t acc = kb > 0 || ks > 0 ? 1u : 0u;
          tc::mma_bf16(d_main, da[0], dx[0], a.idesc, acc);
          tc::mma_bf16(d_corr, da[0], dx[1], a.idesc, acc);
          tc::mma_bf16(d_corr, da[1], dx[0], a.idesc, 1u);
          tc::mma_bf16(d_corr, da[2], dx[0], a.idesc, 1u);
          tc::mma_bf16(d_corr, da[0], dx[2], a.idesc, 1u);
          tc::mma_bf16(d_corr, da[1], dx[1], a.idesc, 1u);
        }
        tc::mma_commit(&empty[stage]);
      }
      if (!ok) break;
      tc::mma_commit(&accf[ab]);
    }
    if (!ok) post_timeout(a.info);
    tc::mma_commit(done);   // no MMA in flight at teardown
    if (!tc::mbar_wait(done, 0, kWaitLimit)) post_timeout(a.info);
  } else if (warp < 4) {
    // ------------------------------------------------ epilogue: TMEM -> global
    const int row = warp * 32 + lane;
    for (int t = t0; t < t1; ++t) {
      const int seg = t - t0, ab = seg % a.nbuf;
      // One thread waits; the verdict is shared so the four warps stay in step.
      if (threadIdx.x == 0) *epi_ok = tc::mbar_wait(&accf[ab], (uint32_t)((seg / a.nbuf) & 1), kWaitLimit) ? 1 : 0;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (*epi_ok == 0) {
        if (threadIdx.x == 0) post_timeout(a.info);
        break;
      }
      tc::tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)(ab * 2 * a.npad);
      const long long gm = (long long)t * BM + row;
      float* dst = a.out + gm * a.ldo;
      const int ncols = gm < a.M ? a.d : 0;
      for (int c0 = 0; c0 < a.npad; c0 += 32) {   // (32 columns a step: their loads overlap)
        float v[2][16];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c0 + 16 * h;
          if (cc >= a.npad) continue;   // uniform across the warp
          float w[16];
          tc::tmem_ld16(taddr + (uint32_t)cc, v[h]);
          tc::tmem_ld16(taddr + (uint32_t)(a.npad + cc), w);
#pragma unroll
          for (int i = 0; i < 16; ++i) v[h][i] += w[i];
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c0 + 16 * h;
          if (cc >= a.npad) continue;
          if (a.vec_out != 0 && cc + 16 <= ncols) {
            float4* d4 = reinterpret_cast<float4*>(dst + cc);
#pragma unroll
            for (int q = 0; q < 4; ++q) d4[q] = make_float4(v[h][4 * q], v[h][4 * q + 1], v[h][4 * q + 2], v[h][4 * q + 3]);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (cc + i < ncols) dst[cc + i] = v[h][i];
          }
        }
      }
      tc::tc_fence_before();
      tc::mbar_arrive(&acce[ab]);
    }
  }

  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 5) tc::tmem_dealloc(tmem_base, a.tmem_cols);
}

// Gram matrix of a split tall matrix on the tensor cores: G = X^T X for
// X = X_hi + X_lo (rows x cols, cols <= 256), products hi^T hi + hi^T lo +
// lo^T hi in FP32. CTA c takes an even share of the rows; each stage holds
// one 32-row chunk of X as 64-column MN-major boxes (128B swizzle), which
// serves as the A operand (X^T, one or two 128-row tiles of G, one TMEM
// accumulator each) and as the B operand (X, N = round16(cols)). Each CTA
// writes its partial G to its own slot; tc_gram_reduce_kernel adds the slots
// in CTA order.
struct GramArgs {
  int rows, cols, npad, kblocks, G, stages, mtiles, nbox;
  float* part;               // G slots of (mtiles * 128) x npad floats
  int* info;
  uint32_t idesc, stage_bytes, tmem_cols;
};

__global__ void __launch_bounds__(kThreads, 1)
tc_gram_kernel(const __grid_constant__ CUtensorMap tmHi, const __grid_constant__ CUtensorMap tmLo,
               const GramArgs a) {
  grid_wait();
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = a.stages;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)S * a.stage_bytes);
  uint64_t* empty = full + S;
  uint64_t* accf = empty + S;
  uint64_t* done = accf + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  int* epi_ok = reinterpret_cast<int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cta = blockIdx.x;
  const long long kb0 = (long long)cta * a.kblocks / a.G, kb1 = (long long)(cta + 1) * a.kblocks / a.G;
  const uint32_t half = (uint32_t)a.nbox * 4096u;   // bytes of one (hi or lo) chunk

  if (threadIdx.x == 0) {
    for (int s2 = 0; s2 < S; ++s2) {
      tc::mbar_init(&full[s2], 1);
      tc::mbar_init(&empty[s2], 1);
    }
    tc::mbar_init(accf, 1);
    tc::mbar_init(done, 1);
    tc::fence_barrier_init();
  }
  if (warp == 5) {
    tc::tmem_alloc(tmem_slot, a.tmem_cols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 4 && lane == 0) {
    tc::prefetch_tmap(&tmHi);
    tc::prefetch_tmap(&tmLo);
    long long issued = 0;
    bool ok = true;
    for (long long kb = kb0; kb < kb1; ++kb, ++issued) {
      const int stage = (int)(issued % S);
      if (!tc::mbar_wait(&empty[stage], (uint32_t)((issued / S) & 1) ^ 1u, kWaitLimit)) { ok = false; break; }
      unsigned char* base = smem + (size_t)stage * a.stage_bytes;
      tc::mbar_expect_tx(&full[stage], 2 * half);
      for (int b = 0; b < a.nbox; ++b) {   // panel b, 32 rows
        tc::tma_load_3d(base + b * 4096, &tmHi, &full[stage], 0, (int)(kb * BK), b);
        tc::tma_load_3d(base + half + b * 4096, &tmLo, &full[stage], 0, (int)(kb * BK), b);
      }
    }
    if (!ok) post_timeout(a.info);
    for (long long i = issued > S ? issued - S : 0; i < issued; ++i)
      if (!tc::mbar_wait(&full[i % S], (uint32_t)((i / S) & 1), kWaitLimit)) post_timeout(a.info);
  } else if (warp == 5 && lane == 0) {
    long long consumed = 0;
    bool ok = true;
    for (long long kb = kb0; kb < kb1; ++kb, ++consumed) {
      const int stage = (int)(consumed % S);
      if (!tc::mbar_wait(&full[stage], (uint32_t)((consumed / S) & 1), kWaitLimit)) { ok = false; break; }
      tc::tc_fence_after();
      const uint32_t hi = tc::smem_u32(smem + (size_t)stage * a.stage_bytes), lo = hi + half;
#pragma unroll
      for (int ks = 0; ks < BK / 16; ++ks) {
        const uint32_t koff = ks * 2048;
        const uint64_t bh = tc::smem_desc(hi + koff, 4096, 1024, tc::kSwizzle128);
        const uint64_t bl = tc::smem_desc(lo + koff, 4096, 1024, tc::kSwizzle128);
        for (int mt = 0; mt < a.mtiles; ++mt) {
          const uint64_t ah = tc::smem_desc(hi + mt * 8192 + koff, 4096, 1024, tc::kSwizzle128);
          const uint64_t al = tc::smem_desc(lo + mt * 8192 + koff, 4096, 1024, tc::kSwizzle128);
          const uint32_t d_tmem = tmem_base + (uint32_t)(mt * a.npad);
          const uint32_t acc = (kb > kb0 || ks > 0) ? 1u : 0u;
          tc::mma_bf16(d_tmem, ah, bh, a.idesc, acc);
          tc::mma_bf16(d_tmem, ah, bl, a.idesc, 1u);
          tc::mma_bf16(d_tmem, al, bh, a.idesc, 1u);
        }
      }
      tc::mma_commit(&empty[stage]);
    }
    if (!ok) post_timeout(a.info);
    tc::mma_commit(accf);
    tc::mma_commit(done);
    if (!tc::mbar_wait(done, 0, kWaitLimit)) post_timeout(a.info);
  } else if (warp < 4) {
    if (threadIdx.x == 0) *epi_ok = tc::mbar_wait(accf, 0, kWaitLimit) ? 1 : 0;
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (*epi_ok == 0) {
      if (threadIdx.x == 0) post_timeout(a.info);
    } else {
      tc::tc_fence_after();
      const int row = warp * 32 + lane;
      for (int mt = 0; mt < a.mtiles; ++mt) {
        const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)(mt * a.npad);
        float* dst = a.part + ((long long)cta * a.mtiles * BM + mt * BM + row) * a.npad;
        for (int c0 = 0; c0 < a.npad; c0 += 16) {
          float v[16];
          tc::tmem_ld16(taddr + (uint32_t)c0, v);
          float4* d4 = reinterpret_cast<float4*>(dst + c0);
#pragma unroll
          for (int q = 0; q < 4; ++q) d4[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
      }
    }
  }

  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (warp == 5) tc::tmem_dealloc(tmem_base, a.tmem_cols);
}

// G[i][j] = sum over CTA slots of part (fixed order, Kahan-compensated FP32),
// for j <= i: the Cholesky reads the lower triangle only. Eight slots are
// loaded ahead of their adds, so a thread waits on about G / 8 round trips
// to L2 instead of G.
__global__ void tc_gram_reduce_kernel(const float* __restrict__ part, int G, int mtiles, int npad, int cols,
                                      float* __restrict__ out, long long ldo) {
  grid_wait();
  const long long slot = (long long)mtiles * BM * npad;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < cols * cols; e += gridDim.x * blockDim.x) {
    const int i = e / cols, j = e % cols;
    if (j > i) continue;
    const float* p = part + (long long)i * npad + j;
    float s = 0.f, c = 0.f;
    int z = 0;
    for (; z + 8 <= G; z += 8) {
      float v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcg(p + (long long)(z + u) * slot);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float y = v[u] - c, t = s + y;
        c = (t - s) - y;
        s = t;
      }
    }
    for (; z < G; ++z) {
      const float y = __ldcg(p + (long long)z * slot) - c, t = s + y;
      c = (t - s) - y;
      s = t;
    }
    out[(long long)i * ldo + j] = s;
  }
}

// A (m x n FP32) -> its three BF16 parts A_hi, A_lo, A_lo2 (the differences are exact
// in FP32), in 64-column panels: element (r, c) at ((c / 64) m + r) 64 + c % 64, columns
// n..npan*64-1 zero.
__global__ void split_a_kernel(const float* __restrict__ A, long long m, long long n, long long lda, bool vec,
                               bf16* __restrict__ hi, bf16* __restrict__ lo, bf16* __restrict__ lo2, long long npan) {
  grid_wait();
  const long long cpr = npan * 8, total = m * cpr;
  for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (long long)gridDim.x * blockDim.x) {
    const long long r = idx / cpr, c0 = (idx % cpr) * 8;
    const float* src = A + r * lda + c0;
    float x[8];
    if (vec && c0 + 8 <= n) {
      const float4 p = *reinterpret_cast<const float4*>(src);
      const float4 q = *reinterpret_cast<const float4*>(src + 4);
      x[0] = p.x; x[1] = p.y; x[2] = p.z; x[3] = p.w; x[4] = q.x; x[5] = q.y; x[6] = q.z; x[7] = q.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) x[i] = (c0 + i < n) ? src[i] : 0.f;
    }
    __align__(16) bf16 h[8];
    __align__(16) bf16 l[8];
    __align__(16) bf16 l2[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      h[i] = __float2bfloat16_rn(x[i]);
      const float r1 = x[i] - __bfloat162float(h[i]);
      l[i] = __float2bfloat16_rn(r1);
      l2[i] = __float2bfloat16_rn(r1 - __bfloat162float(l[i]));
    }
    const long long o = ((c0 >> 6) * m + r) * 64 + (c0 & 63);
    *reinterpret_cast<uint4*>(hi + o) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + o) = *reinterpret_cast<const uint4*>(l);
    *reinterpret_cast<uint4*>(lo2 + o) = *reinterpret_cast<const uint4*>(l2);
  }
}

// X (rows x d FP32) -> its three parts transposed (d x ldk BF16, K-major). A block of
// 32 x 8 threads transposes a 64 (K) x 32 (d) tile through shared memory; each thread
// then writes two consecutive K entries of a column as one 32-bit pair, so a warp
// stores 128 contiguous bytes of a row of X^T (ldk is a multiple of 8).
constexpr int kPrepRows = 64;
__global__ void prep_x_kernel(const float* __restrict__ X, long long rows, int d, long long ldx,
                              bf16* __restrict__ th, bf16* __restrict__ tl, bf16* __restrict__ tl2, long long ldk) {
  grid_wait();
  __shared__ float tile[kPrepRows][33];
  const long long r0 = (long long)blockIdx.x * kPrepRows;
  const int c0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < kPrepRows; i += blockDim.y) {
    const long long r = r0 + i;
    const int c = c0 + threadIdx.x;
    tile[i][threadIdx.x] = (r < rows && c < d) ? X[r * ldx + c] : 0.f;
  }
  __syncthreads();
  const long long r = r0 + 2 * threadIdx.x;   // this thread's pair of K entries
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i;
    if (c >= d || r >= ldk) continue;
    bf16 h[2], l[2], l2[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float x = tile[2 * threadIdx.x + e][i];
      h[e] = __float2bfloat16_rn(x);
      const float r1 = x - __bfloat162float(h[e]);
      l[e] = __float2bfloat16_rn(r1);
      l2[e] = __float2bfloat16_rn(r1 - __bfloat162float(l[e]));
    }
    const long long o = (long long)c * ldk + r;
    *reinterpret_cast<__nv_bfloat162*>(th + o) = __halves2bfloat162(h[0], h[1]);
    *reinterpret_cast<__nv_bfloat162*>(tl + o) = __halves2bfloat162(l[0], l[1]);
    *reinterpret_cast<__nv_bfloat162*>(tl2 + o) = __halves2bfloat162(l2[0], l2[1]);
  }
}

// ---------------------------------------------------------------- host side
// 2-D BF16 tensor map: dims {inner, outer}, row pitch in elements, box {bi, bo}.
bool make_map(CUtensorMap* map, const void* base, long long inner, long long outer, long long pitch, int bi,
              int bo, CUtensorMapSwizzle sw) {
  EncodeFn fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)outer};
  cuuint64_t strides[1] = {(cuuint64_t)(pitch * 2)};
  cuuint32_t box[2] = {(cuuint32_t)bi, (cuuint32_t)bo};
  cuuint32_t es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 3-D BF16 tensor map over the 64-column panel layout of m rows: dims {64,
// m, panels}, box {bi, bo, bp}.
bool make_panel_map(CUtensorMap* map, const void* base, long long m, long long panels, int bi, int bo, int bp,
                    CUtensorMapSwizzle sw) {
  EncodeFn fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[3] = {64, (cuuint64_t)m, (cuuint64_t)panels};
  cuuint64_t strides[2] = {128, (cuuint64_t)(m * 128)};
  cuuint32_t box[3] = {(cuuint32_t)bi, (cuuint32_t)bo, (cuuint32_t)bp};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int npad_of(int d) { return (int)round_up(std::max(d, 16), 16); }
uint32_t tmem_cols_of(int cols) {
  uint32_t c = 32;
  while (c < (uint32_t)cols) c <<= 1;
  return c;
}
uint32_t stage_bytes_of(int npad, int bkp) { return 3u * (uint32_t)(BM + npad) * bkp * 2; }

// Pipeline stages of a product (>= 1: at d = 256 and 64 of K one fits).
int stages_of(int npad, int bkp) {
  const size_t avail = smem_optin() - 1024 - 512;
  int s = (int)(avail / stage_bytes_of(npad, bkp));
  return std::max(1, std::min(kMaxStages, s));
}
int pass_bk(int npad) { return stages_of(npad, 64) >= 3 ? 64 : 32; }

template <int BKP>
cudaError_t launch_pass(const CUtensorMap& ah, const CUtensorMap& al, const CUtensorMap& xh,
                        const CUtensorMap& xl, const CUtensorMap& al2, const CUtensorMap& xl2, const TcArgs& a,
                        int ctas, cudaStream_t st) {
  const size_t smem = (size_t)a.stages * a.stage_bytes + 1024 + 512;
  static PerDevice<char> once;
  CK(allow_smem(&once, tc_pass_kernel<BKP>, smem_optin()));
  launch_pdl(tc_pass_kernel<BKP>, ctas, kThreads, smem, st, ah, al, xh, xl, al2, xl2, a);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

EncodeFn encode_fn() {
  static const EncodeFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<EncodeFn>(p);
  }();
  return fn;
}

bool tc_supported(const float* A, int64_t lda, const float* Omega, int64_t ldo) {
  (void)A; (void)lda; (void)Omega; (void)ldo;
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess)
    return false;
  return major == 10 && minor == 3 && encode_fn() != nullptr;
}

constexpr int kGramMaxCtas = 64;

void TcEngine::layout(Arena& ar, int64_t rows_cap, int cols_cap) {
  rows_cap_ = rows_cap;
  cols_cap_ = cols_cap;
  G_ = sm_count();
  const size_t panels = (size_t)(rows_cap * round_up(cols_cap, 64)), xt = (size_t)cols_cap * round_up(cols_cap, 8);
  Ahi_ = ar.take<uint16_t>(panels);
  Alo_ = ar.take<uint16_t>(panels);
  Alo2_ = ar.take<uint16_t>(panels);
  Xhi_ = ar.take<uint16_t>(xt);
  Xlo_ = ar.take<uint16_t>(xt);
  Xlo2_ = ar.take<uint16_t>(xt);
  gpart_ = ar.take<float>((size_t)kGramMaxCtas * cdiv(cols_cap, BM) * BM * npad_of(cols_cap));
}

cudaError_t TcEngine::split(const float* A, int64_t rows, int64_t cols, int64_t lda, cudaStream_t st) {
  if (rows > rows_cap_ || cols > cols_cap_) return cudaErrorInvalidValue;
  const bool vec = (reinterpret_cast<uintptr_t>(A) % 16 == 0) && (lda % 4 == 0);
  const long long npan = cdiv(cols, 64);
  const long long total = rows * npan * 8;
  const int blocks = (int)std::min<long long>(cdiv(total, 256), (long long)G_ * 8);
  launch_pdl(split_a_kernel, blocks, 256, 0, st, A, rows, cols, lda, vec, reinterpret_cast<bf16*>(Ahi_),
             reinterpret_cast<bf16*>(Alo_), reinterpret_cast<bf16*>(Alo2_), npan);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  split_of_ = A;
  m_ = rows;
  n_ = cols;
  return cudaSuccess;
}

cudaError_t TcEngine::product(const float* X, int64_t ldx, int d, float* out, int64_t ldout, int* info,
                              cudaStream_t st) {
  const int64_t m = m_, n = n_, K = n_;
  if (d > cols_cap_ || split_of_ == nullptr || K <= 0) return cudaErrorInvalidValue;
  cudaError_t e;
  const int npad_ = npad_of(d);
  {
    dim3 grid((unsigned)cdiv(round_up(K, 8), kPrepRows), (unsigned)cdiv(d, 32));
    launch_pdl(prep_x_kernel, grid, dim3(32, 8), 0, st, X, K, d, ldx, reinterpret_cast<bf16*>(Xhi_),
               reinterpret_cast<bf16*>(Xlo_), reinterpret_cast<bf16*>(Xlo2_), round_up(K, 8));
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  CUtensorMap ah, al, xh, xl, al2, xl2;
  const long long ldk = round_up(K, 8);
  bool ok;
  const long long npan = cdiv(n, 64);
  const int bkp = pass_bk(npad_);
  const CUtensorMapSwizzle ksw = bkp == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B;
  // K-major tiles, box bkp (j) x 128 (i), swizzle = the row
  ok = make_panel_map(&ah, Ahi_, m, npan, bkp, BM, 1, ksw) && make_panel_map(&al, Alo_, m, npan, bkp, BM, 1, ksw) &&
       make_panel_map(&al2, Alo2_, m, npan, bkp, BM, 1, ksw);
  ok = ok && make_map(&xh, Xhi_, K, d, ldk, bkp, npad_, ksw) &&
       make_map(&xl, Xlo_, K, d, ldk, bkp, npad_, ksw) &&
       make_map(&xl2, Xlo2_, K, d, ldk, bkp, npad_, ksw);
  if (!ok) return cudaErrorInvalidValue;

  TcArgs a;
  a.M = (int)m;
  a.d = d;
  a.npad = npad_;
  a.kblocks = (int)cdiv(K, bkp);
  a.tiles = (int)cdiv(m, BM);
  // K = d: split tiles would cost more in the epilogue than they save, so
  // each CTA takes whole tiles.
  a.tpc = (int)cdiv(a.tiles, G_);
  a.vec_out = ((reinterpret_cast<uintptr_t>(out) % 16) == 0 && ldout % 4 == 0) ? 1 : 0;
  // Two pairs of accumulators where they fit in tensor memory (npad <= 128); with one
  // the epilogue holds the MMAs for the drain of each tile.
  a.nbuf = 4 * npad_ <= 512 ? 2 : 1;
  a.stages = stages_of(npad_, bkp);
  a.out = out;
  a.ldo = ldout;
  a.info = info;
  a.idesc = tc::idesc_bf16(BM, npad_, false, false);
  a.stage_bytes = stage_bytes_of(npad_, bkp);
  a.tmem_cols = tmem_cols_of(a.nbuf * 2 * npad_);
  const int ctas = (int)cdiv(a.tiles, a.tpc);
  return bkp == 64 ? launch_pass<64>(ah, al, xh, xl, al2, xl2, a, ctas, st)
                   : launch_pass<32>(ah, al, xh, xl, al2, xl2, a, ctas, st);
}

cudaError_t TcEngine::gram(float* Gout, int64_t ldg, int* info, cudaStream_t st) {
  if (split_of_ == nullptr || n_ > 256) return cudaErrorInvalidValue;
  const int cols = (int)n_;
  const int npad = npad_of(cols);
  const int mtiles = (int)cdiv(cols, BM);
  GramArgs a;
  a.rows = (int)m_;
  a.cols = cols;
  a.npad = npad;
  a.kblocks = (int)cdiv(m_, BK);
  a.G = std::max(1, std::min({a.kblocks / 8, kGramMaxCtas, G_}));
  a.mtiles = mtiles;
  a.nbox = std::max((int)cdiv(npad, 64), 2 * mtiles);
  a.stage_bytes = 2u * (uint32_t)a.nbox * 4096u;
  a.stages = std::max(2, std::min(kMaxStages, (int)((smem_optin() - 1024 - 512) / a.stage_bytes)));
  a.part = gpart_;
  a.info = info;
  a.idesc = tc::idesc_bf16(BM, npad, true, true);
  {
    uint32_t need = (uint32_t)(mtiles * npad), c = 32;
    while (c < need) c <<= 1;
    a.tmem_cols = c;
  }
  CUtensorMap hi, lo;
  if (!make_panel_map(&hi, Ahi_, m_, cdiv(cols, 64), 64, BK, 1, CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_panel_map(&lo, Alo_, m_, cdiv(cols, 64), 64, BK, 1, CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  static PerDevice<char> once;
  CK(allow_smem(&once, tc_gram_kernel, smem_optin()));
  const size_t smem = (size_t)a.stages * a.stage_bytes + 1024 + 512;
  launch_pdl(tc_gram_kernel, a.G, kThreads, smem, st, hi, lo, a);
  note_launch();
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int blocks = std::max(1, std::min(G_ * 2, (cols * cols + 255) / 256));
  launch_pdl(tc_gram_reduce_kernel, blocks, 256, 0, st, gpart_, a.G, mtiles, npad, cols, Gout, ldg);
  note_launch();
  return cudaGetLastError();
}

}  // namespace rqlp
