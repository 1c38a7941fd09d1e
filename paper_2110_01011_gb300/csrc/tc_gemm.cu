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
#include <mutex>

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
// K per pipeline stage of a pass: 64 (128-byte rows, 128B swizzle) where at
// least three such stages fit in shared memory, else 32 (64-byte rows, 64B
// swizzle). Larger TMA boxes stream A faster (measured: 7.1 vs 5.2 TB/s of
// A_hi + A_lo in the A^T X order at d = 64), but the pipeline needs stages in
// flight: at d = 224 only two K = 64 stages fit, and K = 32 with five is as fast.
// The FP32 accumulation of tcgen05.mma in TMEM loses a little of every add in
// the same direction: over K = 20000 a pass shrinks by ~1.5e-6 relative to
// its partial sums, which the cancelling small-singular-value columns of
// A P~ turn into ~1e-4 of their own size (and into the leading diagonal of
// L). Accumulation chains in TMEM are therefore cut every kChunkK of K
// (K = 4096); the epilogue adds the chunks in FP32 with round-to-nearest.
// The error falls linearly with the chunk (leading diagonal of L on the
// 20000^2 class: 4.2e-5, 2.1e-5, 9.4e-6 at K = 8192, 4096, 2048) and the time
// rises ~3% per halving.
constexpr int kChunkK = 4096;

struct TcArgs {
  int M, K, d, npad, kblocks, tiles, G, stages;
  int tpc;                   // whole tiles per CTA
  int vec_out;               // out rows are 16-byte aligned (float4 stores)
  float* out;
  long long ldo;
  const int* xlo_nonzero;    // 1 when X has a nonzero low part
  int exact;                 // 1: A and X in three parts, six products
  int chunk;                 // k-blocks per accumulation chain in TMEM
  int split_acc;             // 1: correction products in their own accumulator
  int nbuf;                  // accumulator buffers (2: the epilogue overlaps the next chain)
  int bufcols;               // TMEM columns of one buffer (npad, or 2 npad when split_acc)
  int* info;                 // status word (may be null)
  uint32_t idesc, stage_bytes, tmem_cols;
};

// First unit of CTA c: tpc whole tiles of kblocks units each.
__device__ inline long long cta_begin(int c, int tpc, int tiles, int kblocks) {
  return (long long)min(c * tpc, tiles) * kblocks;
}

// End of the accumulation chunk that starts at unit u (a CTA's range [.., u1)).
__device__ inline long long chunk_end(long long u, long long u1, int KB, int chunk) {
  const long long t_end = (u / KB + 1) * (long long)KB;
  return min(min(u1, t_end), u + chunk);
}

__device__ void post_timeout(int* info) {
  if (info != nullptr && atomicCAS(info, 0, RQLP_ERR_TIMEOUT) == 0) info[1] = 0;
}

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
  const int cta = blockIdx.x;
  const long long u0 = cta_begin(cta, a.tpc, a.tiles, a.kblocks);
  const long long u1 = cta_begin(cta + 1, a.tpc, a.tiles, a.kblocks);
  if (u0 >= u1) return;   // no work for this CTA (uniform)
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
  // Stage layout: A_hi, A_lo[, A_lo2], X_hi[, X_lo[, X_lo2]].
  const bool ex = a.exact != 0;
  const int nx = ex ? 3 : ((*a.xlo_nonzero) ? 2 : 1);
  constexpr uint32_t kAP = BM * BKP * 2;   // one BF16 A tile
  const int kChunk = a.chunk;
  constexpr uint32_t kRow = BKP * 2;        // bytes of a K-major row: the swizzle span
  constexpr uint32_t kSbo = 8 * kRow;       // 8-row swizzle atom of the K-major operands
  constexpr uint32_t kSw = BKP == 64 ? tc::kSwizzle128 : tc::kSwizzle64;
  const uint32_t xbytes = (uint32_t)a.npad * BKP * 2;
  const uint32_t xoff = (ex ? 3u : 2u) * kAP;

  if (warp == 4 && lane == 0) {
    // ------------------------------------------------ TMA producer
    tc::prefetch_tmap(&tmAhi);
    tc::prefetch_tmap(&tmAlo);
    tc::prefetch_tmap(&tmXhi);
    tc::prefetch_tmap(&tmXlo);
    if (ex) {
      tc::prefetch_tmap(&tmAlo2);
      tc::prefetch_tmap(&tmXlo2);
    }
    long long issued = 0;
    bool ok = true;
    for (long long u = u0; u < u1; ++u, ++issued) {
      const int stage = (int)(issued % S);
      const uint32_t par = (uint32_t)((issued / S) & 1);
      if (!tc::mbar_wait(&empty[stage], par ^ 1u, kWaitLimit)) { ok = false; break; }
      const int t = (int)(u / KB), kb = (int)(u % KB);
      unsigned char* base = smem + (size_t)stage * a.stage_bytes;
      tc::mbar_expect_tx(&full[stage], xoff + (uint32_t)nx * xbytes);
      // A maps are 3-D over the panel layout: {column in panel, row, panel}.
      // 128 rows (M) x BKP columns (K) of panel kb BKP / 64
      const int kx = (kb * BKP) & 63, kp = (kb * BKP) >> 6, mr = t * BM;
      tc::tma_load_3d(base, &tmAhi, &full[stage], kx, mr, kp);
      tc::tma_load_3d(base + kAP, &tmAlo, &full[stage], kx, mr, kp);
      if (ex) tc::tma_load_3d(base + 2 * kAP, &tmAlo2, &full[stage], kx, mr, kp);
      tc::tma_load_2d(base + xoff, &tmXhi, &full[stage], kb * BKP, 0);
      if (nx >= 2) tc::tma_load_2d(base + xoff + xbytes, &tmXlo, &full[stage], kb * BKP, 0);
      if (nx == 3) tc::tma_load_2d(base + xoff + 2 * xbytes, &tmXlo2, &full[stage], kb * BKP, 0);
    }
    if (!ok) post_timeout(a.info);
    // Drain: every load this thread started has landed before the CTA exits.
    for (long long i = issued > S ? issued - S : 0; i < issued; ++i)
      if (!tc::mbar_wait(&full[i % S], (uint32_t)((i / S) & 1), kWaitLimit)) post_timeout(a.info);
  } else if (warp == 5 && lane == 0) {
    // ------------------------------------------------ MMA issuer
    long long consumed = 0;
    int seg = 0;
    bool ok = true;
    long long u = u0;
    while (u < u1 && ok) {
      const long long seg_begin = u, seg_end = chunk_end(u, u1, KB, kChunk);
      const int ab = seg % a.nbuf;
      if (!tc::mbar_wait(&acce[ab], (uint32_t)(((seg / a.nbuf) & 1) ^ 1), kWaitLimit)) { ok = false; break; }
      tc::tc_fence_after();
      const uint32_t d_tmem = tmem_base + (uint32_t)(ab * a.bufcols);
      // The products of the low parts are ~2^-8 of A_hi X_hi or smaller. Added
      // into the same FP32 accumulator they lose bits to its large magnitude
      // at every MMA; with split_acc they accumulate on their own and the
      // epilogue adds the two sums with round-to-nearest.
      const uint32_t d_corr = a.split_acc ? d_tmem + (uint32_t)a.npad : d_tmem;
      for (; u < seg_end; ++u, ++consumed) {
        const int stage = (int)(consumed % S);
        if (!tc::mbar_wait(&full[stage], (uint32_t)((consumed / S) & 1), kWaitLimit)) { ok = false; break; }
        tc::tc_fence_after();
        const uint32_t base = tc::smem_u32(smem + (size_t)stage * a.stage_bytes);
        const uint32_t ahi = base, alo = base + kAP, alo2 = base + 2 * kAP, xhi = base + xoff,
                       xlo = xhi + xbytes, xlo2 = xlo + xbytes;
#pragma unroll
        for (int ks = 0; ks < BKP / 16; ++ks) {
          uint64_t dah, dal, dal2;
          // K-major: 16 k-columns = 32 bytes into the row
          dah = tc::smem_desc(ahi + ks * 32, 16, kSbo, kSw);
          dal = tc::smem_desc(alo + ks * 32, 16, kSbo, kSw);
          dal2 = tc::smem_desc(alo2 + ks * 32, 16, kSbo, kSw);
          const uint64_t dxh = tc::smem_desc(xhi + ks * 32, 16, kSbo, kSw);
          const uint64_t dxl = tc::smem_desc(xlo + ks * 32, 16, kSbo, kSw);
          const uint64_t dxl2 = tc::smem_desc(xlo2 + ks * 32, 16, kSbo, kSw);
          const uint32_t acc = (u > seg_begin || ks > 0) ? 1u : 0u;
          // the first correction product of a chain starts d_corr when it is separate
          const uint32_t acc_c = a.split_acc ? acc : 1u;
          tc::mma_bf16(d_tmem, dah, dxh, a.idesc, acc);
          if (nx >= 2) {
            tc::mma_bf16(d_corr, dah, dxl, a.idesc, acc_c);
            tc::mma_bf16(d_corr, dal, dxh, a.idesc, 1u);
          } else {
            tc::mma_bf16(d_corr, dal, dxh, a.idesc, acc_c);
          }
          if (ex) {
            tc::mma_bf16(d_corr, dal2, dxh, a.idesc, 1u);
            tc::mma_bf16(d_corr, dah, dxl2, a.idesc, 1u);
            tc::mma_bf16(d_corr, dal, dxl, a.idesc, 1u);
          }
        }
        tc::mma_commit(&empty[stage]);
      }
      if (!ok) break;
      tc::mma_commit(&accf[ab]);
      ++seg;
    }
    if (!ok) post_timeout(a.info);
    tc::mma_commit(done);   // no MMA in flight at teardown
    if (!tc::mbar_wait(done, 0, kWaitLimit)) post_timeout(a.info);
  } else if (warp < 4) {
    // ------------------------------------------------ epilogue: TMEM -> global
    const int row = warp * 32 + lane;
    int seg = 0;
    long long u = u0;
    while (u < u1) {
      const int t = (int)(u / KB);
      const long long seg_begin = u, seg_end = chunk_end(u, u1, KB, kChunk);
      const long long tb = (long long)t * KB;
      const bool first_chunk = seg_begin == tb;
      const int ab = seg % a.nbuf;
      // One thread waits; the verdict is shared so the four warps stay in step.
      if (threadIdx.x == 0) *epi_ok = tc::mbar_wait(&accf[ab], (uint32_t)((seg / a.nbuf) & 1), kWaitLimit) ? 1 : 0;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (*epi_ok == 0) {
        if (threadIdx.x == 0) post_timeout(a.info);
        break;
      }
      tc::tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(warp * 32) << 16) + (uint32_t)(ab * a.bufcols);
      const long long gm = (long long)t * BM + row;
      float* dst;
      int ncols;
      dst = a.out + gm * a.ldo;
      ncols = gm < a.M ? a.d : 0;
      const bool vec = a.vec_out != 0;
      // 32 columns per step: the row's earlier sums (this thread wrote them)
      // are all loaded before the step's stores, so the loads of a step
      // overlap instead of queueing behind stores to the same array.
      for (int c0 = 0; c0 < a.npad; c0 += 32) {
        float v[2][16];
        float4 o[2][4];
        float os[2][16];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c0 + 16 * h;
          if (cc >= a.npad || first_chunk) continue;
          if (vec && cc + 16 <= ncols) {
            const float4* d4 = reinterpret_cast<const float4*>(dst + cc);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[h][q] = d4[q];
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i) os[h][i] = cc + i < ncols ? dst[cc + i] : 0.f;
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c0 + 16 * h;
          if (cc >= a.npad) continue;   // uniform across the warp
          tc::tmem_ld16(taddr + (uint32_t)cc, v[h]);
          if (a.split_acc) {
            float w[16];
            tc::tmem_ld16(taddr + (uint32_t)(a.npad + cc), w);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[h][i] += w[i];
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int cc = c0 + 16 * h;
          if (cc >= a.npad) continue;
          float* vv = v[h];
          if (vec && cc + 16 <= ncols) {
            float4* d4 = reinterpret_cast<float4*>(dst + cc);
            if (!first_chunk) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                vv[4 * q] += o[h][q].x; vv[4 * q + 1] += o[h][q].y;
                vv[4 * q + 2] += o[h][q].z; vv[4 * q + 3] += o[h][q].w;
              }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) d4[q] = make_float4(vv[4 * q], vv[4 * q + 1], vv[4 * q + 2], vv[4 * q + 3]);
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (cc + i < ncols) dst[cc + i] = first_chunk ? vv[i] : os[h][i] + vv[i];
          }
        }
      }
      tc::tc_fence_before();
      tc::mbar_arrive(&acce[ab]);
      u = seg_end;
      ++seg;
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

// A (m x n FP32) -> A_hi, A_lo (BF16) and ||A||_F^2, in 64-column panels:
// element (r, c) at ((c / 64) m + r) 64 + c % 64, columns n..npan*64-1 zero.
// lo2 (optional) receives bf16(A - A_hi - A_lo); both differences are exact in FP32.
// Rows row0 .. row0 + m - 1 of a matrix of mstride rows (the panel height).
__global__ void split_a_kernel(const float* __restrict__ A, long long m, long long n, long long lda, bool vec,
                               bf16* __restrict__ hi, bf16* __restrict__ lo, bf16* __restrict__ lo2, long long npan,
                               double* sumsq, long long mstride, long long row0) {
  grid_wait();
  const long long cpr = npan * 8, total = m * cpr;
  float s = 0.f, comp = 0.f;
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
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      h[i] = __float2bfloat16_rn(x[i]);
      const float r1 = x[i] - __bfloat162float(h[i]);
      l[i] = __float2bfloat16_rn(r1);
      l2[i] = __float2bfloat16_rn(r1 - __bfloat162float(l[i]));
      ss = fmaf(x[i], x[i], ss);
    }
    const long long o = ((c0 >> 6) * mstride + row0 + r) * 64 + (c0 & 63);
    *reinterpret_cast<uint4*>(hi + o) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + o) = *reinterpret_cast<const uint4*>(l);
    if (lo2 != nullptr) *reinterpret_cast<uint4*>(lo2 + o) = *reinterpret_cast<const uint4*>(l2);
    const float y = ss - comp, tt = s + y;
    comp = (tt - s) - y;
    s = tt;
  }
  if (sumsq == nullptr) return;
  __shared__ double red[32];
  double v = (double)s - (double)comp;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    atomicAdd(sumsq, t);
  }
}

// X (rows x d FP32) -> X_hi^T, X_lo^T (d x ldk BF16, K-major); flags a nonzero low part.
// tl2 (optional) receives bf16(X - X_hi - X_lo). A block of 32 x 8 threads
// transposes a 64 (K) x 32 (d) tile through shared memory; each thread then
// writes two consecutive K entries of a column as one 32-bit pair, so a warp
// stores 128 contiguous bytes of a row of X^T (ldk is a multiple of 8).
constexpr int kPrepRows = 64;
__global__ void prep_x_kernel(const float* __restrict__ X, long long rows, int d, long long ldx,
                              bf16* __restrict__ th, bf16* __restrict__ tl, bf16* __restrict__ tl2, long long ldk,
                              int* nonzero_lo) {
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
  bool any = false;
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
      any |= __bfloat162float(l[e]) != 0.f;
    }
    const long long o = (long long)c * ldk + r;
    *reinterpret_cast<__nv_bfloat162*>(th + o) = __halves2bfloat162(h[0], h[1]);
    *reinterpret_cast<__nv_bfloat162*>(tl + o) = __halves2bfloat162(l[0], l[1]);
    if (tl2 != nullptr) *reinterpret_cast<__nv_bfloat162*>(tl2 + o) = __halves2bfloat162(l2[0], l2[1]);
  }
  // One vote per block, and none once another block has raised the flag.
  if (__syncthreads_or(any) && threadIdx.x == 0 && threadIdx.y == 0 && *(volatile int*)nonzero_lo == 0)
    atomicOr(nonzero_lo, 1);
}

// ---------------------------------------------------------------- host side
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
  });
  return fn;
}

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
uint32_t stage_bytes_of(int npad, bool exact, int bkp) {
  return (exact ? 3u : 2u) * (uint32_t)(BM * bkp * 2) + (exact ? 3u : 2u) * (uint32_t)npad * bkp * 2;
}

// Pipeline stages of a pass (>= 1; the exact mode's stages at d = 256 hold
// one at a time, which its short K does not need more than).
int stages_of(int npad, bool exact, int bkp) {
  const size_t avail = smem_optin() - 1024 - 512;
  int s = (int)(avail / stage_bytes_of(npad, exact, bkp));
  return std::max(1, std::min(kMaxStages, s));
}
int pass_bk(int npad, bool exact) { return stages_of(npad, exact, 64) >= 3 ? 64 : 32; }

template <int BKP>
cudaError_t launch_pass(const CUtensorMap& ah, const CUtensorMap& al, const CUtensorMap& xh,
                        const CUtensorMap& xl, const CUtensorMap& al2, const CUtensorMap& xl2, const TcArgs& a,
                        cudaStream_t st) {
  const size_t smem = (size_t)a.stages * a.stage_bytes + 1024 + 512;
  static PerDevice<char> once;
  CK(allow_smem(&once, tc_pass_kernel<BKP>, smem_optin()));
  launch_pdl(tc_pass_kernel<BKP>, a.G, kThreads, smem, st, ah, al, xh, xl, al2, xl2, a);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

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

void TcEngine::layout(Arena& ar, int64_t rows_cap, int64_t cols_cap, int d_cap, int64_t k_cap, bool gram,
                      bool three_part) {
  rows_cap_ = rows_cap;
  cols_cap_ = cols_cap;
  d_cap_ = d_cap;
  k_cap_ = k_cap;
  ldb_ = round_up(cols_cap, 64);   // whole 64-column panels
  G_ = sm_count();
  Ahi_ = ar.take<uint16_t>((size_t)(rows_cap * ldb_));
  Alo_ = ar.take<uint16_t>((size_t)(rows_cap * ldb_));
  Alo2_ = three_part ? ar.take<uint16_t>((size_t)(rows_cap * ldb_)) : nullptr;
  Xhi_ = ar.take<uint16_t>((size_t)d_cap * round_up(k_cap, 8));
  Xlo_ = ar.take<uint16_t>((size_t)d_cap * round_up(k_cap, 8));
  Xlo2_ = three_part ? ar.take<uint16_t>((size_t)d_cap * round_up(k_cap, 8)) : nullptr;
  flag_ = ar.take<int>(4);
  if (gram) {
    const int gp = npad_of((int)cols_cap);
    gpart_ = ar.take<float>((size_t)kGramMaxCtas * cdiv(cols_cap, BM) * BM * gp);
  }
}

cudaError_t TcEngine::split(const float* A, int64_t rows, int64_t cols, int64_t lda, double* sumsq,
                            cudaStream_t st) {
  if (rows > rows_cap_ || cols > cols_cap_) return cudaErrorInvalidValue;
  const bool vec = (reinterpret_cast<uintptr_t>(A) % 16 == 0) && (lda % 4 == 0);
  const long long npan = cdiv(cols, 64);
  const long long total = rows * npan * 8;
  const int blocks = (int)std::min<long long>(cdiv(total, 256), (long long)G_ * 8);
  launch_pdl(split_a_kernel, blocks, 256, 0, st, A, rows, cols, lda, vec, reinterpret_cast<bf16*>(Ahi_),
             reinterpret_cast<bf16*>(Alo_), reinterpret_cast<bf16*>(Alo2_), npan, sumsq, rows, 0);
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
  if (d > d_cap_ || split_of_ == nullptr || Alo2_ == nullptr || K <= 0 || K > k_cap_) return cudaErrorInvalidValue;
  cudaError_t e;
  const int npad_ = npad_of(d);
  if ((e = cudaMemsetAsync(flag_, 0, sizeof(int), st)) != cudaSuccess) return e;
  {
    dim3 grid((unsigned)cdiv(round_up(K, 8), kPrepRows), (unsigned)cdiv(d, 32));
    launch_pdl(prep_x_kernel, grid, dim3(32, 8), 0, st, X, K, d, ldx, reinterpret_cast<bf16*>(Xhi_),
               reinterpret_cast<bf16*>(Xlo_), reinterpret_cast<bf16*>(Xlo2_), round_up(K, 8), flag_);
    note_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  CUtensorMap ah, al, xh, xl, al2, xl2;
  const long long ldk = round_up(K, 8);
  bool ok;
  const long long npan = cdiv(n, 64);
  const int bkp = pass_bk(npad_, true);
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
  a.K = (int)K;
  a.d = d;
  a.npad = npad_;
  a.kblocks = (int)cdiv(K, bkp);
  a.tiles = (int)cdiv(m, BM);
  // K = d: split tiles would cost more in the epilogue than they save, so
  // each CTA takes whole tiles.
  a.tpc = (int)cdiv(a.tiles, G_);
  a.G = (int)cdiv(a.tiles, a.tpc);
  a.vec_out = ((reinterpret_cast<uintptr_t>(out) % 16) == 0 && ldout % 4 == 0) ? 1 : 0;
  a.exact = 1;
  a.chunk = kChunkK / bkp;
  // Correction products get their own accumulator where two such buffer
  // pairs fit in TMEM's 512 columns (npad <= 128), and always in exact mode
  // (single-buffered above npad = 128: the epilogue then holds the MMAs for
  // the drain of each chain).
  a.split_acc = 1;
  a.bufcols = (a.split_acc ? 2 : 1) * npad_;
  a.nbuf = 2 * a.bufcols <= 512 ? 2 : 1;
  a.stages = stages_of(npad_, true, bkp);
  a.out = out;
  a.ldo = ldout;
  a.xlo_nonzero = flag_;
  a.info = info;
  a.idesc = tc::idesc_bf16(BM, npad_, false, false);
  a.stage_bytes = stage_bytes_of(npad_, true, bkp);
  a.tmem_cols = tmem_cols_of(a.nbuf * a.bufcols);
  return bkp == 64 ? launch_pass<64>(ah, al, xh, xl, al2, xl2, a, st)
                   : launch_pass<32>(ah, al, xh, xl, al2, xl2, a, st);
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
