// Grouped split products for the batched form: the passes over every problem's
// A of one step of the chain (Y = A^T X or Z = A X) in one launch, with the
// split of A and the arithmetic of split_gemm.cu.
//
// A work unit is one 256-row tile of one problem's output over that problem's
// whole K; the host balances the units over the CTA pairs (longest first, onto
// the least loaded pair), so no tile is split and no pair waits for another.
// A's FP32 tiles come by TMA through four maps per problem (its rows may start at
// any 4-byte address), X's parts through a fifth over the stage images that
// split_x_grouped_kernel writes before the pass. The earlier form kept A's
// parts in memory (a split of every A first, then 4 or 6 bytes per element and
// pass); reading A in FP32 takes 4 and no split. Every wait is bounded.
#include <algorithm>

#include "split_device.cuh"
#include "split_gemm.cuh"

namespace rqlp {
namespace {

using namespace sp;

constexpr int kGroupedCols = 4;   // 16-column groups of a drain warp: N <= 128

struct GroupArgs {
  const SplitJob* jobs;
  const int2* units;        // (job, tile)
  const int* cta_start;     // pair p takes units cta_start[p] .. cta_start[p + 1] - 1
  int* info;
  int npm;                  // largest npad: the layout of shared and tensor memory
  int sx, sf, sa, nbuf, corr, corr_first, chunk, flush, stall;
  float down;               // (see split_gemm.cu)
};

template <bool TRANS, int PARTS>
__global__ void __launch_bounds__(kThreads, 1) split_grouped_kernel(const GroupArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t stage_bytes = (uint32_t)PARTS * (a.npm / CG) * BK * 2;
  unsigned char* fstage = smem;
  unsigned char* xstage = smem + a.sf * kClassBytes;
  uint64_t* xfull = reinterpret_cast<uint64_t*>(xstage + (size_t)a.sx * stage_bytes);
  uint64_t* xempty = xfull + kMaxStages;
  uint64_t* ffull = xempty + kMaxStages;
  uint64_t* fempty = ffull + kMaxStages;
  uint64_t* afull = fempty + kMaxStages;
  uint64_t* aempty = afull + kMaxASlots;
  uint64_t* accf = aempty + kMaxASlots;
  uint64_t* acce = accf + 2;
  uint64_t* corre = acce + 2;
  uint64_t* done = corre + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform
  const int pair = (int)blockIdx.x / CG, rank = (int)blockIdx.x % CG;
  const int ub = a.cta_start[pair], ue = a.cta_start[pair + 1];
  if (ub >= ue) return;   // no units (the same for both CTAs)

  if (threadIdx.x == 0) {
    for (int s = 0; s < a.sx; ++s) {
      tc::mbar_init(&xfull[s], 1);
      tc::mbar_init(&xempty[s], 1);
    }
    for (int s = 0; s < a.sf; ++s) {
      tc::mbar_init(&ffull[s], 1);
      tc::mbar_init(&fempty[s], 4);
    }
    for (int s = 0; s < a.sa; ++s) {
      tc::mbar_init(&afull[s], 4 * CG);
      tc::mbar_init(&aempty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      tc::mbar_init(&accf[b], 1);
      tc::mbar_init(&acce[b], 8 * CG);
    }
    tc::mbar_init(corre, 8 * CG);
    tc::mbar_init(done, 1);
    tc::fence_barrier_init();
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(tc::smem_u32(tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc::tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t corr_base = tmem + (uint32_t)(a.nbuf * a.npm);
  const uint32_t a_base = corr_base + (a.corr ? (uint32_t)a.npm : 0u);
  const uint32_t smem_x = tc::smem_u32(xstage);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");   // 40 + 2 x 112 + 2 x 104 <= 5 x 96
    if (warp == 0) {
      // ------------------------------------------------ X stages
      const uint32_t xfull0 = leader_addr(xfull);
      bool ok = true;
      Ring r;
      int i = 0;
      for (int ui = ub; ui < ue && ok; ++ui) {
        const SplitJob& j = a.jobs[a.units[ui].x];
        const CUtensorMap* map = static_cast<const CUtensorMap*>(j.maps) + 4;
        const int kb = j.kb, nx = *j.xlo ? PARTS : 1, rows = j.npad / CG * BK / kImgRow;   // image rows of a part
        const uint32_t part = (uint32_t)rows * kImgRow * 2;
        for (int k = 0; k < kb; ++k, ++i) {
          if (!wait_warp(&xempty[r.s], r.ph ^ 1u)) {
            ok = false;
            break;
          }
          // Test hook: the first CTA withholds its first stage, so that the
          // waits on it run out and report.
          if (elect() && !(a.stall != 0 && blockIdx.x == 0 && i == 0)) {
            if (rank == 0) tc::mbar_expect_tx(&xfull[r.s], (uint32_t)(CG * nx) * part);
            for (int p = 0; p < nx; ++p)
              load_image(xstage + (size_t)r.s * stage_bytes + p * part, map, xfull0 + 8 * r.s,
                         ((k * CG + rank) * PARTS + p) * rows);
          }
          r.next(a.sx);
        }
      }
      if (!ok) post_timeout(a.info);
      // No copy in flight at exit (the leader's barriers count the peer's copies as well).
      for (int s = rank == 0 ? max(0, i - a.sx) : i; s < i; ++s)
        if (!wait(&xfull[s % a.sx], (uint32_t)((s / a.sx) & 1))) post_timeout(a.info);
    } else if (warp == 1) {
      // ------------------------------------------------ MMAs (the pair's leader)
      bool ok = true;
      if (rank == 0) {
        Ring rx, ra, rb;
        uint32_t cph = 0;   // (timeouts: see split_gemm.cu)
        for (int ui = ub; ui < ue; ++ui) {
          const SplitJob& j = a.jobs[a.units[ui].x];
          const uint32_t part = (uint32_t)(j.npad / CG) * BK * 2, idesc = j.idesc;
          const int nx = *j.xlo ? PARTS : 1;
          int left = j.kb;
          while (left > 0) {
            const int n = min(left, a.chunk);
            ok = ok && wait(&acce[rb.s], rb.ph ^ 1u) && (!a.corr || wait(corre, cph ^ 1u));
            const uint32_t d = tmem + (uint32_t)(rb.s * a.npm), dc = a.corr ? corr_base : d;
            uint32_t acc = 0, cacc = a.corr ? 0u : 1u;   // (with one accumulator the main product comes first)
            for (int i = 0; i < n; ++i) {
              ok = ok && wait(&xfull[rx.s], rx.ph) && wait(&afull[ra.s], ra.ph);
              tc::tc_fence_after();
              if (elect() && ok) {
                uint64_t x[PARTS];
#pragma unroll
                for (int p = 0; p < PARTS; ++p)
                  x[p] = tc::smem_desc(smem_x + (uint32_t)rx.s * stage_bytes + p * part, 16, 512, tc::kSwizzle64);
                issue_products<PARTS>(d, dc, a_base + (uint32_t)(ra.s * PARTS * 16), x, idesc, nx, a.corr_first != 0, acc,
                                      cacc);
                commit(&xempty[rx.s]);
                commit(&aempty[ra.s]);
              }
              acc = cacc = 1;
              rx.next(a.sx);
              ra.next(a.sa);
            }
            if (elect() && ok) commit(&accf[rb.s]);
            rb.next(a.nbuf);
            left -= n;
            if (a.corr) cph ^= 1u;   // drained with every chain
          }
        }
        if (elect()) commit(done);   // no MMA in flight at teardown
      }
      if (!ok) post_timeout(a.info);
      if (!wait(done, 0)) post_timeout(a.info);
    } else if (warp == 3) {
      // ------------------------------------------------ FP32 tiles of A
      bool ok = true;
      Ring r;
      int i = 0;
      for (int ui = ub; ui < ue && ok; ++ui) {
        const int2 un = a.units[ui];
        const SplitJob& j = a.jobs[un.x];
        const CUtensorMap* m = static_cast<const CUtensorMap*>(j.maps);
        Classes cl;
#pragma unroll
        for (int c = 0; c < 4; ++c) cl.past[c] = j.past[c];
        const int n = j.kb, row = (un.y * CG + rank) * BM;
        for (int k = 0; k < n; ++k, ++i) {
          if (!wait_warp(&fempty[r.s], r.ph ^ 1u)) {
            ok = false;
            break;
          }
          if (elect())
            load_classes<TRANS>(fstage + r.s * kClassBytes, m, m + 1, m + 2, m + 3, cl, &ffull[r.s], k * BK, row);
          r.next(a.sf);
        }
      }
      if (!ok) post_timeout(a.info);
      for (int s = max(0, i - a.sf); s < i; ++s)
        if (!wait(&ffull[s % a.sf], (uint32_t)((s / a.sf) & 1))) post_timeout(a.info);
    }
  } else if (warp < 12) {
    // -------------------------------------------------- A: split, store to tensor memory
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    const int w = warp & 3, odd = (warp >> 2) - 1;   // two warpgroups take the units of K by turns
    const uint32_t lanes = (uint32_t)(32 * w) << 16;
    bool ok = true;
    Ring ra, rf;
    if (odd) {
      ra.next(a.sa);
      rf.next(a.sf);
    }
    const uint32_t afull0 = leader_addr(afull);
    const bool scaled = PARTS == 3 && a.down != 1.f;
    int turn = odd;   // this warpgroup's first unit of K within the tile
    for (int ui = ub; ui < ue && ok; ++ui) {
      const SplitJob& j = a.jobs[a.units[ui].x];
      const bool sq = j.sumsq != nullptr;
      Squares sum;
      Classes cl;
#pragma unroll
      for (int c = 0; c < 4; ++c) cl.shift[c] = j.shift[c];
      const int n = j.kb;
      for (int k = turn; k < n; k += 2) {
        const unsigned char* f = fstage + rf.s * kClassBytes;
        ok = wait_warp(&ffull[rf.s], rf.ph);
        if (!ok) break;
        float v[16];
        uint32_t o[PARTS][8];
        read_classes<TRANS>(f, cl, w, 0, lane, v);
        ok = wait_warp(&aempty[ra.s], ra.ph ^ 1u);
        if (!ok) break;
        tc::tc_fence_after();
        split_half<PARTS>(v, o, scaled, sq, sum);
        read_classes<TRANS>(f, cl, w, 1, lane, v);
        const uint32_t ta = a_base + lanes + (uint32_t)(ra.s * PARTS * 16);
#pragma unroll
        for (int q = 0; q < PARTS; ++q) st_row8(ta + q * 16, o[q]);
        split_half<PARTS>(v, o, scaled, sq, sum);
        arrive_read(&fempty[rf.s], lane);
#pragma unroll
        for (int q = 0; q < PARTS; ++q) st_row8(ta + q * 16 + 8, o[q]);
        if (sq) sum.fold();
        st_wait();
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) arrive_remote(afull0 + 8 * ra.s);
        ra.next(a.sa);
        ra.next(a.sa);
        rf.next(a.sf);
        rf.next(a.sf);
      }
      if (n & 1) turn ^= 1;   // the other warpgroup begins the next tile
      if (sq) sum.add(j.sumsq, lane);
    }
    if (!ok && lane == 0) post_timeout(a.info);
  } else {
    // -------------------------------------------------- drain: TMEM -> registers -> global
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    const int e = warp - 12, half = e >> 2;
    const uint32_t lanes = (uint32_t)(32 * (e & 3)) << 16;
    float s[kGroupedCols][16];
    bool ok = true;   // after a timeout the loop runs on without waiting
    Ring rb;
    for (int ui = ub; ui < ue; ++ui) {
      const int2 un = a.units[ui];
      const SplitJob& j = a.jobs[un.x];
      const int groups = j.npad / 16, g0 = half ? (groups + 1) / 2 : 0, ng = half ? groups / 2 : (groups + 1) / 2;
      // (TMEM lane -> row: see read_classes)
      const long long gm = (long long)(un.y * CG + rank) * BM + (TRANS ? 32 * (e & 3) + lane : 4 * lane + (e & 3));
      float* dst = j.out + gm * j.ldo;
      const int ncols = gm < j.M ? j.N : 0;
      clear_sums(s);
      bool flushed = false;
      int left = j.kb, since = 0;
      while (left > 0) {
        const int n = min(left, a.chunk);
        if (ok && !wait_warp(&accf[rb.s], rb.ph)) {
          ok = false;
          if (lane == 0) post_timeout(a.info);
        }
        if (ok) {
          tc::tc_fence_after();
          drain_columns(s, tmem + lanes + (uint32_t)(rb.s * a.npm + 16 * g0), ng, a.down);
          if (lane == 0) arrive_leader(&acce[rb.s]);
          if (a.corr) {
            drain_columns(s, corr_base + lanes + (uint32_t)(16 * g0), ng, a.down);
            if (lane == 0) arrive_leader(corre);
          }
        }
        rb.next(a.nbuf);
        left -= n;
        since += n;
        if (left > 0 && since < a.flush) continue;
        if (!ok) lose_sums(s);
        if (PARTS == 3 && j.bad != nullptr) check_sums(s, g0, ng, ncols, j.bad);
        store_sums(s, dst, 4, g0, ng, ncols, j.vec_out != 0, flushed);
        clear_sums(s);
        flushed = true;
        since = 0;
      }
    }
  }

  tc::tc_fence_before();
  __syncthreads();
  cluster_sync();   // no remote arrival is still on its way
  tc::tc_fence_after();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// Block -> problem: the last b with start[b] <= blk (start has count + 1 entries).
__device__ __forceinline__ int problem_of(const int* __restrict__ start, int count, int blk) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (start[mid] <= blk) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(256)
split_x_grouped_kernel(const SplitXJob* __restrict__ jobs, const int* __restrict__ start, int count, int parts, bool scaled) {
  const int b = problem_of(start, count, blockIdx.x);
  const SplitXJob j = jobs[b];
  const int local = (int)blockIdx.x - start[b], kt = (int)cdiv(j.K, 64);
  split_x_tile(j.X, j.K, j.N, j.ldx, j.img, j.npad, parts, (int)cdiv(j.K, BK), (long long)(local % kt) * 64,
               local / kt * 32, j.xlo, scaled);
}

template <bool TRANS, int PARTS>
cudaError_t launch(const GroupArgs& a, int pairs, size_t smem, cudaStream_t st) {
  static PerDevice<char> once;
  CK(allow_smem(&once, split_grouped_kernel<TRANS, PARTS>, smem_optin()));
  if (pairs <= 0) return cudaSuccess;   // configuration only
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CG;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)(pairs * CG));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, split_grouped_kernel<TRANS, PARTS>, a);
  note_launch();
  return e;
}

}  // namespace

int split_npad(int n) { return (int)round_up(n, 16); }
size_t split_image_bytes(int64_t K, int n, int parts) { return (size_t)round_up(K, BK) * split_npad(n) * parts * 2; }
uint32_t split_idesc(int npad) { return tc::idesc_bf16(BM * CG, npad, false, false); }
bool split_job_maps(void* maps, SplitJob* j, const float* A, int64_t rows, int64_t cols, int64_t lda, bool trans,
                    const uint16_t* img, int parts) {
  Classes cl;
  CUtensorMap* m = static_cast<CUtensorMap*>(maps);
  if (!class_maps(m, &cl, A, rows, cols, lda, trans) || !image_map(m + 4, img, j->kb, j->npad, parts)) return false;
  for (int c = 0; c < 4; ++c) {
    j->shift[c] = cl.shift[c];
    j->past[c] = cl.past[c];
  }
  return true;
}
int split_x_blocks(int64_t K, int npad) { return (int)(cdiv(K, 64) * cdiv(npad, 32)); }

cudaError_t split_x_grouped(const SplitXJob* jobs, const int* start, int count, int total, SplitMode mode,
                            cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  split_x_grouped_kernel<<<total, 256, 0, st>>>(jobs, start, count, mode == kSplitTwo ? 2 : 3, mode == kSplitFp32);
  note_launch();
  return cudaGetLastError();
}

cudaError_t split_grouped(bool transA, const SplitJob* jobs, const int2* units, const int* cta_start, int pairs,
                          int npad_max, SplitMode mode, int* info, int stall, cudaStream_t st) {
  const int parts = mode == kSplitTwo ? 2 : 3;
  GroupArgs a = {};
  a.jobs = jobs;
  a.units = units;
  a.cta_start = cta_start;
  a.info = info;
  a.npm = std::max(npad_max, 16);
  a.stall = stall;
  a.down = mode == kSplitFp32 ? kScaleDown : 1.f;
  a.corr = mode == kSplitFp32 ? 0 : 1;
  a.corr_first = mode == kSplitFp32 ? 1 : 0;
  a.chunk = mode == kSplitFp32 ? 1 : kChainBatch;
  a.flush = mode == kSplitFp32 ? 64 : 1 << 30;
  const int cc = a.corr ? a.npm : 0;
  a.nbuf = 2 * a.npm + cc + 2 * parts * 16 <= 512 ? 2 : 1;
  a.sa = std::min(kMaxASlots, (512 - a.nbuf * a.npm - cc) / (parts * 16));
  const size_t stage = (size_t)parts * (a.npm / CG) * BK * 2, extra = 2048;
  const size_t avail = smem_optin() - extra;
  a.sf = (int)std::min<size_t>(kMaxStages, (avail - 4 * stage) / kClassBytes);
  a.sx = (int)std::min<size_t>(kMaxStages, (avail - a.sf * kClassBytes) / stage);
  if (a.sa < 2) return cudaErrorInvalidValue;
  const size_t smem = a.sf * kClassBytes + a.sx * stage + extra;
  if (transA) return parts == 3 ? launch<true, 3>(a, pairs, smem, st) : launch<true, 2>(a, pairs, smem, st);
  return parts == 3 ? launch<false, 3>(a, pairs, smem, st) : launch<false, 2>(a, pairs, smem, st);
}

}  // namespace rqlp
