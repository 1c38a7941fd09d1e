// out = op(A) X (N <= 256 columns) on the tensor cores, with A read once in
// FP32 and split into BF16 parts inside the kernel.
//
// A = A_1 + A_2 [+ A_3] and X likewise, each part the BF16 rounding of what
// the earlier ones leave. Two parts: A_1 X_1 + A_1 X_2 + A_2 X_1 (the BF16x3
// form, products above 2^-16). Three parts hold all 24 bits of an FP32 value; of
// their nine products the six above 2^-24 are taken. In FP32 (chains of one unit)
// a result is off by 1.5e-7 of its norm on average where FMAs in two levels of
// sums leave 2.9e-7 (10007 x 6001 and 16384 x 12288); 4.5e-8 of it is a loss
// toward zero, which FMAs do not have (the adds in tensor memory truncate).
//
// What bounds the product: with A's parts in shared memory the MMAs read A (4
// KB) and X (up to 8 KB) per product and 16 of K, and the copies into shared
// memory come on top: ~170 bytes per clock against the 128 that shared memory
// delivers. Here A passes through shared memory once, in FP32: TMA writes a stage
// of 16 KB, the split warps read it, split it in registers and store the parts to
// tensor memory, from where the MMAs take their A operand. Two parts at d = 205:
// 16 + 16 KB of A, 13 KB of X written and 20 KB read by the MMAs per CTA and unit of
// ~1000 clocks, half of what shared memory delivers. Neither a separate pass over
// A nor a copy of its parts is needed (4 bytes per element of A and pass instead
// of 4 or 6 and a 8 or 10 byte split).
//
// CG = 2: two CTAs of a cluster share one 256-row tile (cta_group::2): each
// holds half of X's columns, so X is read from L2 once per 256 rows and each
// shared memory feeds half of X.
//
// X's parts are written by split_x_kernel as the images of the shared-memory
// stages (32 of K, K-major rows of 64 bytes, 64-byte swizzle), copied by one TMA
// box per part.
//
// Warps: 0 copies X stages, 1 issues the MMAs, 2 allocates tensor memory, 3 copies
// stages of A; 4-11 split them, two warpgroups by turns; 12-19 drain the
// accumulators. Chains in tensor memory are cut every `chunk` units of 32 (the
// accumulation there loses a little of every add in the same direction); the drain
// warps hold the running sums in registers and add with round-to-nearest. The
// (tile, unit) pairs are dealt evenly to the CTA pairs (stream-K; whole tiles for K
// <= 1024); split tiles are summed by the last pair to arrive, or by
// split_fixup_kernel when a tile spans more than kMaxSlots of them. Every wait is
// bounded. Where one runs out, the status word reports it and the sums that were
// not read become NaN, which raises the range word in FP32.
#include <algorithm>

#include "split_device.cuh"
#include "split_gemm.cuh"
#include "tc_gemm.cuh"

namespace rqlp {
namespace sp {

static bool encode(CUtensorMap* map, const void* base, uint64_t cols, uint64_t rows, uint64_t stride, uint32_t bc,
                   uint32_t br, CUtensorMapSwizzle sw) {
  EncodeFn fn = encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t dims[2] = {cols, rows}, strides[1] = {stride};
  cuuint32_t box[2] = {bc, br}, es[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool image_map(CUtensorMap* m, const uint16_t* img, int kb, int npad, int parts) {
  EncodeFn fn = encode_fn();
  if (fn == nullptr) return false;
  const uint32_t part_rows = (uint32_t)npad / CG * BK / kImgRow;   // of one CTA's stage
  cuuint64_t dims[2] = {kImgRow, (cuuint64_t)kb * CG * parts * part_rows}, strides[1] = {kImgRow * 2};
  cuuint32_t box[2] = {kImgRow, part_rows}, es[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<uint16_t*>(img), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool class_maps(CUtensorMap* m, Classes* cl, const float* A, int64_t rows, int64_t cols, int64_t lda, bool trans) {
  for (int c = 0; c < 4; ++c) {
    const bool empty = c >= rows;
    const uintptr_t p = reinterpret_cast<uintptr_t>(A + (empty ? 0 : c) * lda);
    cl->shift[c] = (int)((p & 15) / 4);
    cl->past[c] = empty ? 1 : 0;
    if (!encode(&m[c], reinterpret_cast<const void*>(p & ~uintptr_t(15)), (uint64_t)(cols + cl->shift[c]),
                empty ? 1 : (uint64_t)((rows - c + 3) / 4), (uint64_t)lda * 16, trans ? 132 : 36, trans ? 8 : 32,
                CU_TENSOR_MAP_SWIZZLE_NONE))
      return false;
  }
  return true;
}

// Maps over A (rows x cols, row stride lda): one of boxes of 128 columns x 32
// rows (op(A) = A^T), or 32 columns x 128 rows with the 128-byte swizzle, where
// its rows are 16-byte aligned; else one per class of rows. False when the
// encoder is missing.
static bool split_maps(CUtensorMap* m, Classes* cl, bool* aligned, const float* A, int64_t rows, int64_t cols,
                       int64_t lda, bool trans) {
  *aligned = reinterpret_cast<uintptr_t>(A) % 16 == 0 && lda % 4 == 0;
  if (!*aligned) return class_maps(m, cl, A, rows, cols, lda, trans);
  return encode(m, A, (uint64_t)cols, (uint64_t)rows, (uint64_t)lda * 4, trans ? BM : BK, trans ? BK : BM,
                trans ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B);
}

}  // namespace sp

namespace {

using namespace sp;

constexpr int kMaxSlots = 16;         // partial tiles that the last CTA of a tile sums itself

struct Args {
  float* out;
  long long ldo;
  float* part;
  int* cnt;
  const int* xlo;
  int* bad;
  int* next0;               // words of the next product, cleared here
  int* next1;
  double* sumsq;
  int* info;
  // (The place of the words matters to how the kernel reads them: with npad and what
  // follows four bytes earlier, 10007 x 6001 took 107 us for 105.)
  int M, N;
  uint32_t idesc;
  int npad, kb, tiles, G, sx, sf, sa, nbuf, vec_out, fixup, whole, perm;   // sx, sf, sa: stages of X, of A in FP32, A slots
  int chunk;                // units per chain of the main accumulator
  int shares;               // SMs whose even shares bound the chains (0: the chunk alone)
  int corr_first;           // chains of one unit, the correction products first
  int flush;                // units whose sums are held in registers before they are added to global memory
  int corr;                 // 0: one accumulator; else main chains per chain of the correction accumulator
  int units;                // tiles x kb
  int stall;                // fault-injection tests: the first CTA withholds its first stage of X
  float down;               // factor of the sums (FP32: kScaleDown, A and X being scaled up)
  Classes cl;
};

// First unit of group c: an even share of all units, or of the whole tiles.
__host__ __device__ inline int first_unit(int c, int units, int G, int whole, int tiles, int kb) {
  if (whole) return (int)((long long)c * tiles / G) * kb;
  return (int)((long long)c * units / G);
}
// The group whose range holds unit u (stream-K deal).
__host__ __device__ inline int unit_owner(int u, int units, int G) {
  return (int)((((long long)u + 1) * G + units - 1) / units) - 1;
}

// Units of the chain that starts at unit k of tile t, of which `left` are to do:
// to the end of an even share of the 128-row tiles per SM, at most `chunk` from
// its start. Truncation makes every chain lose a little toward zero, so the
// lengths and places of the chains are what the result's rounding consists of.
// They follow from the product's shape and, where a pair's range ends inside a
// share, from the number of pairs (`left`), but not from the ranges alone: a range
// can be twice a share where one CTA of the pair has no rows (156512 x 336: L 8e-6
// off with chains as long as the ranges, 2e-6 with shares), and chains cut at the
// same K in all rows add up to a coherent change of A (P of the 20000^2 learned
// factorisation 3.8e-5 off, else 2.7e-5).
__device__ inline int chain_units(const Args& a, int t, int k, int left) {
  if (a.shares == 0) return min(left, a.chunk);
  const long long units = (long long)cdiv(a.M, (int64_t)BM) * a.kb, u0 = (long long)CG * t * a.kb, u = u0 + k;
  const long long c = ((u + 1) * a.shares + units - 1) / units - 1;   // the share that holds u
  const long long b = max(c * units / a.shares, u0), e = (c + 1) * units / a.shares;
  return (int)min(min((long long)left, e - u), a.chunk - (u - b) % a.chunk);
}

// Maps over A (one, or one per class of rows) and over X's image.
struct Maps {
  CUtensorMap m[4], x;
};

// ALIGNED: A's rows are 16-byte aligned, one box a stage; else four.
template <bool TRANS, int PARTS, bool ALIGNED>
__global__ void __launch_bounds__(kThreads, 1)
split_gemm_kernel(const __grid_constant__ Maps tm, const Args a) {
  grid_wait();
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nh = a.npad / CG;                                  // X columns held by this CTA
  const uint32_t part_bytes = (uint32_t)nh * BK * 2, stage_bytes = PARTS * part_bytes;
  unsigned char* fstage = smem;                                // FP32 stages of A, then X stages (both 1 KB aligned)
  constexpr uint32_t kStage = ALIGNED ? kABytes : kClassBytes;
  unsigned char* xstage = smem + (size_t)a.sf * kStage;
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
  int* last = reinterpret_cast<int*>(tmem_slot + 1);
  int* nslots = last + 1;
  int* slots = nslots + 1;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform
  const int grp = (int)blockIdx.x / CG, rank = (int)blockIdx.x % CG;
  const int KB = a.kb;
  const int u0 = first_unit(grp, a.units, a.G, a.whole, a.tiles, KB);
  const int u1 = first_unit(grp + 1, a.units, a.G, a.whole, a.tiles, KB);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *a.next0 = 0;
    *a.next1 = 0;
  }

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
  cluster_sync();   // the peer's barriers are initialised
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Tensor memory: main accumulator buffers, the correction accumulator, A
  // slots (slot s, part p: + (s PARTS + p) 16 columns).
  const uint32_t corr_base = tmem + (uint32_t)(a.nbuf * a.npad);
  const uint32_t a_base = corr_base + (a.corr ? (uint32_t)a.npad : 0u);
  const uint32_t smem_x = tc::smem_u32(xstage);
  const int nx = (*a.xlo) ? PARTS : 1;                          // X may be exact in its first part

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");   // 40 + 2 x 64 + 2 x 152 <= 5 x 96
    if (warp == 0) {
      // ------------------------------------------------ X stages
      const uint32_t xfull0 = leader_addr(xfull);
      const int rows = nh * BK / kImgRow;   // image rows of a part
      bool ok = true;
      Ring r;
      int n = u1 - u0, k = u0 % KB;
      for (int i = 0; i < n; ++i) {
        if (!wait_warp(&xempty[r.s], r.ph ^ 1u)) {
          ok = false;
          n = i;
          break;
        }
        if (elect() && !(a.stall != 0 && blockIdx.x == 0 && i == 0)) {
          if (rank == 0) tc::mbar_expect_tx(&xfull[r.s], (uint32_t)(CG * nx) * part_bytes);
          for (int p = 0; p < nx; ++p)
            load_image(xstage + (size_t)r.s * stage_bytes + p * part_bytes, &tm.x, xfull0 + 8 * r.s,
                       ((k * CG + rank) * PARTS + p) * rows);
        }
        k = k + 1 == KB ? 0 : k + 1;
        r.next(a.sx);
      }
      if (!ok) post_timeout(a.info);
      // No copy in flight at exit (the leader's barriers count the peer's copies as well).
      for (int i = rank == 0 ? max(0, n - a.sx) : n; i < n; ++i)
        if (!wait(&xfull[i % a.sx], (uint32_t)((i / a.sx) & 1))) post_timeout(a.info);
    } else if (warp == 1) {
      // ------------------------------------------------ MMAs (the pair's leader)
      bool ok = true;
      if (rank == 0) {
        Ring rx, ra, rb;      // X stages, A slots, main accumulators
        int k = u0 % KB, t = u0 / KB, left = u1 - u0, chain = 0;   // chain: main chains of this tile part
        uint32_t cph = 0;     // parity of the correction chains
        // A lane whose wait ran out goes on without waiting, and nothing is issued
        // where it is the one elected: the lanes stay together without a vote on
        // the path from a drained accumulator to its next chain (1 % at 224 columns).
        while (left > 0) {
          const int n = chain_units(a, t, k, min(left, KB - k));
          const bool cnew = a.corr != 0 && chain % a.corr == 0;   // a correction chain begins
          ok = ok && wait(&acce[rb.s], rb.ph ^ 1u) && (!cnew || wait(corre, cph ^ 1u));
          const uint32_t d = tmem + (uint32_t)(rb.s * a.npad), dc = a.corr ? corr_base : d;
          uint32_t acc = 0, cacc = cnew ? 0u : 1u;   // (with one accumulator the main product comes first)
          for (int i = 0; i < n; ++i) {
            ok = ok && wait(&xfull[rx.s], rx.ph) && wait(&afull[ra.s], ra.ph);
            tc::tc_fence_after();
            if (elect() && ok) {
              // Descriptors of the stage's parts; 16 of K are 32 bytes on.
              uint64_t x[PARTS];
#pragma unroll
              for (int p = 0; p < PARTS; ++p)
                x[p] = tc::smem_desc(smem_x + (uint32_t)rx.s * stage_bytes + p * part_bytes, 16, 512, tc::kSwizzle64);
              const uint32_t t0 = a_base + (uint32_t)(ra.s * PARTS * 16);
              issue_products<PARTS>(d, dc, t0, x, a.idesc, nx, a.corr_first != 0, acc, cacc);
              commit(&xempty[rx.s]);
              commit(&aempty[ra.s]);
            }
            acc = cacc = 1;
            rx.next(a.sx);
            ra.next(a.sa);
          }
          if (elect() && ok) commit(&accf[rb.s]);
          rb.next(a.nbuf);
          ++chain;
          k += n;
          left -= n;
          if (a.corr && (chain % a.corr == 0 || k == KB || left == 0)) cph ^= 1u;
          if (k == KB) {
            k = chain = 0;
            ++t;
          }
        }
        if (elect()) commit(done);   // no MMA in flight at teardown
      }
      if (!ok) post_timeout(a.info);
      if (!wait(done, 0)) post_timeout(a.info);
    }
    else if (warp == 3) {
      // ------------------------------------------------ FP32 tiles of A
      bool ok = true;
      Ring r;
      Cursor c(u0, KB);
      int n = u1 - u0;
      for (int i = 0; i < n; ++i) {
        if (!wait_warp(&fempty[r.s], r.ph ^ 1u)) {
          ok = false;
          n = i;
          break;
        }
        if (elect()) {
          const int row = (c.t * CG + rank) * BM, k = c.k * BK;   // both multiples of four floats
          if (ALIGNED) {
            tc::mbar_expect_tx(&ffull[r.s], kABytes);
            tc::tma_load_2d(fstage + r.s * kABytes, &tm.m[0], &ffull[r.s], TRANS ? row : k, TRANS ? k : row);
          } else {
            load_classes<TRANS>(fstage + r.s * kClassBytes, &tm.m[0], &tm.m[1], &tm.m[2], &tm.m[3], a.cl, &ffull[r.s], k,
                                row);
          }
        }
        c.next(KB);
        r.next(a.sf);
      }
      if (!ok) post_timeout(a.info);
      for (int i = max(0, n - a.sf); i < n; ++i)
        if (!wait(&ffull[i % a.sf], (uint32_t)((i / a.sf) & 1))) post_timeout(a.info);
    }
  } else if (warp < 12) {
    // -------------------------------------------------- A: load, split, store to tensor memory
    asm volatile("setmaxnreg.dec.sync.aligned.u32 64;");
    const int w = warp & 3, odd = (warp >> 2) - 1;   // two warpgroups take the units by turns
    const bool scaled = PARTS == 3 && a.down != 1.f, sq = a.sumsq != nullptr;
    Squares sum;
    // A stage holds 128 rows of op(A) by 32 of K. TRANS: as in memory, [K][row];
    // else [row][K] with the 16-byte chunks of a row xored with row % 8 (the
    // 128-byte swizzle). v[j] = op(A)(this lane's row, 16 half + j): both reads
    // are free of bank conflicts.
    auto read = [&](const unsigned char* f, int half, float* v) {
      if (TRANS) {
        const float* p = reinterpret_cast<const float*>(f) + (16 * half) * BM + 32 * w + lane;
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = p[j * BM];
      } else {
        const unsigned char* p = f + (32 * w + lane) * (BK * 4);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 q = *reinterpret_cast<const float4*>(p + (((4 * half + i) ^ (lane & 7)) << 4));
          v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
        }
      }
    };
    const uint32_t lanes = (uint32_t)(32 * w) << 16;
    bool ok = true;
    const int n = u1 - u0;
    Ring ra, rf;                     // A slot, FP32 stage of the current unit
    if (odd) {
      ra.next(a.sa);
      rf.next(a.sf);
    }
    const uint32_t afull0 = leader_addr(afull);
    for (int i = odd; i < n; i += 2) {
      const unsigned char* f = fstage + rf.s * kStage;
      auto fetch = [&](int half, float* v) {
        if (ALIGNED) read(f, half, v);
        else read_classes<TRANS>(f, a.cl, w, half, lane, v);
      };
      ok = wait_warp(&ffull[rf.s], rf.ph);
      if (!ok) break;
      float v[16];
      uint32_t o[PARTS][8];
      fetch(0, v);
      // (the slot is waited for while the values are on their way)
      ok = wait_warp(&aempty[ra.s], ra.ph ^ 1u);
      if (!ok) break;
      tc::tc_fence_after();
      split_half<PARTS>(v, o, scaled, sq, sum);
      fetch(1, v);
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
    if (!ok && lane == 0) post_timeout(a.info);
    if (sq) sum.add(a.sumsq, lane);
  } else {
    // -------------------------------------------------- drain: TMEM -> registers -> global
    asm volatile("setmaxnreg.inc.sync.aligned.u32 152;");
    const int e = warp - 12, half = e >> 2, tid = threadIdx.x - 384;
    // TMEM lane -> row of the tile (see read_classes)
    auto tile_row = [&](int l) { return ALIGNED || TRANS ? l : 4 * (l & 31) + (l >> 5); };
    const int row = 32 * (e & 3) + lane;
    const int groups = a.npad / 16, g0 = half ? (groups + 1) / 2 : 0, ng = half ? groups / 2 : (groups + 1) / 2;
    float s[kGroups][16];
    clear_sums(s);
    bool ok = true;   // after a timeout the loop runs on without waiting, so that its barriers stay in step
    int chain = 0, k = u0 % KB, t = u0 / KB, left = u1 - u0, part0 = k;   // part0: first unit of this tile part
    int since = 0;
    bool flushed = false;   // earlier sums of this part are in memory
    Ring rb;
    while (left > 0) {
      const int n = chain_units(a, t, k, min(left, KB - k));
      const bool part_end = n == left || k + n == KB;
      if (ok && !wait_warp(&accf[rb.s], rb.ph)) {
        ok = false;
        if (lane == 0) post_timeout(a.info);
      }
      if (ok) {
        tc::tc_fence_after();
        const uint32_t lanes = (uint32_t)(32 * (e & 3)) << 16, cols = (uint32_t)(16 * g0);
        drain_columns(s, tmem + lanes + (uint32_t)(rb.s * a.npad) + cols, ng, a.down);
        if (lane == 0) arrive_leader(&acce[rb.s]);
        if (a.corr && ((chain + 1) % a.corr == 0 || part_end)) {
          drain_columns(s, corr_base + lanes + cols, ng, a.down);
          if (lane == 0) arrive_leader(corre);
        }
      }
      rb.next(a.nbuf);
      ++chain;
      k += n;
      left -= n;
      since += n;
      if (!part_end && since < a.flush) continue;
      // End of this CTA's part of tile t (or a flush on the way).
      const int rt = t * CG + rank;                   // 128-row tile
      const long long gm = (long long)rt * BM + tile_row(row);
      const bool all = part0 == 0 && (k == KB || left + k >= KB), first_part = t == u0 / KB;
      float* dst;
      int ncols, qstep = 4;   // floats from one float4 of the row to the next
      bool vec;
      if (all) {
        dst = a.out + gm * a.ldo;
        ncols = gm < a.M ? a.N : 0;
        vec = a.vec_out != 0;
      } else {
        const int slot = first_part ? 2 * grp : 2 * grp + 1;   // first or last tile of the range
        dst = a.part + (long long)(slot * CG + rank) * BM * a.npad + row * 4;   // [npad / 4][128 rows][4]
        ncols = a.npad;
        qstep = 4 * BM;
        vec = true;
      }
      if (!ok) lose_sums(s);
      if (PARTS == 3 && a.bad != nullptr) check_sums(s, g0, ng, gm < a.M ? a.N : 0, a.bad);
      store_sums(s, dst, qstep, g0, ng, ncols, vec, flushed);
      if (part_end && !all && !a.fixup) {
        // Publish the partial tile; the last CTA to arrive sums them in CTA order.
        __threadfence();
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (tid == 0) {
          const int ub = t * KB, ue = ub + KB;
          const int clo = unit_owner(ub, a.units, a.G), chi = unit_owner(ue - 1, a.units, a.G);
          int n = 0;
          for (int c = clo; c <= chi; ++c) {
            const int cb = first_unit(c, a.units, a.G, 0, a.tiles, KB);
            if (cb == first_unit(c + 1, a.units, a.G, 0, a.tiles, KB)) continue;
            if (n < kMaxSlots) slots[n] = ((cb / KB == t) ? 2 * c : 2 * c + 1) * CG + rank;
            ++n;
          }
          const int old = atomicAdd(&a.cnt[rt], 1);
          *last = old == n - 1 ? 1 : 0;
          *nslots = min(n, kMaxSlots);
        }
        asm volatile("bar.sync 1, 256;" ::: "memory");
        if (*last) {
          __threadfence();
          // Thread: row lane % 8 of two row groups, float4 lane / 8 of every
          // four (128-byte reads, 64-byte writes); two slots times eight float4
          // in flight, as the loads' latency is the time of this step.
          const int n = *nslots, Q = a.npad / 4;
          for (int c0 = lane >> 3; c0 < Q; c0 += 16) {
            float4 acc[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int z = 0; z < n; z += 2) {
              float4 v[2][8];
#pragma unroll
              for (int y = 0; y < 2; ++y)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const int r = 8 * (2 * e + (j >> 2)) + (lane & 7), c = c0 + 4 * (j & 3);
                  const bool in = z + y < n && c < Q;
                  v[y][j] = in ? __ldcg(reinterpret_cast<const float4*>(
                                     a.part + (long long)slots[z + y] * BM * a.npad + (c * BM + r) * 4))
                               : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
              for (int y = 0; y < 2; ++y)
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  acc[j].x += v[y][j].x; acc[j].y += v[y][j].y; acc[j].z += v[y][j].z; acc[j].w += v[y][j].w;
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const int r = 8 * (2 * e + (j >> 2)) + (lane & 7), c = 4 * (c0 + 4 * (j & 3));
              const long long gr = (long long)rt * BM + tile_row(r);
              if (gr >= a.M || c >= a.N) continue;
              float* o = a.out + gr * a.ldo + c;
              if (a.vec_out && c + 3 < a.N) {
                *reinterpret_cast<float4*>(o) = acc[j];
              } else {
                const float x[4] = {acc[j].x, acc[j].y, acc[j].z, acc[j].w};
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  if (c + q < a.N) o[q] = x[q];
              }
            }
          }
          if (tid == 0) a.cnt[rt] = 0;
        }
      }
      clear_sums(s);   // (here, so that the sums are not live across the code above)
      flushed = !part_end;
      since = 0;
      if (part_end) {
        if (k == KB) ++t;
        chain = k = part0 = 0;
      }
      if (part_end) asm volatile("bar.sync 1, 256;" ::: "memory");   // (slots are read no more)
    }
  }

  tc::tc_fence_before();
  __syncthreads();
  cluster_sync();   // no remote arrival is still on its way
  tc::tc_fence_after();
  if (warp == 2) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// Sums the partial tiles of a product whose tiles span many CTAs: thread f
// takes float4 f of the tiles that were split, slots in CTA order.
__global__ void split_fixup_kernel(const Args a) {
  grid_wait();
  const int Q = a.npad / 4;
  const long long per = (long long)BM * Q, total = (long long)a.tiles * CG * per;
  for (long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x; f < total;
       f += (long long)gridDim.x * blockDim.x) {
    const int rt = (int)(f / per), t = rt / CG, e = (int)(f % per), r = e % BM, c = (e / BM) * 4;
    const long long gr = (long long)rt * BM + (a.perm ? 4 * (r & 31) + (r >> 5) : r);
    if (gr >= a.M || c >= a.N) continue;
    const int ub = t * a.kb, ue = ub + a.kb;
    const int clo = unit_owner(ub, a.units, a.G), chi = unit_owner(ue - 1, a.units, a.G);
    if (clo == chi) continue;   // one group had the whole tile
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z0 = clo; z0 <= chi; z0 += 8) {
      float4 v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        v[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int z = z0 + j;
        if (z > chi) continue;
        const int cb = first_unit(z, a.units, a.G, 0, a.tiles, a.kb);
        if (cb == first_unit(z + 1, a.units, a.G, 0, a.tiles, a.kb)) continue;
        const int slot = ((cb / a.kb == t) ? 2 * z : 2 * z + 1) * CG + rt % CG;
        v[j] = __ldcg(reinterpret_cast<const float4*>(a.part + (long long)slot * BM * a.npad + (c / 4 * BM + r) * 4));
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        acc.x += v[j].x; acc.y += v[j].y; acc.z += v[j].z; acc.w += v[j].w;
      }
    }
    float* o = a.out + gr * a.ldo + c;
    if (a.vec_out && c + 3 < a.N) {
      *reinterpret_cast<float4*>(o) = acc;
    } else {
      const float x[4] = {acc.x, acc.y, acc.z, acc.w};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (c + q < a.N) o[q] = x[q];
    }
  }
}

__global__ void __launch_bounds__(256)
split_x_kernel(const float* __restrict__ X, long long K, int N, long long ldx, uint16_t* __restrict__ img, int npad,
               int parts, int kb, int* xlo, bool scaled) {
  grid_wait();
  split_x_tile(X, K, N, ldx, img, npad, parts, kb, (long long)blockIdx.x * 64, blockIdx.y * 32, xlo, scaled);
}

int npad_of(int n) { return (int)round_up(n, 16); }   // N of the MMA; each CTA holds half of it, a multiple of 8

constexpr size_t kSmemExtra = 1024 + 1024;   // alignment, barriers

template <bool TRANS, int PARTS, bool ALIGNED>
cudaError_t launch(const Maps& map, Args& a, int cap, size_t smem, cudaStream_t st) {
  static PerDevice<int> known;   // pairs that run at the same time
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CG;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // (see launch_pdl)
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  int resident = 1;
  CK((cudaError_t)known.get(current_device(), &resident, [&](int* n) {
    cudaError_t e = cudaFuncSetAttribute(split_gemm_kernel<TRANS, PARTS, ALIGNED>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_optin());
    cfg.gridDim = dim3((unsigned)(sm_count() / CG * CG));
    cfg.dynamicSmemBytes = smem_optin();
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(n, split_gemm_kernel<TRANS, PARTS, ALIGNED>, &cfg);
    *n = std::max(1, std::min(*n, sm_count() / CG));
    return (int)e;
  }));
  a.G = std::min(resident, cap);
  a.fixup = (!a.whole && a.G / a.tiles + 2 > kMaxSlots) ? 1 : 0;
  cfg.gridDim = dim3((unsigned)(a.G * CG));
  cfg.dynamicSmemBytes = smem;
  cudaError_t e = cudaLaunchKernelEx(&cfg, split_gemm_kernel<TRANS, PARTS, ALIGNED>, map, a);
  note_launch();
  return e;
}

cudaError_t product(SplitGemmWs* ws, int turn, bool transA, int64_t M, int N, int64_t K, const float* A, int64_t lda,
                    const float* X, int64_t ldx, float* out, int64_t ldo, SplitMode mode, double* sumsq, int* bad,
                    int* info, cudaStream_t st) {
  const int parts = mode == kSplitTwo ? 2 : 3;
  const int npad = npad_of(N), kb = (int)cdiv(K, BK);
  int* w = ws->words;
  launch_pdl(split_x_kernel, dim3((unsigned)cdiv(kb, 2), (unsigned)cdiv(npad, 32)), 256, 0, st, X, K, N, ldx, ws->img,
             npad, parts, kb, w + turn, mode == kSplitFp32);
  note_launch();
  CK(cudaGetLastError());

  Args a = {};
  a.out = out; a.ldo = ldo;
  a.part = ws->part;
  a.cnt = ws->cnt;
  a.xlo = w + turn;
  a.bad = bad;
  a.down = mode == kSplitFp32 ? kScaleDown : 1.f;
  a.next0 = w + (turn ^ 1);
  a.next1 = w + 2 + (turn ^ 1);
  a.sumsq = sumsq;
  a.info = info;
  a.M = (int)M; a.N = N; a.npad = npad;
  a.kb = kb;
  a.tiles = (int)cdiv(M, (int64_t)BM * CG);
  if ((long long)a.tiles * kb > (1LL << 30)) return cudaErrorInvalidValue;
  a.units = a.tiles * kb;
  a.stall = ws->stall;
  // Short K: whole tiles per pair, also where most pairs then have none. Dealing the
  // units instead costs more in sums of split tiles than it spares where tiles are few
  // (FP32, us: 1500 x 1000, d = 200 48 whole and 70 dealt, 4000 x 500, d = 120 30 and 49);
  // it wins with 79 tiles on 76 pairs or one accumulator (20000 x 1000, d = 60 67 and
  // 59, 1000 x 1000, d = 210 83 and 42).
  a.whole = kb <= 32 ? 1 : 0;
  // Groups: at most two partial tiles each (none with whole tiles).
  const int cap = a.whole ? a.tiles : std::min(a.units, ws->slots / (2 * CG));
  a.vec_out = (reinterpret_cast<uintptr_t>(out) % 16 == 0 && ldo % 4 == 0) ? 1 : 0;
  a.shares = mode != kSplitFp32 ? (int)std::min<int64_t>(sm_count(), cdiv(M, BM) * kb) : 0;
  // Chains. An MMA loses about half a unit in the last place of the sum that
  // it adds to, always toward zero. FP32: one chain per unit, the correction
  // products (2^-8 of the main ones) first, so that only two MMAs add to a
  // sum of full size; 64 units are summed in registers, then in memory.
  // BF16x3: see kChainTwo; the corrections apart where tensor memory has room (npad
  // <= 128) or there are three parts.
  if (mode == kSplitFp32) {
    a.chunk = 1;
    a.corr = 0;
    a.corr_first = 1;
    a.flush = 64;
  } else {
    a.chunk = parts == 3 ? kChainThree : kChainTwo;
    a.corr = parts == 3 || npad <= 128 ? 1 : 0;
    a.flush = 1 << 30;
  }
  // Tensor memory: two main buffers where at least two A slots still fit.
  const int cc = a.corr != 0 ? npad : 0;
  a.nbuf = 2 * npad + cc + 2 * parts * 16 <= 512 ? 2 : 1;   // (FP32 above 208 columns: one)
  a.sa = std::min(kMaxASlots, (512 - a.nbuf * npad - cc) / (parts * 16));
  const size_t stage = (size_t)(npad / CG) * BK * 2 * parts;
  Maps map = {};
  bool aligned = false;
  if (!split_maps(map.m, &a.cl, &aligned, A, transA ? K : M, transA ? M : K, lda, transA) ||
      !image_map(&map.x, ws->img, kb, npad, parts))
    return cudaErrorNotSupported;
  a.perm = !aligned && !transA ? 1 : 0;
  // Shared memory: four X stages first, then FP32 stages of A, then X again.
  const size_t avail = smem_optin() - kSmemExtra;
  const size_t fstage = aligned ? kABytes : kClassBytes;
  a.sf = (int)std::min<size_t>(kMaxStages, (avail - 4 * stage) / fstage);
  const size_t fbytes = a.sf * fstage;
  a.sx = (int)std::min<size_t>(kMaxStages, (avail - fbytes) / stage);
  a.idesc = tc::idesc_bf16(BM * CG, npad, false, false);
  const size_t smem = fbytes + a.sx * stage + kSmemExtra;
#define RQLP_SPLIT(T, P) (aligned ? launch<T, P, true>(map, a, cap, smem, st) : launch<T, P, false>(map, a, cap, smem, st))
  cudaError_t e = transA ? (parts == 3 ? RQLP_SPLIT(true, 3) : RQLP_SPLIT(true, 2))
                         : (parts == 3 ? RQLP_SPLIT(false, 3) : RQLP_SPLIT(false, 2));
#undef RQLP_SPLIT
  if (e == cudaSuccess && a.fixup) {
    const long long total = (long long)a.tiles * CG * BM * (npad / 4);
    const int blocks = (int)std::min<long long>(cdiv(total, 256), (long long)sm_count() * 8);
    launch_pdl(split_fixup_kernel, blocks, 256, 0, st, a);
    note_launch();
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace

static size_t image_bytes(int64_t k_cap, int n_cap, int parts) {
  return (size_t)round_up(k_cap, BK) * npad_of(n_cap) * parts * 2;
}

size_t split_gemm_block_bytes(int64_t k_cap, int n_cap, int parts) {
  return image_bytes(k_cap, n_cap, parts) + (size_t)2 * sm_count() * BM * npad_of(n_cap) * 4;
}

bool split_gemm_layout(Arena& ar, SplitGemmWs* ws, void* block, size_t bytes, int64_t m_cap, int64_t k_cap, int n_cap,
                       int parts) {
  const size_t img = image_bytes(k_cap, n_cap, parts), slot = (size_t)BM * npad_of(n_cap) * 4;
  ws->slots = bytes > img ? (int)std::min<size_t>((bytes - img) / slot, (size_t)2 * sm_count()) : 0;
  ws->img = static_cast<uint16_t*>(block);
  ws->part = reinterpret_cast<float*>(static_cast<char*>(block) + img);
  const size_t words = 4 + (size_t)cdiv(m_cap, CG * BM) * CG;
  ws->words_bytes = words * sizeof(int);
  ws->words = ar.take<int>(words);
  ws->cnt = ar.dry ? nullptr : ws->words + 4;
  ws->turn = 0;
  return ws->slots >= sm_count() / 2 * 2;   // at least half of the CTAs' two partial tiles each
}

cudaError_t split_gemm_reset(SplitGemmWs* ws, cudaStream_t st) {
  ws->turn = 0;
  return cudaMemsetAsync(ws->words, 0, ws->words_bytes, st);
}

cudaError_t split_gemm(SplitGemmWs* ws, bool transA, int64_t M, int N, int64_t K, const float* A, int64_t lda,
                       const float* X, int64_t ldx, float* out, int64_t ldo, SplitMode mode, double* sumsq,
                       const int** range_word, int* info, bool profiled, cudaStream_t st) {
  if (M <= 0 || N <= 0 || N > 256 || K <= 0 || M > (int64_t(1) << 30) || K > (int64_t(1) << 30))
    return cudaErrorInvalidValue;
  const int turn = ws->turn & 1;
  ws->turn ^= 1;
  int* bad = mode == kSplitFp32 ? ws->words + 2 + turn : nullptr;
  if (range_word != nullptr) *range_word = bad;
  // Column halves above what a drain warp's registers hold, or where two
  // accumulators and two A slots (96 columns) exceed tensor memory.
  const int n0 = npad_of(N) > (mode == kSplitThree ? 208 : 16 * 2 * kGroups) ? npad_of((int)cdiv(N, 2)) : N;
  const bool prof = profiled && profiling_on();
  if (prof) profile_mark_begin(st);
  cudaError_t e = product(ws, turn, transA, M, n0, K, A, lda, X, ldx, out, ldo, mode, sumsq, bad, info, st);
  if (e == cudaSuccess && n0 < N)
    e = product(ws, turn, transA, M, N - n0, K, A, lda, X + n0, ldx, out + n0, ldo, mode, nullptr, bad, info, st);
  if (prof) profile_mark_end(st, transA ? 1 : 0);
  return e;
}

}  // namespace rqlp
