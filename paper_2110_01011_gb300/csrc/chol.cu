// Cholesky factor and inverse of the d x d Gram matrix of CholeskyQR: G = L L^T
// (R = L^T, upper, positive diagonal) and W = L^{-1} (R^{-1} = W^T).
//
// Blocked right-looking elimination on the augmented matrix [G | I] with
// 32-column panels J (16 in FP64). L lives in the lower triangle of one square
// buffer S and W^T in its strict upper triangle (W's diagonal in a side array),
// so that one rule updates both: S(r, c) -= S(r, J) . S(c, J) for every row r
// of S and the columns c right of the panel (below the diagonal for rows below
// the panel).
//   (1) warp 0 factors the diagonal block, the one serial chain, while
//       the other warps apply the previous panel to the rest of S, tiles
//       from a shared counter;
//   (2) o = L_JJ^{-1} v by forward substitution, a thread per row of S;
//   (3) the next diagonal block is updated ahead of the rest, for (1).
// On one SM (chol_body: FP64, and a batch's problems) the row solves and the
// tiles are bound by shared memory, (1) by its chain of a root, two products
// and a shuffle per column (~140 clocks); one FP32 matrix takes a cluster of
// ceil(d / 32) SMs (chol_cluster_kernel). Measured per factorisation, FP32, d =
// 69, 136, 205, 256: one SM with 16-column panels and the whole update of the
// lower part between (2) and (1) 23, 43, 78 and 230 us; one SM as above 17,
// 35, 68 and 186 us; the cluster 18, 29, 43 and 52 us.
// The Gram's lower triangle reaches shared memory by 16-byte asynchronous
// copies (FP32 factor, aligned rows), all of them in flight at once.
//
// A pivot that is not clearly positive restarts the elimination on G + s I
// (shifted CholeskyQR, Fukaya et al. 2020) and raises the caller's gate flag.
// The shift starts small, s0 = 10 d u trace(G), and grows tenfold while the
// shifted factor still breaks down (three shifts at most; then
// RQLP_ERR_BREAKDOWN and identities): X R^{-1} has condition number about
// sqrt(s / sigma_min(X)^2), so the smallest shift that factors leaves the
// least for the next CholeskyQR pass. With s0 = 100 d u trace(G) one FP32
// pass left a 317 x 66 sketch with kappa = 8e5 at kappa = 1.6e4, beyond what
// CholeskyQR2 can finish; with s0 = 10 d u trace(G), at 5e3.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace rqlp {
namespace {

// Panel width: 32 in FP32; 16 in FP64, whose chain and sums are bound by the
// FP64 units' rate.
template <typename T> struct Panel;
template <> struct Panel<float> { static constexpr int NB = 32; };
template <> struct Panel<double> { static constexpr int NB = 16; };
constexpr int kDtPad = 4;   // pitch of D's columns: 4 banks off a multiple of 32
// Factorisation attempts: unshifted, then shifts s0, 10 s0, 100 s0 with
// s0 = 10 d u trace(G) (u: unit roundoff of the factor's type).
constexpr int kAttempts = 4;
constexpr int kMaxD = RQLP_MAX_D;
constexpr int kThreads = 512;
constexpr int kBatchThreads = 128;

template <typename T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<double> { using type = double4_32a; };

template <typename T>
__device__ __forceinline__ void ld4(const T* p, T* v) {
  const typename Vec4<T>::type q = *reinterpret_cast<const typename Vec4<T>::type*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <typename T>
__device__ __forceinline__ void st4(T* p, const T* v) {
  typename Vec4<T>::type q;
  q.x = v[0]; q.y = v[1]; q.z = v[2]; q.w = v[3];
  *reinterpret_cast<typename Vec4<T>::type*>(p) = q;
}

template <typename T> struct Eps;
template <> struct Eps<float> { static constexpr float u = 5.9604645e-8f; };
template <> struct Eps<double> { static constexpr double u = 1.1102230246251565e-16; };

// Row pitch of the square buffer: a multiple of 4 elements (16-byte rows) and
// 4 banks off a multiple of 32, so consecutive rows start in different banks.
__host__ __device__ inline int lds_of(int d) { return (int)round_up(d, 32) + 4; }

template <typename T> struct IsF32 { static constexpr bool value = false; };
template <> struct IsF32<float> { static constexpr bool value = true; };

__device__ void post_error(int* info, int code, int detail) {
  if (info != nullptr && atomicCAS(info, 0, code) == 0) info[1] = detail;
}

__device__ void write_identity(int d, float* R, float* Rinv, int64_t ldr) {
  for (int i = threadIdx.x >> 5; i < d; i += blockDim.x >> 5)
    for (int l = threadIdx.x & 31; l < d; l += 32) {
      const float v = i == l ? 1.f : 0.f;
      if (R != nullptr) R[i * ldr + l] = v;
      Rinv[i * ldr + l] = v;
    }
}

// Dot products of NB entries for a 4 x 4 block of results: rows 8 i of `a`
// (pitch lda), rows 4 j of `b` (pitch ldb). Pitches are 4 banks off a multiple
// of 32, so that the eight rows (four columns) of a warp's step lie in
// different banks. FP32: even and odd entries in a pair of sums, two products
// an instruction. Shared memory bounds this: a load of 16 bytes takes four
// clocks whether the lanes' addresses differ or not.
template <int NB>
__device__ __forceinline__ void dot_block(const float* a, int lda, const float* b, int ldb, const bool* va,
                                          const bool* vb, float (&acc)[4][4]) {
  unsigned long long s[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) s[i][j] = 0;
#pragma unroll
  for (int k = 0; k < NB; k += 4) {
    ulonglong2 av[4], bv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const ulonglong2*>(a + (va[i] ? 8 * i * lda : 0) + k);
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const ulonglong2*>(b + (vb[j] ? 4 * j * ldb : 0) + k);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s[i][j]) : "l"(av[i].x), "l"(bv[j].x));
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(s[i][j]) : "l"(av[i].y), "l"(bv[j].y));
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      acc[i][j] = __uint_as_float((uint32_t)s[i][j]) + __uint_as_float((uint32_t)(s[i][j] >> 32));
}
template <int NB>
__device__ __forceinline__ void dot_block(const double* a, int lda, const double* b, int ldb, const bool* va,
                                          const bool* vb, double (&acc)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0;
#pragma unroll
  for (int k = 0; k < NB; k += 4) {
    double av[4][4], bv[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) ld4(a + (va[i] ? 8 * i * lda : 0) + k, av[i]);
#pragma unroll
    for (int j = 0; j < 4; ++j) ld4(b + (vb[j] ? 4 * j * ldb : 0) + k, bv[j]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += av[i][u] * bv[j][u];
  }
}

// One tile of NB rows and 16 columns of the update S(r, c) -= S(r, J) . S(c, J)
// after panel J = [j0, jn), by a warp. Tiles run over the strips of NB rows
// below jn (columns jn .. r; the next panel's diagonal block is not among them)
// and, with columns jn .. d - 1, the strips above it; the panel's own strip
// takes its rows from DT. False past the last tile.
template <typename T>
__device__ __forceinline__ bool update_tile(T* S, int LDS, const T* DT, int d, int j0, int jn, int t, int lane) {
  constexpr int NB = Panel<T>::NB, kDtLd = NB + kDtPad;
  const int nct = (d - jn + 15) / 16, nrs = (d - jn + NB - 1) / NB;
  constexpr int CPS = NB / 16;   // column strips a row strip adds
  int r0, c0, q = 1;
  while (q < nrs && t >= min(CPS * (q + 1), nct)) {
    t -= min(CPS * (q + 1), nct);
    ++q;
  }
  const bool lower = q < nrs;
  if (lower) {
    r0 = jn + NB * q;
    c0 = jn + 16 * t;
  } else {
    if (t >= jn / NB * nct) return false;
    r0 = NB * (t / nct);
    c0 = jn + 16 * (t % nct);
  }
  const int r = r0 + (lane >> 2), c = c0 + (lane & 3);   // this lane: rows r + 8 i, columns c + 4 j
  bool va[4], vb[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    va[i] = 8 * i < NB && r + 8 * i < d;
    vb[i] = c + 4 * i < d;
  }
  T acc[4][4];
  const T* a = r0 == j0 ? DT + (lane >> 2) * kDtLd : &S[(size_t)(va[0] ? r : r0) * LDS + j0];
  dot_block<NB>(a, r0 == j0 ? kDtLd : LDS, &S[(size_t)(vb[0] ? c : c0) * LDS + j0], LDS, va, vb, acc);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (va[i] && vb[j] && (!lower || c + 4 * j <= r + 8 * i)) S[(size_t)(r + 8 * i) * LDS + c + 4 * j] -= acc[i][j];
  return true;
}

// Warp 0 (lane = row): L_JJ of the jb x jb diagonal block at D (pitch ld), in
// place (zeros above the diagonal); LT its columns, rdiag 1 / L_jj. Column t is
// scaled by 1 / sqrt(pivot) and later columns c take l_it l_ct. On the path
// from a pivot to the next lie its root, two products and a shuffle; the
// columns after next take column t from LT a step later, while the next root
// is on its way. tol: this lane's pivot bound. Returns the first failing
// column, or -1 (the block is then left as it was).
template <typename T, int NB>
__device__ __forceinline__ int factor_diagonal(T* D, int ld, int jb, T tol, T* LT, T* rdiag, int lane) {
  T a[NB], lc[NB];   // the lane's row; the column before the current one
#pragma unroll
  for (int k = 0; k < NB; k += 4) {
    if (lane < jb) ld4(&D[(size_t)lane * ld + k], &a[k]);
    else a[k] = a[k + 1] = a[k + 2] = a[k + 3] = (T)0;
  }
  int f = -1;
  T piv = __shfl_sync(0xffffffffu, a[0], 0), lp = 0;
#pragma unroll
  for (int t = 0; t < NB; ++t) {
    if (t >= jb) break;
    const T rl = rsqrt(piv);   // (what a failing pivot gives is dropped with the attempt)
    if (t > 0) {
#pragma unroll
      for (int c = t + 1; c < NB; ++c) a[c] -= lp * lc[c];
    }
    const bool ok = a[t] > tol && isfinite(a[t]);   // (lane t: the pivot)
    const T l = lane >= t ? a[t] * rl : (T)0;
    if (t + 1 < NB) {
      piv = __shfl_sync(0xffffffffu, a[t + 1] - l * l, t + 1);
      a[t + 1] -= l * __shfl_sync(0xffffffffu, l, t + 1);
    }
    if (lane < NB) LT[t * NB + lane] = l;
    if ((__ballot_sync(0xffffffffu, ok) >> t & 1) == 0 && f < 0) f = t;
    if (lane == t) rdiag[t] = rl;
    a[t] = lp = l;
    __syncwarp();
#pragma unroll
    for (int c = (t + 2) / 4 * 4; c < NB; c += 4) ld4(&LT[t * NB + c], &lc[c]);
  }
  if (f < 0 && lane < jb) {
#pragma unroll
    for (int k = 0; k < NB; k += 4) {
      T o[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) o[u] = k + u <= lane ? a[k + u] : (T)0;
      st4(&D[(size_t)lane * ld + k], o);
    }
  }
  return f;
}

// What 1 / sqrt(pivot) = r, with l = pivot r on L's diagonal, lacks relative to
// itself (one Newton step). rsqrtf is 5e-8 low on average next to 1, where the
// pivots of a second CholeskyQR pass lie: every column of the result came out short by
// that and L with it (30 FP32 factorisations: L off by 2.6e-7; 1.7e-7 with the
// step). Column t of L and row t of W carry the factor; both are corrected on their
// way out (in the chain above, or behind it, the step took 0.3 us per panel).
template <typename T>
__device__ __forceinline__ T root_correction(T l, T r) { return (T)0.5 * fma(-l, r, (T)1); }

// v = L_JJ^{-1} v by forward substitution, column by column: an entry is final
// one product after the one before it.
template <typename T, int NB>
__device__ __forceinline__ void solve_row(T (&v)[NB], const T* LT, const T* rdiag, int jb) {
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    if (c >= jb) break;
    v[c] *= rdiag[c];
#pragma unroll
    for (int k = (c + 1) / 4 * 4; k < NB; k += 4) {
      T l[4];
      ld4(&LT[c * NB + k], l);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k + u > c) v[k + u] -= l[u] * v[c];
    }
  }
}

// The factorisation of one problem by the whole CTA (any multiple of 32
// threads up to kThreads). gS: the square buffer in global memory (used
// when !kShared).
template <typename T, bool kShared>
__device__ __forceinline__ void chol_body(int d, const float* __restrict__ G, int64_t ldg, float* __restrict__ R,
                                          float* __restrict__ Rinv, int64_t ldr, int* info, double* shift_count,
                                          int* gate_out, const int* gate_in, T* gS) {
  extern __shared__ __align__(32) unsigned char smem_raw[];
  constexpr int NB = Panel<T>::NB, kDtLd = NB + kDtPad;
  const int LDS = lds_of(d);
  T* dyn = reinterpret_cast<T*>(smem_raw);
  T* DT = dyn;                 // D = L_JJ^{-1} by columns: DT[c][k] = D_kc
  T* LT = DT + NB * kDtLd;     // L_JJ by columns: LT[t][i] = L_it (zero above the diagonal)
  T* S = kShared ? LT + NB * NB : gS;
  __shared__ __align__(32) T gdiag[kMaxD];   // G's diagonal; W's once a panel is done
  __shared__ T rdiag[NB];                    // 1 / L_jj of the current diagonal block
  __shared__ T corr[kMaxD];                  // root_correction of every column
  __shared__ int s_fail, s_tile;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;

  if (gate_in != nullptr && *gate_in == 0) return;   // pass not needed: nothing reads R or R^{-1}

  const T rel_tol = (T)64 * Eps<T>::u;
  T shift = 0;
  int fail = -1;
  for (int attempt = 0; attempt < kAttempts; ++attempt) {
    // attempt a >= 1 factors G + 10^(a-1) s0 I: the smallest shift that
    // succeeds reduces kappa(X R^{-1}) the most
    if (attempt > 1) shift *= (T)10;
    const T sh = attempt == 0 ? (T)0 : shift;
    // Lower triangle of G (+ sh I) into S, zeros above.
    bool loaded = false;
    if constexpr (kShared && IsF32<T>::value) {
      if ((reinterpret_cast<uintptr_t>(G) & 15) == 0 && (ldg & 3) == 0) {
        // 16-byte chunks: those that reach the diagonal are copied
        // asynchronously (all in flight at once), the others cleared; then
        // the diagonal chunk's entries above the diagonal are cleared and
        // the shift added. Chunk c of row i ends at 4 c + 3 < round_up(d, 4)
        // <= ldg, and S's rows hold LDS > 4 c + 3 entries.
        const int nch = (d + 3) >> 2;
        for (int e = tid; e < d * nch; e += blockDim.x) {
          const int i = e / nch, c4 = 4 * (e - i * nch);
          T* dst = &S[(size_t)i * LDS + c4];
          if (c4 <= i) {
            cp_async16(dst, &G[(int64_t)i * ldg + c4]);
          } else {
            const T z[4] = {(T)0, (T)0, (T)0, (T)0};
            st4(dst, z);
          }
        }
        cp_async_wait_all();
        __syncthreads();
        for (int i = tid; i < d; i += blockDim.x) {
          const int ce = min(d, (i & ~3) + 4);
          for (int j = i + 1; j < ce; ++j) S[(size_t)i * LDS + j] = (T)0;
          const T x = S[(size_t)i * LDS + i] + sh;
          S[(size_t)i * LDS + i] = x;
          gdiag[i] = x;
        }
        loaded = true;
      }
    }
    // Otherwise a warp per group of four rows, lanes over columns, all of a
    // group's loads issued before its stores.
    for (int i0 = 4 * warp; !loaded && i0 < d; i0 += 4 * nwarps) {
      T v[4][kMaxD / 32];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int t = 0; t < kMaxD / 32; ++t) {
          const int i = i0 + r, j = lane + 32 * t;
          v[r][t] = (i < d && j <= i) ? (T)G[(int64_t)i * ldg + j] : (T)0;
        }
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int t = 0; t < kMaxD / 32; ++t) {
          const int i = i0 + r, j = lane + 32 * t;
          if (i < d && j < d) {
            const T x = v[r][t] + (j == i ? sh : (T)0);
            S[(size_t)i * LDS + j] = x;
            if (j == i) gdiag[i] = x;
          }
        }
    }
    __syncthreads();
    if (attempt == 0) {   // trace(G), reduced by every warp in the same order
      T tr = 0;
      for (int i = lane; i < d; i += 32) tr += gdiag[i];
      for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
      if (!isfinite(tr)) {
        if (tid == 0) post_error(info, RQLP_ERR_NONFINITE, 0);
        write_identity(d, R, Rinv, ldr);
        return;
      }
      shift = (T)(10.0 * d) * Eps<T>::u * tr;
    }
    fail = -1;
    for (int j0 = 0; j0 < d; j0 += NB) {
      const int jb = min(NB, d - j0), jn = j0 + jb;
      // (1) Warp 0 factors the diagonal block; the other warps, and warp 0 when
      // it is done, apply the previous panel to the rest of S.
      if (warp == 0) {
        const int f = factor_diagonal<T, NB>(&S[(size_t)j0 * LDS + j0], LDS, jb,
                                             lane < jb ? rel_tol * gdiag[j0 + lane] : (T)0, LT, rdiag, lane);
        if (lane == 0) s_fail = f < 0 ? -1 : j0 + f;
      }
      // (warps 4, 8 and 12 leave warp 0 its scheduler: beside three working warps
      // its chain took twice as long)
      if (j0 > 0 && (warp == 0 || nwarps < 8 || (warp & 3) != 0)) {
        for (;;) {
          int t = 0;
          if (lane == 0) t = atomicAdd(&s_tile, 1);
          t = __shfl_sync(0xffffffffu, t, 0);
          if (!update_tile<T>(S, LDS, DT, d, j0 - NB, j0, t, lane)) break;
        }
      }
      __syncthreads();
      if (tid == 0) s_tile = 0;
      if (s_fail >= 0) {
        fail = s_fail;
        break;
      }
      // (2) o = L_JJ^{-1} v for every row of S, a thread per row: v = its panel
      // columns, in place (L_IJ below the panel, W_J,: above it); the panel's
      // own rows start from unit vectors and give D. An entry is final one
      // product after the one before it.
      for (int r = tid; r < d; r += blockDim.x) {
        T* row = &S[(size_t)r * LDS + j0];
        const int cc = r - j0;   // 0 .. jb - 1: the panel's own rows
        const bool own = cc >= 0 && cc < jb;
        T v[NB];
#pragma unroll
        for (int k = 0; k < NB; k += 4) {
          T x[4];
          ld4(&row[k], x);
#pragma unroll
          for (int u = 0; u < 4; ++u) v[k + u] = own ? (k + u == cc ? (T)1 : (T)0) : (k + u < jb ? x[u] : (T)0);
        }
        solve_row<T, NB>(v, LT, rdiag, jb);
        if (own) {
          gdiag[r] = rdiag[cc];
          corr[r] = root_correction(LT[cc * NB + cc], rdiag[cc]);
#pragma unroll
          for (int k = 0; k < NB; k += 4) st4(&DT[cc * kDtLd + k], &v[k]);
#pragma unroll
          for (int k = 0; k < NB; ++k)
            if (k > cc && k < jb) row[k] = v[k];
        } else {
#pragma unroll
          for (int k = 0; k < NB; k += 4) st4(&row[k], &v[k]);
        }
      }
      __syncthreads();
      // (3) The next diagonal block, which step (1) waits for: entries
      // (r, c), (r + NB / 2, c) and (r + NB / 2, c + NB / 2) per thread.
      if (jn < d) {
        constexpr int H = NB / 2;
        for (int t = tid; t < H * H; t += blockDim.x) {
          const int r = jn + t / H, c = jn + t % H;
          const bool r1 = r + H < d, c1 = c + H < d;
          if (r >= d || c >= d) continue;
          T a00 = 0, a10 = 0, a11 = 0;
          const T* pr = &S[(size_t)r * LDS + j0];
          const T* pc = &S[(size_t)c * LDS + j0];
          const size_t up = (size_t)H * LDS;
#pragma unroll
          for (int k = 0; k < NB; k += 4) {
            T x0[4], x1[4], y0[4], y1[4];
            ld4(pr + k, x0);
            ld4(pr + (r1 ? up : 0) + k, x1);
            ld4(pc + k, y0);
            ld4(pc + (c1 ? up : 0) + k, y1);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              a00 += x0[u] * y0[u];
              a10 += x1[u] * y0[u];
              a11 += x1[u] * y1[u];
            }
          }
          if (c <= r) S[(size_t)r * LDS + c] -= a00;
          if (r1) S[(size_t)(r + H) * LDS + c] -= a10;
          if (r1 && c1 && c <= r) S[(size_t)(r + H) * LDS + c + H] -= a11;
        }
        __syncthreads();
      }
    }
    if (fail < 0) break;
    __syncthreads();
    if (attempt == 0 && tid == 0) {
      if (gate_out != nullptr) *gate_out = 1;
      if (shift_count != nullptr) atomicAdd(shift_count, 1.0);
    }
  }

  if (fail >= 0) {
    if (tid == 0) post_error(info, RQLP_ERR_BREAKDOWN, fail + 1);
    write_identity(d, R, Rinv, ldr);
    return;
  }
  __syncthreads();   // (d <= NB: step (2) was the last)
  // R = L^T (upper); R^{-1} = W^T: strict upper part from S, diagonal from gdiag.
  for (int i = warp; i < d; i += nwarps) {   // a warp per row, lanes over columns, a row's loads before its stores
    float* r = R != nullptr ? R + (int64_t)i * ldr : nullptr;
    float* ri = Rinv + (int64_t)i * ldr;
    float x[kMaxD / 32], y[kMaxD / 32];
#pragma unroll
    for (int t = 0; t < kMaxD / 32; ++t) {
      const int l = lane + 32 * t;
      const T v = l < d && l >= i ? (l > i ? S[(size_t)i * LDS + l] : gdiag[i]) : (T)0;
      const T w = l < d && l >= i && R != nullptr ? S[(size_t)l * LDS + i] : (T)0;
      x[t] = (float)fma(v, l < d ? corr[l] : (T)0, v);
      y[t] = (float)fma(w, corr[i], w);
    }
#pragma unroll
    for (int t = 0; t < kMaxD / 32; ++t) {
      const int l = lane + 32 * t;
      if (l < d) {
        ri[l] = x[t];
        if (R != nullptr) r[l] = y[t];
      }
    }
  }
}

template <typename T, bool kShared>
__global__ void __launch_bounds__(kThreads)
chol_blocked_kernel(int d, const float* __restrict__ G, int64_t ldg, float* __restrict__ R, float* __restrict__ Rinv,
                    int64_t ldr, int* info, double* shift_count, int* gate_out, const int* gate_in, T* gS) {
  grid_wait();
  chol_body<T, kShared>(d, G, ldg, R, Rinv, ldr, info, shift_count, gate_out, gate_in, gS);
}

// FP32 factorisation of one matrix by a cluster: CTA s holds rows 32 s .. 32 s +
// 31 of S (ceil(d / 32) CTAs, at most 8). The steps are chol_body's; a panel's
// owner factors its diagonal block and the others copy L_JJ from its shared
// memory, each CTA solves its own rows, and the rows' panel entries are
// gathered from their owners for the update. On the path from one panel to the
// next lie the diagonal block (one warp), a cluster barrier, the copy of L_JJ,
// one row solve and the next owner's update of its own diagonal block; the
// rest of the update runs beside the next diagonal block on all SMs of the
// cluster.
constexpr int kClusterThreads = 256;

__device__ __forceinline__ uint32_t remote_addr(const void* p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ float4 remote_ld4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a)
               : "memory");
  return v;
}
__device__ __forceinline__ int remote_ld(uint32_t a) {
  int v;
  asm volatile("ld.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <int NB>
size_t cluster_smem_bytes(int d) {
  return ((size_t)NB * lds_of(d) + (size_t)round_up(d, NB) * (NB + kDtPad) + NB * (NB + kDtPad) + NB * NB + NB) *
         sizeof(float);
}

// NB: 32, or 16 for one CTA of d <= 16.
template <int NB>
__global__ void __launch_bounds__(kClusterThreads)
chol_cluster_kernel(int d, const float* __restrict__ G, int64_t ldg, float* __restrict__ R, float* __restrict__ Rinv,
                    int64_t ldr, int* info, double* shift_count, int* gate_out, const int* gate_in) {
  grid_wait();
  extern __shared__ __align__(32) unsigned char smem_raw[];
  constexpr int kCLd = NB + kDtPad;
  const int LDS = lds_of(d), rank = blockIdx.x, P = gridDim.x;
  float* S = reinterpret_cast<float*>(smem_raw);   // rows 32 rank .. of S
  float* C = S + NB * LDS;                         // S(c, J) of the other rows, pitch kCLd (row c at c)
  float* DT = C + (size_t)round_up(d, NB) * kCLd;
  float* LT = DT + NB * kCLd;                      // L_JJ by columns: the owner's, or a copy
  float* rdiag = LT + NB * NB;                     // (behind LT: one copy takes both)
  __shared__ float gdiag[NB];                      // G's diagonal; W's once the panel is done
  __shared__ float corr[kMaxD];                    // root_correction of every column
  __shared__ int s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kClusterThreads / 32;
  const int i0 = NB * rank, rows = min(NB, d - i0);

  if (gate_in != nullptr && *gate_in == 0) return;   // pass not needed (the same for every CTA)

  const float rel_tol = 64 * Eps<float>::u;
  float shift = 0;
  int fail = -1;
  for (int attempt = 0; attempt < kAttempts; ++attempt) {
    if (attempt > 1) shift *= 10.f;
    if (attempt == 0) {   // trace(G), by every warp in the same order
      float tr = 0;
      for (int i = lane; i < d; i += 32) tr += G[(int64_t)i * ldg + i];
      for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
      if (!isfinite(tr)) {
        if (rank == 0) {
          if (tid == 0) post_error(info, RQLP_ERR_NONFINITE, 0);
          write_identity(d, R, Rinv, ldr);
        }
        return;
      }
      shift = (float)(10.0 * d) * Eps<float>::u * tr;
    }
    const float sh = attempt == 0 ? 0.f : shift;
    // The rows' lower part of G (+ sh I), zeros above.
    for (int e = tid; e < rows * (LDS / 4); e += kClusterThreads) {
      const int i = e / (LDS / 4), c = 4 * (e % (LDS / 4)), gi = i0 + i;
      float x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        x[u] = c + u <= gi ? G[(int64_t)gi * ldg + c + u] + (c + u == gi ? sh : 0.f) : 0.f;
      st4(&S[i * LDS + c], x);
      if (gi >= c && gi < c + 4) gdiag[i] = x[gi - c];
    }
    __syncthreads();
    fail = -1;
    for (int J = 0; J < P; ++J) {
      const int j0 = NB * J, jb = min(NB, d - j0);
      // (1) beside the update with the previous panel (arrivals: end of (2))
      if (rank == J && warp == 0) {
        const int f = factor_diagonal<float, NB>(&S[j0], LDS, jb, lane < jb ? rel_tol * gdiag[lane] : 0.f, LT, rdiag,
                                                 lane);
        if (lane == 0) s_fail = f < 0 ? -1 : j0 + f;
        if (J > 0) cluster_wait();
      } else if (J > 0) {
        cluster_wait();   // every CTA's rows of panel J - 1 are solved
        const int p0 = j0 - NB;
        // Columns c of the update: j0 .. r below the panel (the owner of J has
        // done its diagonal block), j0 .. d - 1 above.
        const bool lower = rank >= J;
        const int cend = lower ? min(d, i0 + NB) : d;
        if (!(rank == J)) {
          for (int e = tid; e < (cend - j0) * (NB / 4); e += kClusterThreads) {
            const int c = j0 + e / (NB / 4), k = 4 * (e % (NB / 4)), o = c / NB;
            const float4 v = remote_ld4(remote_addr(&S[(c - NB * o) * LDS + p0 + k], o));
            *reinterpret_cast<float4*>(&C[(c - j0) * kCLd + k]) = v;
          }
          __syncthreads();
          for (int t = warp; j0 + 16 * t < cend; t += nwarps) {
            const int r = lane >> 2, c = j0 + 16 * t + (lane & 3);   // rows r + 8 i, columns c + 4 j
            bool va[4], vb[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              va[i] = r + 8 * i < rows;
              vb[i] = c + 4 * i < cend;
            }
            float acc[4][4];
            const bool own = rank == J - 1;
            const float* a = own ? DT + r * kCLd : &S[(va[0] ? r : 0) * LDS + p0];
            dot_block<NB>(a, own ? kCLd : LDS, &C[(vb[0] ? c - j0 : 0) * kCLd], kCLd, va, vb, acc);
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (va[i] && vb[j] && (!lower || c + 4 * j <= i0 + r + 8 * i)) S[(r + 8 * i) * LDS + c + 4 * j] -= acc[i][j];
          }
        }
      }
      __syncwarp();
      cluster_arrive();
      cluster_wait();
      // (2)
      if (rank != J) {
        for (int e = tid; e < (NB * NB + NB) / 4; e += kClusterThreads)
          *reinterpret_cast<float4*>(&LT[4 * e]) = remote_ld4(remote_addr(&LT[4 * e], J));
      }
      fail = remote_ld(remote_addr(&s_fail, J));
      __syncthreads();
      if (fail >= 0) break;
      if (warp == 0) {
        const bool in = lane < rows, own = rank == J;
        float* row = &S[(in ? lane : 0) * LDS + j0];
        float v[NB];
#pragma unroll
        for (int k = 0; k < NB; k += 4) {
          float x[4];
          ld4(&row[k], x);
#pragma unroll
          for (int u = 0; u < 4; ++u) v[k + u] = own ? (k + u == lane ? 1.f : 0.f) : (k + u < jb ? x[u] : 0.f);
        }
        solve_row<float, NB>(v, LT, rdiag, jb);
        if (own) {
          if (in) {
            gdiag[lane] = rdiag[lane];
#pragma unroll
            for (int k = 0; k < NB; k += 4) st4(&DT[lane * kCLd + k], &v[k]);
#pragma unroll
            for (int k = 0; k < NB; ++k)
              if (k > lane && k < jb) row[k] = v[k];
          }
        } else if (in) {
#pragma unroll
          for (int k = 0; k < NB; k += 4) st4(&row[k], &v[k]);
        }
      } else if (warp == 1 && lane < jb) {
        corr[j0 + lane] = root_correction(LT[lane * NB + lane], rdiag[lane]);
      }
      __syncthreads();
      if (J + 1 == P) break;
      cluster_arrive();   // waited for in (1) of the next panel
      // (3) the next owner's diagonal block
      if (rank == J + 1) {
        for (int t = tid; t < 256; t += kClusterThreads) {
          const int r = t >> 4, c = t & 15;
          const bool r1 = r + 16 < rows, c1 = c + 16 < rows;
          if (r >= rows || c >= rows) continue;
          float a00 = 0, a10 = 0, a11 = 0;
          const float *pr = &S[r * LDS + j0], *pc = &S[c * LDS + j0];
#pragma unroll
          for (int k = 0; k < NB; k += 4) {
            float x0[4], x1[4], y0[4], y1[4];
            ld4(pr + k, x0);
            ld4(pr + (r1 ? 16 * LDS : 0) + k, x1);
            ld4(pc + k, y0);
            ld4(pc + (c1 ? 16 * LDS : 0) + k, y1);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              a00 += x0[u] * y0[u];
              a10 += x1[u] * y0[u];
              a11 += x1[u] * y1[u];
            }
          }
          if (c <= r) S[r * LDS + i0 + c] -= a00;
          if (r1) S[(r + 16) * LDS + i0 + c] -= a10;
          if (r1 && c1 && c <= r) S[(r + 16) * LDS + i0 + c + 16] -= a11;
        }
        __syncthreads();
      }
    }
    cluster_arrive();   // no CTA reads another's shared memory any more
    cluster_wait();
    if (fail < 0) break;
    if (attempt == 0 && rank == 0 && tid == 0) {
      if (gate_out != nullptr) *gate_out = 1;
      if (shift_count != nullptr) atomicAdd(shift_count, 1.0);
    }
  }
  if (fail >= 0) {
    if (rank == 0) {
      if (tid == 0) post_error(info, RQLP_ERR_BREAKDOWN, fail + 1);
      write_identity(d, R, Rinv, ldr);
    }
    return;
  }
  // R^{-1} = W^T: this CTA's rows. R = L^T: its columns.
  for (int i = warp; i < rows; i += nwarps) {
    float* ri = Rinv + (int64_t)(i0 + i) * ldr;
#pragma unroll
    for (int t = 0; t < kMaxD / 32; ++t) {
      const int l = lane + 32 * t;
      if (32 * t >= d) break;
      if (l < d) {
        const float v = l > i0 + i ? S[i * LDS + l] : (l == i0 + i ? gdiag[i] : 0.f);
        ri[l] = fmaf(v, corr[l], v);
      }
    }
  }
  if (R != nullptr && lane < rows) {
#pragma unroll 4
    for (int i = warp; i < d; i += nwarps) {
      const float v = i <= i0 + lane ? S[lane * LDS + i] : 0.f;
      R[(int64_t)i * ldr + i0 + lane] = fmaf(v, corr[i], v);
    }
  }
}

// One CTA per problem of a batch; every square buffer in shared memory.
template <typename T>
__global__ void __launch_bounds__(kBatchThreads, 3)
chol_batched_kernel(const CholJob* __restrict__ jobs, int count) {
  const int b = blockIdx.x;
  if (b >= count) return;
  const CholJob j = jobs[b];
  chol_body<T, true>(j.d, j.G, j.ldg, j.R, j.Rinv, j.ldr, j.info, j.shift_count, j.gate_out, j.gate_in, nullptr);
}

template <typename T>
size_t square_bytes(int d) { return (size_t)d * lds_of(d) * sizeof(T); }
template <typename T>
size_t panel_bytes() { return (size_t)Panel<T>::NB * (2 * Panel<T>::NB + kDtPad) * sizeof(T); }
template <typename T>
size_t static_bytes() { return (2 * kMaxD + Panel<T>::NB) * sizeof(T) + 96; }
template <typename T>
bool square_in_smem(int d) {
  return square_bytes<T>(d) + panel_bytes<T>() + static_bytes<T>() <= smem_optin();
}

template <typename T>
cudaError_t launch(int d, const float* G, int64_t ldg, float* R, float* Rinv, int64_t ldr, int* info,
                   double* shift_count, int* gate_out, const int* gate_in, void* gstore, cudaStream_t st) {
  static PerDevice<char> once[2];
  CK(allow_smem(&once[0], chol_blocked_kernel<T, true>, smem_optin() - static_bytes<T>()));
  CK(allow_smem(&once[1], chol_blocked_kernel<T, false>, smem_optin() - static_bytes<T>()));
  const bool in_smem = square_in_smem<T>(d);
  if (!in_smem && gstore == nullptr) return cudaErrorInvalidValue;
  const size_t dyn = panel_bytes<T>() + (in_smem ? square_bytes<T>(d) : 0);
  if (in_smem)
    launch_pdl(chol_blocked_kernel<T, true>, 1, kThreads, dyn, st, d, G, ldg, R, Rinv, ldr, info, shift_count,
               gate_out, gate_in, nullptr);
  else
    launch_pdl(chol_blocked_kernel<T, false>, 1, kThreads, dyn, st, d, G, ldg, R, Rinv, ldr, info, shift_count,
               gate_out, gate_in, reinterpret_cast<T*>(gstore));
  note_launch();
  return cudaGetLastError();
}

template <int NB>
cudaError_t launch_cluster(int d, const float* G, int64_t ldg, float* R, float* Rinv, int64_t ldr, int* info,
                           double* shift_count, int* gate_out, const int* gate_in, cudaStream_t st) {
  static PerDevice<char> once;
  CK(allow_smem(&once, chol_cluster_kernel<NB>, cluster_smem_bytes<NB>(kMaxD)));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cdiv(d, NB);
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // (see launch_pdl)
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)cdiv(d, NB));
  cfg.blockDim = dim3(kClusterThreads);
  cfg.dynamicSmemBytes = cluster_smem_bytes<NB>(d);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  const cudaError_t e =
      cudaLaunchKernelEx(&cfg, chol_cluster_kernel<NB>, d, G, ldg, R, Rinv, ldr, info, shift_count, gate_out, gate_in);
  note_launch();
  return e;
}

template <typename T>
cudaError_t launch_batched(const CholJob* jobs, int count, int dmax, cudaStream_t st) {
  static PerDevice<char> once;
  CK(allow_smem(&once, chol_batched_kernel<T>, smem_optin() - static_bytes<T>()));
  if (count <= 0) return cudaSuccess;   // configuration only
  if (!square_in_smem<T>(dmax)) return cudaErrorInvalidValue;
  const size_t dyn = panel_bytes<T>() + square_bytes<T>(dmax);
  chol_batched_kernel<T><<<count, kBatchThreads, dyn, st>>>(jobs, count);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

bool chol_batched_fits(int dmax, bool fp64) {
  return fp64 ? square_in_smem<double>(dmax) : square_in_smem<float>(dmax);
}

cudaError_t chol_inv_batched(const CholJob* jobs, int count, int dmax, bool fp64, cudaStream_t st) {
  return fp64 ? launch_batched<double>(jobs, count, dmax, st) : launch_batched<float>(jobs, count, dmax, st);
}

// The square of a single FP64 factor that does not fit in shared memory; one in FP32
// lies in a cluster's.
size_t chol_global_bytes(int d, bool fp64) { return fp64 && !square_in_smem<double>(d) ? square_bytes<double>(d) : 0; }

cudaError_t chol_inv(int d, const float* G, int64_t ldg, float* R, float* Rinv, int64_t ldr, int* info,
                     double* shift_count, int* gate_out, const int* gate_in, void* gstore, bool fp64,
                     cudaStream_t st) {
  if (fp64) return launch<double>(d, G, ldg, R, Rinv, ldr, info, shift_count, gate_out, gate_in, gstore, st);
  return d <= 16 ? launch_cluster<16>(d, G, ldg, R, Rinv, ldr, info, shift_count, gate_out, gate_in, st)
                 : launch_cluster<32>(d, G, ldg, R, Rinv, ldr, info, shift_count, gate_out, gate_in, st);
}

}  // namespace rqlp
