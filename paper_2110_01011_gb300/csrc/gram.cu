// Gram matrix G = X^T X of a long X (lower triangle) in FP32.
//
// Bound by the FMA units (the heavy pipe 65 % busy in the main loop) and, close
// behind, by shared memory: a thread's 8 x 8 block of G takes 16 floats from
// shared memory per 64 FMAs, which is what an SM delivers per FMA it can do.
// FMAs go in pairs (fma.rn.f32x2; plain ones were 5 to 20 % slower). A CTA holds
// the whole triangle in its registers and takes a range of rows: X is read once,
// where the 32 x 32 tiles of the general product read it once per tile row and
// column and spend 12 floats of shared memory per 32 FMAs. Where the triangle has
// fewer blocks than the CTA threads, groups of threads share the rows.
//
// Sums of 64 rows are added up in shared memory, then over the CTAs of a cluster
// of four (distributed shared memory), then over clusters from global memory with
// Kahan's correction, all in a fixed order. The triangle on the tensor cores in
// three BF16 parts was as fast, but its truncating sums doubled the error on the
// diagonal, which sets how orthogonal the result is.
//
// 20000 x 205: 63.4 -> 43.5 us, 100000 x 256: 343 -> 222 us, 100000 x 20: 54 -> 23 us.
#include <algorithm>

#include "gram.cuh"

namespace rqlp {
namespace {

using ull = unsigned long long;
__device__ __forceinline__ ull dup(float x) {
  ull r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void fma2(ull& c, ull a, ull b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 unpack(ull x) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
  return r;
}

constexpr int kGramThreads = 512, kGramMaxThreads = 544;   // a block per thread at d = 256 takes 528
constexpr int kStageFloats = 5120;
constexpr int kGramStages = 4;
constexpr int kCluster = 4;              // (of 38 clusters of four 35 or so fit at once; eight leave more SMs idle)
constexpr int kPromote = 64;             // rows per running sum

__host__ __device__ constexpr int gram_blocks(int d) { return (d + 7) / 8 * ((d + 7) / 8 + 1) / 2; }
__host__ __device__ constexpr int gram_slot(int d) { return 64 * ((gram_blocks(d) + 3) / 4 * 4); }
// Stages of rows, and every thread's sums. Threads: 512 (128 registers each), or what the triangle needs.
constexpr size_t gram_smem(int threads) { return ((size_t)kGramStages * kStageFloats + (size_t)64 * threads) * sizeof(float); }
// Column c of a row in shared memory: 4 floats of padding per 32, so that blocks
// four apart (read by one quarter of a warp) lie in different banks.
__device__ __forceinline__ int pos(int c) { return c + c / 32 * 4; }

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ float4 ld_remote(const float* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(a)
               : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
  return v;
}
// Block t of the lower triangle's 8 x 8 blocks, row by row.
__device__ __forceinline__ void block_of(int t, int* bi, int* bj) {
  int i = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= t) ++i;
  while (i * (i + 1) / 2 > t) --i;
  *bi = i;
  *bj = t - i * (i + 1) / 2;
}

// The cluster's sum over its rows [k0, k1) -> slot.
template <int NT>
__device__ __forceinline__ void gram_rows(const GramJob& j, long long k0, long long k1, float* slot) {
  extern __shared__ __align__(16) float smem[];
  constexpr int nt = NT;
  const int tid = threadIdx.x, d = j.d;
  float* tot = smem + kGramStages * kStageFloats;   // [64][nt]
  const int nb = (d + 7) / 8, T = nb * (nb + 1) / 2, groups = nt / T, d8 = 8 * nb;
  int stride = pos(d8 - 1) + 1;
  stride += stride % 32 == 0 ? 4 : 0;
  const int c = max(1, min(16, kStageFloats / (groups * stride))), kc = groups * c;   // rows per thread, per stage
  // This CTA's rows.
  const int rank = (int)cluster_rank(), ctas = kCluster;
  const long long n = k1 - k0, r0 = k0 + n * rank / ctas, r1 = k0 + n * (rank + 1) / ctas;
  const int stages = (int)cdiv(r1 - r0, (int64_t)kc);
  const int g = tid / T, t = tid - g * T;
  const bool active = g < groups;
  int bi = 0, bj = 0;
  block_of(active ? t : 0, &bi, &bj);

  const int q = d8 / 4, chunks = kc * q;
  const bool vec = (reinterpret_cast<uintptr_t>(j.X) & 15) == 0 && (j.ldx & 3) == 0;
  auto issue = [&](int s) {
    const long long row0 = r0 + (long long)s * kc;
    float* buf = smem + (s % kGramStages) * kStageFloats;
    for (int idx = tid; idx < chunks; idx += nt) {
      const int r = idx / q, col = 4 * (idx - r * q);
      const long long row = row0 + r;
      float* dst = buf + r * stride + pos(col);
      const int left = row < r1 ? d - col : 0;
      const float* src = left > 0 ? j.X + row * j.ldx + col : j.X;
      if (vec) {
        cp_async16(dst, src, 4 * max(0, min(4, left)));
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) cp_async4(dst + i, i < left ? src + i : j.X, i < left ? 4 : 0);
      }
    }
  };

  ull acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[i][k] = 0;
  bool first = true;
  auto flush = [&]() {
    if (!active) return;
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float2 v = unpack(acc[i][k]);
        float* p = tot + (8 * i + 2 * k) * nt + tid;
        if (!first) {
          v.x += p[0];
          v.y += p[nt];
        }
        p[0] = v.x;
        p[nt] = v.y;
        acc[i][k] = 0;
      }
    first = false;
  };

#pragma unroll
  for (int s = 0; s < kGramStages - 1; ++s) {
    if (s < stages) issue(s);
    cp_async_commit();
  }
  int run = 0;
  for (int s = 0; s < stages; ++s) {
    cp_async_wait<kGramStages - 2>();
    __syncthreads();
    if (s + kGramStages - 1 < stages) issue(s + kGramStages - 1);
    cp_async_commit();
    if (active) {
      const float* row = smem + (s % kGramStages) * kStageFloats + g * stride;
      const float* pa = row + pos(8 * bi);
      const float* pb = row + pos(8 * bj);
#pragma unroll 2
      for (int i = 0; i < c; ++i) {
        const float4 a0 = *reinterpret_cast<const float4*>(pa), a1 = *reinterpret_cast<const float4*>(pa + 4);
        const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(pb), b1 = *reinterpret_cast<const ulonglong2*>(pb + 4);
        const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
        for (int r = 0; r < 8; ++r) {
          const ull ar = dup(a[r]);
          fma2(acc[r][0], ar, b0.x);
          fma2(acc[r][1], ar, b0.y);
          fma2(acc[r][2], ar, b1.x);
          fma2(acc[r][3], ar, b1.y);
        }
        pa += groups * stride;
        pb += groups * stride;
      }
    }
    run += c;
    if (run >= kPromote) {
      flush();
      run = 0;
    }
  }
  if (run > 0 || first) flush();
  cp_async_wait_all();
  __syncthreads();

  // Over the groups of the CTA: eight threads per sum where there are as many.
  const int T4 = (T + 3) / 4 * 4;
  const float* loc = tot;
  int ls = nt;
  if (groups > 1) {
    float* red = smem;
    const int lanes = groups >= 8 ? 8 : 1, l = tid % lanes;
    for (int f = tid / lanes; f < 64 * T; f += nt / lanes) {
      const int e = f / T, u = f - e * T;
      const float* p = tot + e * nt + u;
      float s = 0.f;
      for (int h = l; h < groups; h += lanes) s += p[h * T];
      if (lanes == 8) {
        const unsigned mask = 0xffu << (threadIdx.x & 24);
        s += __shfl_xor_sync(mask, s, 4);
        s += __shfl_xor_sync(mask, s, 2);
        s += __shfl_xor_sync(mask, s, 1);
      }
      if (l == 0) red[e * T4 + u] = s;
    }
    loc = red;
    ls = T4;
  }
  cluster_barrier();
  // Over the CTAs of the cluster: each takes a share of the entries.
  const int quads = 16 * T4, f1 = quads * (rank + 1) / ctas;
  for (int f = quads * rank / ctas + tid; f < f1; f += nt) {
    const int e = f / (T4 / 4), u = 4 * (f - e * (T4 / 4));
    const float* p = loc + e * ls + u;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int r = 0; r < ctas; ++r) {
      const float4 v = ld_remote(p, (uint32_t)r);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    *reinterpret_cast<float4*>(slot + e * T4 + u) = s;
  }
  cluster_barrier();   // no CTA leaves while its sums are read
}

// Cluster z takes an even share of the rows.
template <int NT>
__global__ void __launch_bounds__(NT, 1) gram_kernel(const GramJob j, float* part, long long slot) {
  grid_wait();
  if (j.gate != nullptr && *j.gate == 0) return;
  const int z = blockIdx.x / kCluster, nz = gridDim.x / kCluster;
  gram_rows<NT>(j, j.rows * z / nz, j.rows * (z + 1) / nz, part + z * slot);
}

// G = sum of the clusters' slots: four threads per quad of sums, every fourth slot
// each (Kahan), then the four in order.
__global__ void __launch_bounds__(256)
gram_reduce_kernel(const GramJob j, const float* __restrict__ part, long long slot, int slots) {
  grid_wait();
  if (j.gate != nullptr && *j.gate == 0) return;
  const int T = gram_blocks(j.d), T4 = (T + 3) / 4 * 4, l = threadIdx.x & 3;
  for (int f = blockIdx.x * 64 + (threadIdx.x >> 2); f < 16 * T4; f += gridDim.x * 64) {
    float s[4] = {0.f, 0.f, 0.f, 0.f}, c[4] = {0.f, 0.f, 0.f, 0.f};
    for (int z = l; z < slots; z += 32) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u)
        v[u] = z + 4 * u < slots ? __ldcg(reinterpret_cast<const float4*>(part + (z + 4 * u) * slot + 4 * f))
                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float x[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float y = x[i] - c[i], w = s[i] + y;
          c[i] = (w - s[i]) - y;
          s[i] = w;
        }
      }
    }
    const unsigned mask = 0xfu << (threadIdx.x & 28);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s[i] -= c[i];
      s[i] += __shfl_xor_sync(mask, s[i], 2);
      s[i] += __shfl_xor_sync(mask, s[i], 1);
    }
    const int e = f / (T4 / 4), u = 4 * (f - e * (T4 / 4)) + l;   // each thread writes one of the four
    const float x = l == 0 ? s[0] : l == 1 ? s[1] : l == 2 ? s[2] : s[3];
    if (u < T) {
      int xi, xj;
      block_of(u, &xi, &xj);
      const int row = 8 * xi + e / 8, col = 8 * xj + e % 8;
      if (row < j.d && col <= row) j.G[(int64_t)row * j.ldg + col] = x;
    }
  }
}

int gram_threads(int d) { return gram_blocks(d) > kGramThreads ? kGramMaxThreads : kGramThreads; }

// One cluster per share of the rows, all of them resident at the same time.
template <int NT>
cudaError_t launch(const GramJob& j, float* part, size_t part_floats, int* clusters, cudaStream_t st) {
  static PerDevice<int> known;   // clusters that run at the same time
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = gram_smem(NT);
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kCluster;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // (see launch_pdl)
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  int resident = 1;
  CK((cudaError_t)known.get(current_device(), &resident, [&](int* n) {
    cudaError_t e = cudaFuncSetAttribute(gram_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gram_smem(NT));
    cfg.gridDim = dim3((unsigned)(sm_count() / kCluster * kCluster));
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(n, gram_kernel<NT>, &cfg);
    *n = std::max(1, std::min(*n, sm_count() / kCluster));
    return (int)e;
  }));
  const long long slot = gram_slot(j.d);
  *clusters = (int)std::min<long long>(resident, (long long)part_floats / slot);
  cfg.gridDim = dim3((unsigned)(*clusters * kCluster));
  const cudaError_t e = cudaLaunchKernelEx(&cfg, gram_kernel<NT>, j, part, slot);
  note_launch();
  return e;
}

}  // namespace

// Against the 32 x 32 tiles, us: 20000 x 205 44 / 63, 5000 x 255 31 / 34, 65536 x 60
// 37 / 41, 100000 x 20 23 / 54 (the tiles' K slices are long there); 16384 x 136 31 /
// 29, 8192 x 136 25 / 21, 4096 x 205 22 / 23. At least four partial sums have to fit.
bool gram_pays(int64_t rows, int d, size_t part_floats) {
  return d <= 256 && ((double)rows * d * d >= 3.2e8 || rows >= 50000) && part_floats >= 4 * (size_t)gram_slot(d);
}

cudaError_t gram_f32(const GramJob& j, float* part, size_t part_floats, cudaStream_t st) {
  int clusters = 0;
  if (gram_threads(j.d) == kGramThreads) CK(launch<kGramThreads>(j, part, part_floats, &clusters, st));
  else CK(launch<kGramMaxThreads>(j, part, part_floats, &clusters, st));
  const long long slot = gram_slot(j.d);
  launch_pdl(gram_reduce_kernel, (unsigned)cdiv(slot / 4, 64), 256, 0, st, j, part, slot, clusters);
  note_launch();
  return cudaGetLastError();
}

}  // namespace rqlp
