// Gradient g = Aᵀ(b − Ax) − λx of a small matrix in one launch, without
// scratch: one thread-block cluster whose blocks split the rows and add their
// column sums through each other's shared memory.
//
// A small gradient is bound by its launches and the gap between them, and by
// what the host does for it, not by its bytes: at 4096×256 (4 MB) the pass over
// all SMs and its finalize kernel take 5 + 5 µs on the device, and a call took
// 21 µs with the allocation of the partial sums, or 206 µs when the GPU is waited
// for after it (the pool then gives its memory back each time).  This form: 15
// and 27 µs; 8192×256: 22 → 15, 207 → 30 µs.
//
// Block q of 16 takes rows [q·R, q·R + R), its warps every sixteenth of them,
// RW rows at a time (64 floats of A per lane in flight); lane ℓ holds columns
// 4ℓ + 128c of x, of the rows and of their sum.  The warps' sums are added in
// order in shared memory, the blocks' after each has sent the owner of a slice
// of columns its share; the cluster barriers on both sides of that are the only
// ones.
#include "internal.h"

namespace mihs {
namespace {

constexpr int kCluster = 16;
constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kSmallMaxD = 512;
// n × the columns that the lanes cover (256, or 512 from d = 257).  16 SMs draw a
// quarter of the bandwidth that all of them do, and the cost goes by rows as
// much as by bytes.  Up to this line the host still bounds the call: 14.5 µs at
// 8192×512, 16384×256 and 16384×128, where the pass over all SMs takes 20–22;
// twice as far it is 23, 25 and 23 against 20.
constexpr int64_t kSmallElems = 4 << 20;

__device__ __forceinline__ uint32_t mapa_u32(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_f1(uint32_t dst, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

template <int CH, int RW>
__global__ void __launch_bounds__(kThreads, 1)
gradient_small_kernel(const float* __restrict__ A, int n, int d, long long lda, const float* __restrict__ b,
                      const float* x, float lambda, float* g) {
  __shared__ __align__(16) float red[kWarps][CH * 128];    // the warps' column sums
  __shared__ float recv[kCluster][CH * 128 / kCluster];    // the blocks' shares of this block's columns
  constexpr int kSlice = CH * 128 / kCluster;              // columns per owner
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  cluster_arrive();  // every block runs before any is written to

  float4 xv[CH], acc[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int j = 128 * c + 4 * lane;
    xv[c] = make_float4(j < d ? x[j] : 0.f, j + 1 < d ? x[j + 1] : 0.f, j + 2 < d ? x[j + 2] : 0.f,
                        j + 3 < d ? x[j + 3] : 0.f);
    acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const int per = (n + kCluster - 1) / kCluster;
  const int r1 = min(n, ((int)rank + 1) * per);
  for (int i0 = (int)rank * per + warp; i0 < r1; i0 += kWarps * RW) {
    float4 a[RW][CH];
    float s[RW], bi[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      const int i = i0 + r * kWarps;
      const bool on = i < r1;
      bi[r] = on ? __ldg(b + i) : 0.f;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int j = 128 * c + 4 * lane;
        a[r][c] = on && j < d ? __ldg(reinterpret_cast<const float4*>(A + (long long)i * lda + j))
                              : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      s[r] = 0.f;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int j = 128 * c + 4 * lane;
        if (j + 4 > d) {  // the padding of a ragged row may hold anything
          if (j + 1 >= d) a[r][c].y = 0.f;
          if (j + 2 >= d) a[r][c].z = 0.f;
          a[r][c].w = 0.f;
        }
        s[r] = fmaf(a[r][c].x, xv[c].x,
                    fmaf(a[r][c].y, xv[c].y, fmaf(a[r][c].z, xv[c].z, fmaf(a[r][c].w, xv[c].w, s[r]))));
      }
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
      for (int r = 0; r < RW; ++r) s[r] += __shfl_xor_sync(0xffffffffu, s[r], o);
#pragma unroll
    for (int r = 0; r < RW; ++r) {
      // (a row past the block's is zero; its product with an infinite x is not)
      const float res = i0 + r * kWarps < r1 ? bi[r] - s[r] : 0.f;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        acc[c].x = fmaf(res, a[r][c].x, acc[c].x);
        acc[c].y = fmaf(res, a[r][c].y, acc[c].y);
        acc[c].z = fmaf(res, a[r][c].z, acc[c].z);
        acc[c].w = fmaf(res, a[r][c].w, acc[c].w);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < CH; ++c) *reinterpret_cast<float4*>(&red[warp][128 * c + 4 * lane]) = acc[c];
  __syncthreads();
  cluster_wait();
  const int t = threadIdx.x;
  if (t < CH * 128) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) sum += red[w][t];
    st_cluster_f1(mapa_u32(smem_u32(&recv[rank][t % kSlice]), (uint32_t)(t / kSlice)), sum);
  }
  cluster_arrive();
  cluster_wait();
  const int j = (int)rank * kSlice + t;
  if (t < kSlice && j < d) {
    float sum = 0.f;
#pragma unroll
    for (int q = 0; q < kCluster; ++q) sum += recv[q][t];
    g[j] = sum - lambda * x[j];
  }
}

struct SmallKernel {
  const void* fn;
  bool ok;  // a cluster of 16 blocks can be resident
};

SmallKernel probe(const void* fn) {
  SmallKernel k = {fn, false};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(kThreads);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  k.ok = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
         cudaOccupancyMaxActiveClusters(&clusters, fn, &cfg) == cudaSuccess && clusters >= 1;
  if (!k.ok) cudaGetLastError();
  return k;
}

}  // namespace

int launch_gradient_small(const float* A, int64_t n, int64_t d, int64_t lda, const float* b, const float* x,
                          float lambda, float* g, cudaStream_t s) {
  if (d > kSmallMaxD || n * (d <= 256 ? 256 : 512) > kSmallElems) return MIHS_ERR_UNSUPPORTED;
  static const SmallKernel k1 = probe((const void*)&gradient_small_kernel<1, 8>);
  static const SmallKernel k2 = probe((const void*)&gradient_small_kernel<2, 8>);
  static const SmallKernel k4 = probe((const void*)&gradient_small_kernel<4, 4>);
  const SmallKernel& k = d <= 128 ? k1 : d <= 256 ? k2 : k4;
  if (!k.ok) return MIHS_ERR_UNSUPPORTED;
  MIHS_CUDA_TRY(cudaFuncSetAttribute(k.fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));  // (per device)
  int n32 = (int)n, d32 = (int)d;
  long long lda64 = lda;
  void* args[] = {(void*)&A, &n32, &d32, &lda64, (void*)&b, (void*)&x, &lambda, (void*)&g};
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(kCluster);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  timing_begin(kTimerApass, s);
  MIHS_CUDA_TRY(cudaLaunchKernelExC(&cfg, k.fn, args));
  timing_end(kTimerApass, s);
  count_launch();
  return MIHS_OK;
}

}  // namespace mihs
