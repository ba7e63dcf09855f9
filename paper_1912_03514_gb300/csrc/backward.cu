// Gradients of the ridge solution x(A, b, λ) = (AᵀA + λI)⁻¹Aᵀb with respect
// to its inputs, given the adjoint v = (AᵀA + λI)⁻¹ ḡ of an upstream gradient
// ḡ = ∂L/∂x.  Differentiating H x = Aᵀb (H = AᵀA + λI) gives
//   dx = H⁻¹(dAᵀ r − Aᵀ dA x + Aᵀ db − dλ x),  r = b − Ax,
// so dL = ḡᵀdx = rᵀdA v − (Av)ᵀdA x + (Av)ᵀdb − (xᵀv) dλ, i.e.
//   ∂L/∂A = r vᵀ − (Av) xᵀ,  ∂L/∂b = Av,  ∂L/∂λ = −xᵀv.
// (The paper does not differentiate the solve; this is the standard adjoint
// of a linear system with a symmetric matrix, so the same M-IHS solver with
// the same sketch computes v.)
//
// One pass over A: each warp takes whole rows, forms r_i = b_i − A_i·x and
// q_i = A_i·v with warp reductions, and writes the row A-gradient
// r_i v − q_i x and db_i = q_i.  The pass reads A once and writes dA once:
// 8·n·d + 8·n bytes, HBM-bound.
#include "internal.h"

namespace mihs {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;

__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// dλ = −Σ_j x_j v_j, accumulated in fp64 in a fixed order (one block).
__global__ void __launch_bounds__(kThreads) neg_dot_kernel(const float* __restrict__ x,
                                                           const float* __restrict__ v, int d,
                                                           double* __restrict__ out) {
  __shared__ double red[kWarps];
  double s = 0.0;
  for (int j = threadIdx.x; j < d; j += kThreads) s += (double)x[j] * (double)v[j];
  s = warp_sum_f64(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += red[w];
    *out = -t;
  }
}

__device__ __forceinline__ float dot4(const float4 a, const float4 b) {
  return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}

// Columns j … j + 3 of a vector of d elements (zero past it; any alignment).
__device__ __forceinline__ float4 vec4(const float* v, int j, int d) {
  return make_float4(j < d ? v[j] : 0.f, j + 1 < d ? v[j + 1] : 0.f, j + 2 < d ? v[j + 2] : 0.f,
                     j + 3 < d ? v[j + 3] : 0.f);
}

// Rows of A are 16-byte aligned (the interface asks for that); here those of dA, x
// and v are too, and d is a multiple of 4.  Lane `l` holds columns 4(32c + l) …
// 4(32c + l) + 3 of chunk c < CH, CH = ⌈d/128⌉; x and v live in registers
// (CH ≤ 4) or shared memory (CH ≥ 8: held in registers they cap the CTA count per
// SM and, measured at 2²⁰×1024, the pass ran at 0.57 of HBM bandwidth instead of
// 0.97).  RW rows per warp iteration give each warp RW·CH independent 16-byte
// loads in flight.
template <int CH, int RW>
__global__ void __launch_bounds__(kThreads)
    backward_rows_vec_kernel(const float* __restrict__ A, long long n, int d, long long lda,
                             const float* __restrict__ b, const float* __restrict__ x,
                             const float* __restrict__ v, float* __restrict__ dA, long long ldda,
                             float* __restrict__ db) {
  constexpr bool XS = CH >= 8;
  __shared__ float4 xs4[XS ? CH * 32 : 1], vs4[XS ? CH * 32 : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int d4 = d >> 2;
  float4 xr[XS ? 1 : CH], vr[XS ? 1 : CH];
  const float4* x4 = reinterpret_cast<const float4*>(x);
  const float4* v4 = reinterpret_cast<const float4*>(v);
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (XS) {
    for (int i = threadIdx.x; i < CH * 32; i += kThreads) {
      xs4[i] = i < d4 ? x4[i] : z4;
      vs4[i] = i < d4 ? v4[i] : z4;
    }
    __syncthreads();
  } else {
#pragma unroll
    for (int c = 0; c < (XS ? 1 : CH); ++c) {
      const int i = c * 32 + lane;
      xr[c] = i < d4 ? x4[i] : z4;
      vr[c] = i < d4 ? v4[i] : z4;
    }
  }
  const long long nw = (long long)gridDim.x * kWarps;
  for (long long r0 = ((long long)blockIdx.x * kWarps + warp) * RW; r0 < n; r0 += nw * RW) {
    float4 a[RW][CH];
#pragma unroll
    for (int k = 0; k < RW; ++k) {
      const long long row = r0 + k;
      const float4* Ar = reinterpret_cast<const float4*>(A + (row < n ? row : 0) * lda);
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int i = c * 32 + lane;
        a[k][c] = (row < n && i < d4) ? __ldg(Ar + i) : z4;
      }
    }
    float rr[RW], qq[RW];
#pragma unroll
    for (int k = 0; k < RW; ++k) {
      float sx0 = 0.f, sx1 = 0.f, sv0 = 0.f, sv1 = 0.f;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const float4 xc = XS ? xs4[c * 32 + lane] : xr[XS ? 0 : c];
        const float4 vc = XS ? vs4[c * 32 + lane] : vr[XS ? 0 : c];
        if (c & 1) {
          sx1 += dot4(a[k][c], xc);
          sv1 += dot4(a[k][c], vc);
        } else {
          sx0 += dot4(a[k][c], xc);
          sv0 += dot4(a[k][c], vc);
        }
      }
      const long long row = r0 + k;
      const float bi = (row < n && b != nullptr) ? __ldg(b + row) : 0.f;
      rr[k] = bi - warp_sum(sx0 + sx1);
      qq[k] = warp_sum(sv0 + sv1);
    }
#pragma unroll
    for (int k = 0; k < RW; ++k) {
      const long long row = r0 + k;
      if (row >= n) break;
      if (db != nullptr && lane == 0) db[row] = qq[k];
      if (dA == nullptr) continue;
      float4* Dr = reinterpret_cast<float4*>(dA + row * ldda);
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int i = c * 32 + lane;
        if (i < d4) {
          const float4 xc = XS ? xs4[i] : xr[XS ? 0 : c];
          const float4 vc = XS ? vs4[i] : vr[XS ? 0 : c];
          float4 o;
          o.x = fmaf(rr[k], vc.x, -qq[k] * xc.x);
          o.y = fmaf(rr[k], vc.y, -qq[k] * xc.y);
          o.z = fmaf(rr[k], vc.z, -qq[k] * xc.z);
          o.w = fmaf(rr[k], vc.w, -qq[k] * xc.w);
          __stcs(Dr + i, o);  // streamed: dA is written once and not re-read here
        }
      }
    }
  }
}

// Rows of dA that start anywhere (d = 1001, say, with dense rows).  A row whose
// start lies s floats before a 16-byte boundary is stored from there on in
// 16-byte groups, each made of a lane's last 4 − s columns and the next lane's
// first s (at most three shuffles per group), its first s columns by lane 0.
// 200003 rows of 1001 columns: 297 µs with one element per lane throughout (below,
// bound by the store requests), 253 here; of 97, 68 and 46; of 511, 165 and 142.
template <int CH, int RW>
__global__ void __launch_bounds__(kThreads)
    backward_rows_kernel(const float* __restrict__ A, long long n, int d, long long lda,
                         const float* __restrict__ b, const float* __restrict__ x,
                         const float* __restrict__ v, float* __restrict__ dA, long long ldda,
                         float* __restrict__ db) {
  constexpr bool XS = CH >= 5;
  __shared__ float4 xs4[XS ? CH * 32 : 1], vs4[XS ? CH * 32 : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int groups = (d + 3) >> 2, d4 = d >> 2;  // groups of four columns, and those that are full
  float4 xr[XS ? 1 : CH], vr[XS ? 1 : CH];
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (XS) {
    for (int i = threadIdx.x; i < CH * 32; i += kThreads) {
      xs4[i] = vec4(x, 4 * i, d);
      vs4[i] = vec4(v, 4 * i, d);
    }
    __syncthreads();
  } else {
#pragma unroll
    for (int c = 0; c < (XS ? 1 : CH); ++c) {
      const int i = c * 32 + lane;
      xr[c] = vec4(x, 4 * i, d);
      vr[c] = vec4(v, 4 * i, d);
    }
  }
  const long long nw = (long long)gridDim.x * kWarps;
  for (long long r0 = ((long long)blockIdx.x * kWarps + warp) * RW; r0 < n; r0 += nw * RW) {
    float4 a[RW][CH];
#pragma unroll
    for (int k = 0; k < RW; ++k) {
      const long long row = r0 + k;
      const float* Ar = A + (row < n ? row : 0) * lda;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const int i = c * 32 + lane;
        a[k][c] = (row < n && i < d4) ? __ldg(reinterpret_cast<const float4*>(Ar) + i) : z4;
        if (c == CH - 1 && row < n && i == d4 && i < groups) {  // the ragged last group
          a[k][c].x = __ldg(Ar + 4 * i);
          if (4 * i + 1 < d) a[k][c].y = __ldg(Ar + 4 * i + 1);
          if (4 * i + 2 < d) a[k][c].z = __ldg(Ar + 4 * i + 2);
        }
      }
    }
    float rr[RW], qq[RW];
#pragma unroll
    for (int k = 0; k < RW; ++k) {
      float sx0 = 0.f, sx1 = 0.f, sv0 = 0.f, sv1 = 0.f;
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        const float4 xc = XS ? xs4[c * 32 + lane] : xr[XS ? 0 : c];
        const float4 vc = XS ? vs4[c * 32 + lane] : vr[XS ? 0 : c];
        if (c & 1) {
          sx1 += dot4(a[k][c], xc);
          sv1 += dot4(a[k][c], vc);
        } else {
          sx0 += dot4(a[k][c], xc);
          sv0 += dot4(a[k][c], vc);
        }
      }
      const long long row = r0 + k;
      const float bi = (row < n && b != nullptr) ? __ldg(b + row) : 0.f;
      rr[k] = bi - warp_sum(sx0 + sx1);
      qq[k] = warp_sum(sv0 + sv1);
    }
#pragma unroll
    for (int k = 0; k < RW; ++k) {
      const long long row = r0 + k;
      if (row >= n) break;
      if (db != nullptr && lane == 0) db[row] = qq[k];
      if (dA == nullptr) continue;
      float* Dr = dA + row * ldda;
      const int s = (int)((0u - (uint32_t)(uintptr_t)Dr) >> 2) & 3;  // floats before the first boundary
      auto grad = [&](int c) {
        const int i = c * 32 + lane;
        const float4 xc = XS ? xs4[i] : xr[XS ? 0 : c];
        const float4 vc = XS ? vs4[i] : vr[XS ? 0 : c];
        float4 o;
        o.x = fmaf(rr[k], vc.x, -qq[k] * xc.x);
        o.y = fmaf(rr[k], vc.y, -qq[k] * xc.y);
        o.z = fmaf(rr[k], vc.z, -qq[k] * xc.z);
        o.w = fmaf(rr[k], vc.w, -qq[k] * xc.w);
        return o;
      };
      float4 cur = grad(0);
      if (s > 0 && lane == 0) {
        Dr[0] = cur.x;
        if (s > 1 && d > 1) Dr[1] = cur.y;
        if (s > 2 && d > 2) Dr[2] = cur.z;
      }
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        float4 next = z4, o = cur;
        if (c + 1 < CH) next = grad(c + 1);
        if (s > 0) {  // uniform across the warp
          const int from = (lane + 1) & 31;
          const float nx = __shfl_sync(0xffffffffu, lane == 0 ? next.x : cur.x, from);
          if (s == 1) {
            o = make_float4(cur.y, cur.z, cur.w, nx);
          } else {
            const float ny = __shfl_sync(0xffffffffu, lane == 0 ? next.y : cur.y, from);
            if (s == 2) {
              o = make_float4(cur.z, cur.w, nx, ny);
            } else {
              const float nz = __shfl_sync(0xffffffffu, lane == 0 ? next.z : cur.z, from);
              o = make_float4(cur.w, nx, ny, nz);
            }
          }
        }
        const int j = 4 * (c * 32 + lane) + s;
        if (j + 4 <= d) {
          __stcs(reinterpret_cast<float4*>(Dr + j), o);
        } else if (j < d) {
          Dr[j] = o.x;
          if (j + 1 < d) Dr[j + 1] = o.y;
          if (j + 2 < d) Dr[j + 2] = o.z;
        }
        cur = next;
      }
    }
  }
}

// Any d, lda, ldda: x and v in shared memory, two sweeps over each row (the
// second one hits L1/L2), one element per lane: the form for rows off 16 bytes
// whose last chunk of 128 columns is nearly empty.
__global__ void __launch_bounds__(kThreads)
    backward_rows_scalar_kernel(const float* __restrict__ A, long long n, int d, long long lda,
                         const float* __restrict__ b, const float* __restrict__ x,
                         const float* __restrict__ v, float* __restrict__ dA, long long ldda,
                         float* __restrict__ db) {
  __shared__ float xs[kMaxD], vs[kMaxD];
  for (int j = threadIdx.x; j < d; j += kThreads) {
    xs[j] = x[j];
    vs[j] = v[j];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long nw = (long long)gridDim.x * kWarps;
  for (long long row = (long long)blockIdx.x * kWarps + warp; row < n; row += nw) {
    const float* Ar = A + row * lda;
    float sx = 0.f, sv = 0.f;
    for (int j = lane; j < d; j += 32) {
      const float aij = __ldg(Ar + j);
      sx = fmaf(aij, xs[j], sx);
      sv = fmaf(aij, vs[j], sv);
    }
    const float r = (b != nullptr ? __ldg(b + row) : 0.f) - warp_sum(sx);
    const float q = warp_sum(sv);
    if (db != nullptr && lane == 0) db[row] = q;
    if (dA != nullptr) {
      float* Dr = dA + row * ldda;
      for (int j = lane; j < d; j += 32) Dr[j] = fmaf(r, vs[j], -q * xs[j]);
    }
  }
}

template <typename K>
int launch_rows(K kernel, long long n, const void* const* args, cudaStream_t s) {
  int per_sm = 0;
  MIHS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreads, 0));
  if (per_sm < 1) per_sm = 1;
  const long long want = (n + kWarps - 1) / kWarps;
  long long grid = (long long)num_sms() * per_sm;
  if (grid > want) grid = want;
  if (grid < 1) grid = 1;
  MIHS_CUDA_TRY(cudaLaunchKernel((const void*)kernel, dim3((unsigned)grid), dim3(kThreads),
                                 const_cast<void**>(args), 0, s));
  count_launch();
  return MIHS_OK;
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

int launch_backward_grads(const float* A, int64_t n, int64_t d, int64_t lda, const float* b, const float* x,
                          const float* v, float* dA, int64_t ldda, float* db, double* dlambda, cudaStream_t s) {
  if (dlambda != nullptr) {
    neg_dot_kernel<<<1, kThreads, 0, s>>>(x, v, (int)d, dlambda);
    MIHS_CHECK_LAUNCH();
    count_launch();
  }
  if ((dA == nullptr && db == nullptr) || n == 0) return MIHS_OK;
  long long n_ = n, lda_ = lda, ldda_ = dA != nullptr ? ldda : 0;
  int d_ = (int)d;
  const void* args[] = {&A, &n_, &d_, &lda_, &b, &x, &v, &dA, &ldda_, &db};
  const int ch = (int)((d + 127) / 128);
  const bool aligned = d % 4 == 0 && aligned16(x) && aligned16(v) &&
                       (dA == nullptr || (ldda % 4 == 0 && aligned16(dA)));
  timing_begin(kTimerBackward, s);
  int rc;
  if (aligned) {
    if (ch <= 1) rc = launch_rows(backward_rows_vec_kernel<1, 4>, n, args, s);
    else if (ch <= 2) rc = launch_rows(backward_rows_vec_kernel<2, 4>, n, args, s);
    else if (ch <= 4) rc = launch_rows(backward_rows_vec_kernel<4, 2>, n, args, s);
    else if (ch <= 8) rc = launch_rows(backward_rows_vec_kernel<8, 2>, n, args, s);
    else rc = launch_rows(backward_rows_vec_kernel<16, 1>, n, args, s);
  } else {
    // The shuffled stores pay for whole chunks of 128 columns, so they take rows
    // whose last chunk is mostly there: of the 200003 × d below, elements / shuffles
    // took 57 / 72 µs at d = 130, 70 / 78 at 210 and 105 / 82 at 225, 126 / 137 at 450 and 130
    // / 130 at 480, 94 / 94 at 321, 193 / 187 at 705, 258 / 246 at 961; but 177 / 190 at
    // 638, 244 / 251 at 895 and 276 / 360 at 1537.
    const int last = (int)d - 128 * (ch - 1);  // columns of the last chunk
    if (last < (ch == 2 || ch == 4 ? 96 : 64)) rc = launch_rows(backward_rows_scalar_kernel, n, args, s);
    else if (ch == 1) rc = launch_rows(backward_rows_kernel<1, 4>, n, args, s);
    else if (ch == 2) rc = launch_rows(backward_rows_kernel<2, 4>, n, args, s);
    else if (ch == 3) rc = launch_rows(backward_rows_kernel<3, 2>, n, args, s);
    else if (ch == 4) rc = launch_rows(backward_rows_kernel<4, 2>, n, args, s);
    else if (ch == 6) rc = launch_rows(backward_rows_kernel<6, 2>, n, args, s);
    else if (ch == 8) rc = launch_rows(backward_rows_kernel<8, 2>, n, args, s);
    else rc = launch_rows(backward_rows_scalar_kernel, n, args, s);
  }
  timing_end(kTimerBackward, s);
  return rc;
}

}  // namespace mihs
