// AAb_Solver (Algorithm 5, Section 3.6) as one thread-block cluster with SA in
// registers, fused with the heavy-ball step of Eq. mihs1 and the stop test of
// Algorithm 1: the form for every sketch that the registers of up to 16
// blocks hold (m·d ≲ 650 K elements: 588 × 1024 takes 16 blocks).
//
// A pass is a chain of dependent steps (a product with SA, one with SAᵀ, two
// norms), so what bounds it is the length of that chain, not any throughput.
// It is kept short by
//   * SA in registers: warp w of a block keeps rows w, w + 8, … (R of them,
//     lane ℓ the columns 4ℓ + 128c) for the whole solve, so the sweep
//         w_i = SA_i·v − θ·p_i,  u = Σ w_i·SA_i,  ρ² = Σ w_i²
//     reads nothing but v; p and w live in registers too;
//   * pushing instead of pulling: each block stores its share of u straight
//     into the shared memory of the columns' owners (st.async, completion
//     counted in bytes on the owner's mbarrier), and each owner its slice of
//     the next v to every block: two one-way trips per pass, no cluster
//     barrier and no remote load;
//   * one block barrier per pass (the eight warps' shares of u);
//   * scalars off the chain: v is sent before the rotation, the φ recursion
//     and the forward substitution are computed, and the dots start on θv
//     before θ is known.
// 588 × 1024, 30 passes: 141 → 78 µs (2.4 µs per pass; the form with SA in
// shared memory swept it twice per pass and crossed two cluster barriers and
// two remote-load round trips, 4.6 µs).
// Every sum has a fixed order and every block computes the same scalars from
// the same numbers, so all blocks take the same branches.  Quantised SA is
// decoded once, into fp32 registers.
//
// Buffers are reused from pass to pass without further barriers: a block
// sends its share of u(k + 1) only after all of v(k + 1) has arrived, v(k + 1)
// only after all of u(k); so by the time a buffer is written again everyone
// who had to read it has sent something that depends on it.  (The ρ² slots
// are read by warps that send nothing in between: they alternate.)
#include "aab_kernel.cuh"

namespace mihs {
namespace aabk {
namespace {

__device__ int g_aab_reg_error = 0;

__device__ __forceinline__ uint32_t mapa_u32(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}

// Stores into a block of the cluster that count their bytes on a barrier there.
__device__ __forceinline__ void st_async_f4(uint32_t dst, float4 v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void st_async_f1(uint32_t dst, float v, uint32_t bar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];" ::"r"(dst), "f"(v), "r"(bar)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// As mbar_wait, for data that other blocks of the cluster have stored.
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((i & 255u) == 0 && global_timer_ns() - t0 > kWaitLimitNs) return false;
  }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

typedef unsigned long long P2;  // two fp32 values, packed
__device__ __forceinline__ P2 p2_fma(P2 a, P2 b, P2 c) {
  P2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ P2 p2_pack(float x, float y) {
  P2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 p2_unpack(P2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Shared memory of a block (floats; every region a multiple of 4).
struct RegSmem {
  int z, ubuf, wpart, rbuf, tbuf, red, bars, total;
};
__host__ __device__ inline RegSmem reg_smem(int dp, int cl, int cols_per) {
  RegSmem L;
  L.z = 0;                            // dp: θv, all columns (written by the owners)
  L.ubuf = L.z + dp;                  // cl × cols_per: the blocks' shares of u on the own slice
  L.wpart = L.ubuf + cl * cols_per;   // kWarps × dp: the warps' shares of u
  L.rbuf = L.wpart + kWarps * dp;     // 2 × 16: the blocks' shares of ρ²
  L.tbuf = L.rbuf + 32;               // 16: shares of θ² (one per block and slice warp)
  L.red = L.tbuf + 16;                // kWarps + staging
  L.bars = L.red + kWarps;            // two mbarriers
  L.total = L.bars + 4;
  return L;
}

// Σ of up to 16 values in a fixed order (a broadcast read; values past `cnt` are zero).
__device__ __forceinline__ float sum16(const float* p, int cnt) {
  const float4* q = reinterpret_cast<const float4*>(p);
  float4 a = q[0];
  float s = (a.x + a.y) + (a.z + a.w);
  if (cnt > 4) {
    const float4 b = q[1];
    s += (b.x + b.y) + (b.z + b.w);
  }
  if (cnt > 8) {
    const float4 c = q[2], e = q[3];
    s += ((c.x + c.y) + (c.z + c.w)) + ((e.x + e.y) + (e.z + e.w));
  }
  return s;
}

// CH: chunks of 128 columns; R: rows per warp (R·CH·4 ≤ 160 registers).
template <int CH, int R>
__global__ void __launch_bounds__(kThreads, 1) aab_reg_kernel(const AabParams P, int sa_type, int cl) {
  constexpr int NG = CH > 8 ? 2 : 1;  // column groups (16 bytes) per thread: dp/4 ≤ 256·NG
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int d = P.d, dp = P.dp;
  const int li = P.path ? (int)blockIdx.y : 0;
  const float* g_in = P.g + (long long)li * P.path_ldg;
  SolveCtl* ctl_ = P.ctl != nullptr ? P.ctl + li : nullptr;
  float* x_ = P.x != nullptr ? P.x + (long long)li * P.path_ldx : nullptr;
  float* xprev_ = P.x_prev != nullptr ? P.x_prev + (long long)li * P.path_ldg : nullptr;
  float* delta_ = P.path ? nullptr : P.delta;
  int* passes_ = P.path ? nullptr : P.passes;
  float* hist_ = P.path ? nullptr : P.hist;
  const float lam = P.path ? P.ps.lam[li] : P.lambda;
  const float alpha_ = P.path ? P.ps.alpha[li] : P.alpha;
  const float beta_ = P.path ? P.ps.beta[li] : P.beta;

  extern __shared__ float4 smem4[];
  float* sm = reinterpret_cast<float*>(smem4);
  const RegSmem L = reg_smem(dp, cl, P.cols_per);
  float* z = sm + L.z;
  float* ubuf = sm + L.ubuf;
  float* wpart = sm + L.wpart;
  float* rbuf = sm + L.rbuf;
  float* tbuf = sm + L.tbuf;
  float* red = sm + L.red;
  uint64_t* barA = reinterpret_cast<uint64_t*>(sm + L.bars);
  uint64_t* barB = barA + 1;

  // Solve-mode control block: every block reads it before the cluster
  // barrier below; rank 0 writes it only after.
  int done = 0, outer = 0, max_outer = 0, g0known = 0, phase = 1, refresh = 1, corr = 0;
  float tol = 0.f, gnorm0 = 0.f, switch_tol = 0.f;
  if (ctl_ != nullptr) {
    done = ctl_->done;
    outer = ctl_->outer;
    max_outer = ctl_->max_outer;
    g0known = ctl_->gnorm0_known;
    tol = ctl_->tol;
    gnorm0 = ctl_->gnorm0;
    phase = ctl_->phase;
    switch_tol = ctl_->switch_tol;
    refresh = ctl_->refresh;
    corr = ctl_->corr;
  }
  // Column slice of this block: groups (4 columns) [G0, G0 + ng), the first
  // ngr of which lie below dp.  ng is a power of two; with fewer than 32
  // groups the lanes of warp 0 share them, H lanes per group.
  const int ng = P.cols_per >> 2;
  const int G0 = (int)rank * ng, groups = dp >> 2;
  const int ngr = max(0, min(groups - G0, ng));
  const int nw = max(1, min(kWarps, ng >> 5));  // warps that own groups
  const int H = ng < 32 ? 32 / ng : 1;
  if (tid == 0) {
    mbar_init(barA, 1);
    mbar_init(barB, 1);
    fence_mbar_init();
  }
  if (tid < 48) rbuf[tid] = 0.f;  // rbuf and tbuf: slots past the cluster's stay zero
  __syncthreads();
  cluster_arrive();
  if (done) {
    cluster_wait();
    if (P.cond != 0ull && !P.path && rank == 0 && tid == 0)
      cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
    return;
  }

  // Rows of SA into registers; θ₁v = g into shared memory.
  const int r0 = (int)rank * P.rpc;
  const int nr = max(0, min(P.m, r0 + P.rpc) - r0);
  P2 sa[R][CH][2];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = warp + kWarps * r;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int j = 4 * lane + 128 * c;
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < nr && j < dp) {
        const long long o = (long long)(r0 + i) * P.ldsa;
        if (sa_type == MIHS_SA_FP32) {
          t = load4_masked(static_cast<const float*>(P.SA) + o, j, d, P.sa_vec != 0);
        } else if (sa_type == MIHS_SA_BF16) {
          t = load_sa4<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(P.SA) + o, j, d, true, 1.f);
        } else {
          const float sc = P.sa_scale[(size_t)((r0 + i) >> 7) * P.scale_ld + c];
          t = load_sa4<__nv_fp8_e4m3>(static_cast<const __nv_fp8_e4m3*>(P.SA) + o, j, d, true, sc);
        }
      }
      sa[r][c][0] = p2_pack(t.x, t.y);
      sa[r][c][1] = p2_pack(t.z, t.w);
    }
  }
  float gsq = 0.f;
  for (int j = tid; j < dp; j += kThreads) {
    const float gj = j < d ? g_in[j] : 0.f;
    z[j] = gj;
    gsq = fmaf(gj, gj, gsq);
  }
  const float theta1 = sqrtf(block_sum(gsq, red));
  cluster_wait();  // every block has read the control block and set up its barriers

  if (ctl_ != nullptr) {  // stop test of Algorithm 1 on ‖g‖ = θ₁
    const float g0 = g0known ? gnorm0 : theta1;
    if (hist_ != nullptr && rank == 0 && tid == 0 && outer < kHistCap) hist_[outer] = theta1;
    const bool bad = !(theta1 <= 3.0e38f);
    // A refinement correction's gradient is approximate: it never stops the
    // solve; nor does a refinement solve's plain fp32 gradient (phase 0), whose
    // rounding floor lies above the tolerances refinement is asked for (it
    // can round to zero near the solution): only a compensated one certifies.
    const bool correction = phase == 1 && corr && !refresh;
    const bool conv = tol > 0.f && theta1 <= tol * g0 && !correction && phase != 0;
    const bool capped = outer >= max_outer;
    if (rank == 0 && tid == 0) refine_step_update(ctl_, phase, refresh, corr, theta1, g0, tol, switch_tol);
    if (bad || conv || capped) {
      if (rank == 0 && tid == 0) {
        ctl_->gnorm = theta1;
        ctl_->gnorm0 = g0;
        ctl_->gnorm0_known = 1;
        ctl_->status = bad ? MIHS_ERR_NUMERIC : (conv ? MIHS_OK : MIHS_NOT_CONVERGED);
        ctl_->done = 1;
        if (P.path) {
          if (atomicAdd(P.path_ndone, 1) + 1 == P.ps.nl) {  // the last λ of the path to stop
            *P.path_all_done = 1;
            if (P.cond != 0ull) cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
          }
        } else if (P.cond != 0ull) {
          cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
        }
      }
      return;  // nothing has been sent to this block
    }
  }

  // Bytes that arrive here per exchange: the blocks' u on the own slice and
  // their ρ² shares; all of θv and the slice warps' θ² shares.
  const uint32_t bytesA = (uint32_t)cl * (16u * (uint32_t)ngr + 4u);
  const uint32_t bytesB = 16u * (uint32_t)groups + 4u * (uint32_t)(cl * nw);
  const uint32_t a_barA = smem_u32(barA), a_barB = smem_u32(barB);
  const uint32_t a_z = smem_u32(z), a_tbuf = smem_u32(tbuf);
  // Where this thread's column group(s) of u go: owner block and place there.
  uint32_t u_dst[NG], u_bar[NG];
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    const int gq = tid + kThreads * q;
    const uint32_t own = (uint32_t)((4 * gq) >> P.cols_log2);
    const uint32_t o = own < (uint32_t)cl ? own : 0u;
    u_dst[q] = mapa_u32(smem_u32(ubuf) + 4u * (rank * (uint32_t)P.cols_per + (uint32_t)(4 * gq - (int)o * P.cols_per)), o);
    u_bar[q] = mapa_u32(a_barA, o);
  }
  // Slice ownership of this thread: group(s) gsl + 256·q with ranks
  // [h·cl/H …) summed by lane share h (H > 1: warp 0 only).
  const int gsl = H > 1 ? (lane & (ng - 1)) : tid;
  const int hsh = H > 1 ? lane / ng : 0;
  const bool slice_warp = H > 1 ? warp == 0 : warp < nw;
  const int hr0 = hsh * cl / H, hr1 = (hsh + 1) * cl / H;  // ranks this lane sums and sends to
  float4 zo[NG], dv[NG], xs[NG];  // own slice: θv, d, x
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    zo[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    dv[q] = xs[q] = zo[q];
    if (slice_warp && gsl + kThreads * q < ngr) zo[q] = *reinterpret_cast<const float4*>(z + 4 * (G0 + gsl + kThreads * q));
  }

  int k = 0;
  bool ok = true, left = false;
  if (theta1 > 0.f) {
    if (tid == 0) {
      mbar_arrive_expect_tx(barA, bytesA);
      mbar_arrive_expect_tx(barB, bytesB);
    }
    float p[R];
#pragma unroll
    for (int r = 0; r < R; ++r) p[r] = 0.f;
    float rho = 0.f, rhobar = 0.f, c = 0.f, s = 0.f, phi = 0.f, theta = theta1, inv_theta = 1.0f / theta1;
    float t = __int_as_float(0x7f800000);  // +inf
    bool first = true;
    for (uint32_t it = 0;; ++it) {
      const uint32_t par = it & 1u;
      // ---- sweep: w = SA·v − θp with v = z/θ, this warp's rows
      P2 s2[R];
#pragma unroll
      for (int r = 0; r < R; ++r) s2[r] = 0ull;
#pragma unroll
      for (int ch = 0; ch < CH; ++ch) {
        const int j = 4 * lane + 128 * ch;
        const ulonglong2 zz = *reinterpret_cast<const ulonglong2*>(z + (j < dp ? j : 0));  // SA is zero past dp
#pragma unroll
        for (int r = 0; r < R; ++r) {
          s2[r] = p2_fma(sa[r][ch][0], zz.x, s2[r]);
          s2[r] = p2_fma(sa[r][ch][1], zz.y, s2[r]);
        }
      }
      float w[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float2 f = p2_unpack(s2[r]);
        w[r] = f.x + f.y;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) w[r] += __shfl_xor_sync(0xffffffffu, w[r], o);
      }
      float rsq = 0.f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        w[r] = w[r] * inv_theta - theta * p[r];  // rows past nr: zero
        rsq = fmaf(w[r], w[r], rsq);
      }
      // ---- u = Σ w_i·SA_i, chunk by chunk into the warp's share
      float* wp = wpart + (size_t)warp * dp;
#pragma unroll
      for (int ch = 0; ch < CH; ++ch) {
        const int j = 4 * lane + 128 * ch;
        P2 u0 = 0ull, u1 = 0ull;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const P2 wr = p2_pack(w[r], w[r]);
          u0 = p2_fma(sa[r][ch][0], wr, u0);
          u1 = p2_fma(sa[r][ch][1], wr, u1);
        }
        if (j < dp) *reinterpret_cast<ulonglong2*>(wp + j) = make_ulonglong2(u0, u1);
      }
      if (lane == 0) red[warp] = rsq;
      if (!__syncthreads_and(ok)) {  // a wait of this block has run out
        left = true;
        break;
      }
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const int gq = tid + kThreads * q;
        if (gq < groups) {
          float4 a[kWarps];
#pragma unroll
          for (int v = 0; v < kWarps; ++v) a[v] = *reinterpret_cast<const float4*>(wpart + (size_t)v * dp + 4 * gq);
          float4 u;
          u.x = ((a[0].x + a[1].x) + (a[2].x + a[3].x)) + ((a[4].x + a[5].x) + (a[6].x + a[7].x));
          u.y = ((a[0].y + a[1].y) + (a[2].y + a[3].y)) + ((a[4].y + a[5].y) + (a[6].y + a[7].y));
          u.z = ((a[0].z + a[1].z) + (a[2].z + a[3].z)) + ((a[4].z + a[5].z) + (a[6].z + a[7].z));
          u.w = ((a[0].w + a[1].w) + (a[2].w + a[3].w)) + ((a[4].w + a[5].w) + (a[6].w + a[7].w));
          st_async_f4(u_dst[q], u, u_bar[q]);
        }
      }
      if (warp == kWarps - 1 && lane < cl) {
        const float r2 = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
        st_async_f1(mapa_u32(smem_u32(rbuf + 16 * par + rank), (uint32_t)lane), r2, mapa_u32(a_barA, (uint32_t)lane));
      }
      // ---- exchange A: u on the own slice, ρ²
      if (!mbar_wait_cluster(barA, par)) ok = false;
      if (tid == 0) mbar_arrive_expect_tx(barA, bytesA);
      rho = sqrtf(sum16(rbuf + 16 * par, cl));
      const float inv_rho = 1.0f / rho;
      float4 vo[NG];
      if (slice_warp) {  // θ v := SAᵀp − ρ v on the slice, SAᵀp = u/ρ
        float zsq = 0.f;
#pragma unroll
        for (int q = 0; q < NG; ++q) {
          const int gs = gsl + kThreads * q;
          vo[q] = make_float4(zo[q].x * inv_theta, zo[q].y * inv_theta, zo[q].z * inv_theta, zo[q].w * inv_theta);
          float4 u = make_float4(0.f, 0.f, 0.f, 0.f);
          if (gs < ngr) {
#pragma unroll 8
            for (int b = hr0; b < hr1; ++b) {
              const float4 a = *reinterpret_cast<const float4*>(ubuf + b * P.cols_per + 4 * gs);
              u.x += a.x;
              u.y += a.y;
              u.z += a.z;
              u.w += a.w;
            }
          }
          for (int o = ng; o < 32; o <<= 1) {  // the H lanes of a group (none for ng ≥ 32)
            u.x += __shfl_xor_sync(0xffffffffu, u.x, o);
            u.y += __shfl_xor_sync(0xffffffffu, u.y, o);
            u.z += __shfl_xor_sync(0xffffffffu, u.z, o);
            u.w += __shfl_xor_sync(0xffffffffu, u.w, o);
          }
          zo[q].x = u.x * inv_rho - rho * vo[q].x;
          zo[q].y = u.y * inv_rho - rho * vo[q].y;
          zo[q].z = u.z * inv_rho - rho * vo[q].z;
          zo[q].w = u.w * inv_rho - rho * vo[q].w;
          if (gs < ngr) {
            for (int b = hr0; b < hr1; ++b)
              st_async_f4(mapa_u32(a_z + 16u * (uint32_t)(G0 + gs), (uint32_t)b), zo[q], mapa_u32(a_barB, (uint32_t)b));
            if (hsh == 0)
              zsq = fmaf(zo[q].x, zo[q].x, fmaf(zo[q].y, zo[q].y, fmaf(zo[q].z, zo[q].z, fmaf(zo[q].w, zo[q].w, zsq))));
          }
        }
        zsq = warp_sum(zsq);
        if (lane < cl)
          st_async_f1(mapa_u32(a_tbuf + 4u * (rank * (uint32_t)nw + (uint32_t)warp), (uint32_t)lane), zsq,
                      mapa_u32(a_barB, (uint32_t)lane));
      }
      // ---- the recursion's scalars and the slice of d and x, while θv travels
      if (first) {
        rhobar = sqrtf(rho * rho + lam);
        c = rho / rhobar;
        s = sqrtf(lam) / rhobar;
        phi = theta1 / rhobar;
        const float inv = 1.0f / rhobar;
        if (slice_warp) {
#pragma unroll
          for (int q = 0; q < NG; ++q) {
            dv[q] = make_float4(vo[q].x * inv, vo[q].y * inv, vo[q].z * inv, vo[q].w * inv);
            xs[q] = make_float4(phi * dv[q].x, phi * dv[q].y, phi * dv[q].z, phi * dv[q].w);
          }
        }
        first = false;
      } else {
        // Eldén's rotation of √λ into the bidiagonal, then the φ recursion
        // and the forward-substitution update (Section 3.6), on the slice.
        const float lambar = sqrtf(lam + (s * theta) * (s * theta));
        const float thetabar = c * theta;
        rhobar = sqrtf(rho * rho + lambar * lambar);
        const float inv_rhobar = 1.0f / rhobar;
        c = rho * inv_rhobar;
        s = lambar * inv_rhobar;
        phi = -phi * thetabar * inv_rhobar;
        if (slice_warp) {
#pragma unroll
          for (int q = 0; q < NG; ++q) {
            dv[q].x = (vo[q].x - thetabar * dv[q].x) * inv_rhobar;
            dv[q].y = (vo[q].y - thetabar * dv[q].y) * inv_rhobar;
            dv[q].z = (vo[q].z - thetabar * dv[q].z) * inv_rhobar;
            dv[q].w = (vo[q].w - thetabar * dv[q].w) * inv_rhobar;
            xs[q].x = fmaf(phi, dv[q].x, xs[q].x);
            xs[q].y = fmaf(phi, dv[q].y, xs[q].y);
            xs[q].z = fmaf(phi, dv[q].z, xs[q].z);
            xs[q].w = fmaf(phi, dv[q].w, xs[q].w);
          }
        }
        t = fabsf(phi * rhobar) / theta1;
        ++k;
      }
#pragma unroll
      for (int r = 0; r < R; ++r) p[r] = w[r] * inv_rho;
      // ---- exchange B: θv and θ² (also awaited before leaving: nothing may
      // still be on its way to a block that exits)
      if (!mbar_wait_cluster(barB, par)) ok = false;
      if (tid == 0) mbar_arrive_expect_tx(barB, bytesB);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) continue;  // to the block's next barrier, which sends every warp out
      if (!(t >= P.eps && k < P.max_passes && rho > 0.f)) break;  // the same in every block
      theta = sqrtf(sum16(tbuf, cl * nw));
      if (!(theta > 0.f)) break;  // invariant subspace: same decision everywhere
      inv_theta = 1.0f / theta;
    }
    // Warps that left by the tests above meet, at this barrier, any warp of
    // the block whose wait ran out (its barrier is the one in the sweep).
    if (!left) left = !__syncthreads_and(ok);
  }
  if (left && tid == 0) {  // a wait ran out here (and then in every peer)
    atomicExch(&g_aab_reg_error, MIHS_ERR_TIMEOUT);
    if (ctl_ != nullptr) {
      ctl_->status = MIHS_ERR_TIMEOUT;
      if (atomicExch(&ctl_->done, 1) == 0 && P.path && atomicAdd(P.path_ndone, 1) + 1 == P.ps.nl) {
        *P.path_all_done = 1;
        if (P.cond != 0ull) cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
      }
    }
  }

  // Outputs: each block writes its column slice.
  if (slice_warp && hsh == 0) {
#pragma unroll
    for (int q = 0; q < NG; ++q) {
      if (gsl + kThreads * q >= ngr) continue;
      const float xv[4] = {xs[q].x, xs[q].y, xs[q].z, xs[q].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = 4 * (G0 + gsl + kThreads * q) + e;
        if (j >= d) continue;
        const float dj = xv[e];
        if (delta_ != nullptr) delta_[j] = dj;
        if (x_ != nullptr) {
          const float xj = x_[j], xp = xprev_[j];
          x_[j] = xj + alpha_ * dj + beta_ * (xj - xp);
          xprev_[j] = xj;
        }
        if (P.x64 != nullptr) {
          const double xj = P.x64[j], xp = P.x_prev64[j];
          const double xn = xj + P.alpha64 * (double)dj + P.beta64 * (xj - xp);
          P.x64[j] = xn;
          P.x_prev64[j] = xj;
          if (P.x32_shadow != nullptr) P.x32_shadow[j] = (float)xn;
        }
      }
    }
  }
  if (rank == 0 && tid == 0) {
    if (passes_ != nullptr) *passes_ = k;
    if (ctl_ != nullptr) {
      ctl_->outer = outer + 1;
      ctl_->inner_total += k;
      ctl_->gnorm = theta1;
      if (!g0known) {
        ctl_->gnorm0 = theta1;
        ctl_->gnorm0_known = 1;
      }
    }
  }
  __syncwarp();
  cluster_arrive();  // nobody exits while a peer may still store into it
  cluster_wait();
}

using RegKernelFn = void (*)(const AabParams, int, int);

template <int CH>
RegKernelFn reg_kernel_for_rows(int r) {
  constexpr int step = CH <= 2 ? 4 : (CH <= 4 ? 2 : 1);  // kernels for R = step, 2·step, …
  if constexpr (CH == 16) return r <= 1 ? aab_reg_kernel<16, 1> : aab_reg_kernel<16, 2>;
  else {
    if (r <= step) return aab_reg_kernel<CH, step>;
    if (r <= 2 * step) return aab_reg_kernel<CH, 2 * step>;
    if (r <= 3 * step) return aab_reg_kernel<CH, 3 * step>;
    if (r <= 4 * step) return aab_reg_kernel<CH, 4 * step>;
    return aab_reg_kernel<CH, 5 * step>;
  }
}

RegKernelFn reg_kernel(int ch, int r) {
  if (ch <= 2) return reg_kernel_for_rows<2>(r);
  if (ch <= 4) return reg_kernel_for_rows<4>(r);
  if (ch <= 8) return reg_kernel_for_rows<8>(r);
  return reg_kernel_for_rows<16>(r);
}

}  // namespace
}  // namespace aabk

using namespace aabk;

int aab_reg_device_error(int* code) {
  int v = 0, zero = 0;
  MIHS_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_aab_reg_error, sizeof(int)));
  if (v != 0) MIHS_CUDA_TRY(cudaMemcpyToSymbol(g_aab_reg_error, &zero, sizeof(int)));
  *code = v;
  return MIHS_OK;
}

int aabk::aab_reg_rows(int m, int cl, int dp) {
  const int ch = (dp + 127) / 128;
  const int chp = ch <= 2 ? 2 : (ch <= 4 ? 4 : (ch <= 8 ? 8 : 16));
  const int rpc = (m + cl - 1) / cl;
  const int r = (rpc + kWarps - 1) / kWarps;
  return r * chp * 4 <= (chp == 16 ? 128 : 160) ? r : 0;
}

const void* aabk::aab_reg_fn(int dp, int r) { return (const void*)reg_kernel((dp + 127) / 128, r); }

size_t aabk::aab_reg_smem(int dp, int cl, int cols_per) { return sizeof(float) * (size_t)reg_smem(dp, cl, cols_per).total; }

}  // namespace mihs
