// AAb_Solver (Algorithm 5, Section 3.6) as one thread-block cluster with SA in
// registers, fused with the heavy-ball step of Eq. mihs1 and the stop test of
// Algorithm 1, for one λ or for a path (one cluster per λ): the form for every
// sketch that the registers of up to 16 blocks hold.  Rows are padded to 256,
// 512, 1024 or 2048 columns, of which those registers take 2560, 1280, 640 or
// 256 (588 × 1024 takes 16 blocks).
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
//     and the forward substitution are computed; the dots start on θv before θ
//     is known, and θ² is one more of them, taken by every warp from the whole
//     vector rather than exchanged.
// 588 × 1024, 30 passes: 141 → 68 µs, 700 × 256: 177 → 52 µs (the form with SA
// in shared memory swept it twice per pass and crossed two cluster barriers
// and two remote-load round trips).
// Every sum has a fixed order and every block computes the same scalars from
// the same numbers, so all blocks take the same branches.  Quantised SA is
// decoded once, into fp32 registers.
//
// Buffers are reused from pass to pass without further barriers.  θv: a block
// sends its share of u(k + 1) once all its warps have read θv(k) (the block
// barrier of its sweep), and θv(k + 1) goes out only when all shares of
// u(k + 1) have come.  Shares of u and ρ² alternate between two buffers: a
// block may receive those of pass k + 1 while some of its own warps still read
// those of pass k (a peer waits for one copy of the slice's warps, not for
// all), but those of pass k + 2 only after its own share of u(k + 1), which
// all its warps have reached the sweep's barrier for.
#pragma once

#include "aab_kernel.cuh"

namespace mihs {
namespace aabk {
namespace {

// One error word per translation unit (each instantiates one cluster size).
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

// The shape of a cluster: CL blocks, CH chunks of 128 columns (narrower SA is
// zero-padded), all of it known at compile time: a pass has ≈ 550 instructions
// per warp and two warps per scheduler, so every index computed at run time
// lengthens the chain (≈ 6 cycles per instruction; with run-time cluster and
// slice sizes 588 × 1024 took 93 µs).
template <int CL, int CH>
struct RegShape {
  static constexpr int DP = 128 * CH;
  static constexpr int COLS = DP / CL;              // columns of a block's slice
  static constexpr int NGS = COLS / 4;              // groups of four in it
  static constexpr int NG = DP / 4 > kThreads ? DP / 4 / kThreads : 1;   // groups per thread, all columns
  static constexpr int NQ = NGS > kThreads ? NGS / kThreads : 1;         // groups per thread of the slice
  static constexpr int NW = NGS > 32 ? (NGS < kThreads ? NGS / 32 : kWarps) : 1;  // warps that the slice fills
  static constexpr int H = NGS < 32 ? 32 / NGS : 1; // lanes per group of a narrow slice: each sums some ranks
  static constexpr int REPS = kWarps / NW < 4 ? kWarps / NW : 4;  // copies of those warps: each sends to some ranks
  static constexpr int RPL = CL > H ? CL / H : 1;   // ranks summed per lane
  static constexpr int SPL = CL > H * REPS ? CL / (H * REPS) : 1;  // ranks sent to per lane
  // shared memory (floats; every region a multiple of 4)
  static constexpr int z = 0;                       // DP: θv, all columns (written by the owners)
  static constexpr int ubuf = z + DP;               // 2 × CL × COLS: the blocks' shares of u on the own slice
  static constexpr int wpart = ubuf + 2 * DP;       // kWarps × DP: the warps' shares of u
  static constexpr int rbuf = wpart + kWarps * DP;  // 2 × 16: the blocks' shares of ρ²
  static constexpr int red = rbuf + 32;             // kWarps
  static constexpr int bars = red + kWarps;         // two mbarriers
  static constexpr size_t bytes = sizeof(float) * (bars + 4);
};

// Σ of N ≤ 16 values in a fixed order (a broadcast read).
template <int N>
__device__ __forceinline__ float sum_n(const float* p) {
  if constexpr (N < 4) {
    float s = p[0];
#pragma unroll
    for (int i = 1; i < N; ++i) s += p[i];
    return s;
  } else {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < N; i += 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + i);
      s += (a.x + a.y) + (a.z + a.w);
    }
    return s;
  }
}

__device__ __forceinline__ P2 p2_add(P2 a, P2 b) {
  P2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// R: rows per warp (R·CH·4 ≤ 160 registers).
template <int CL, int CH, int R>
__global__ void __launch_bounds__(kThreads, 1) aab_reg_kernel(const AabParams P, int sa_type) {
  using S = RegShape<CL, CH>;
  constexpr int DP = S::DP, NG = S::NG, NQ = S::NQ;
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
  float* z = sm + S::z;
  float* ubuf = sm + S::ubuf;
  float* wpart = sm + S::wpart;
  float* rbuf = sm + S::rbuf;
  float* red = sm + S::red;
  uint64_t* barA = reinterpret_cast<uint64_t*>(sm + S::bars);
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
  if (tid == 0) {
    mbar_init(barA, 1);
    mbar_init(barB, 1);
    fence_mbar_init();
  }
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
  for (int j = tid; j < DP; j += kThreads) {
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
  // their ρ² shares; all of θv.
  constexpr uint32_t bytesA = CL * (16u * S::NGS + 4u), bytesB = 4u * DP;
  const uint32_t a_barA = smem_u32(barA), a_barB = smem_u32(barB);
  // Where this thread's column group(s) of u go: owner block and place there.
  uint32_t u_dst[NG], u_bar[NG];
#pragma unroll
  for (int q = 0; q < NG; ++q) {
    const int gq = min(tid + kThreads * q, DP / 4 - 1);
    const uint32_t o = (uint32_t)(gq / S::NGS);
    u_dst[q] = mapa_u32(smem_u32(ubuf) + 16u * (rank * (uint32_t)S::NGS + (uint32_t)(gq % S::NGS)), o);
    u_bar[q] = mapa_u32(a_barA, o);
  }
  const uint32_t r_dst = mapa_u32(smem_u32(rbuf) + 4u * rank, (uint32_t)(lane % CL));
  const uint32_t r_bar = mapa_u32(a_barA, (uint32_t)(lane % CL));
  // Slice ownership of this thread: group(s) gsl + 256·q.  The H lanes of a
  // group sum the shares of RPL ranks each; every copy of the slice's warps
  // does, and lane share `sh` of the H·REPS sends to SPL ranks.
  const int rep = warp / S::NW;
  const int gsl = S::H > 1 ? lane % S::NGS : (warp % S::NW) * 32 + lane;
  const int hsh = S::H > 1 ? lane / S::NGS : 0, sh = rep * S::H + hsh;
  const bool slice_warp = rep < S::REPS;
  const bool sums = S::H <= CL || hsh < CL, sends = sh * S::SPL < CL;
  const float* u_src = ubuf + (size_t)(hsh * S::RPL) * S::COLS + 4 * gsl;
  const uint32_t z_src = smem_u32(z) + 4u * rank * S::COLS + 16u * (uint32_t)gsl;
  float4 zo[NQ], dv[NQ], xs[NQ];  // own slice: θv, d, x
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    zo[q] = *reinterpret_cast<const float4*>(z + rank * S::COLS + 4 * (gsl + kThreads * q));
    dv[q] = xs[q] = make_float4(0.f, 0.f, 0.f, 0.f);
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
      P2 s2[R + 1];  // the rows' dots, and ‖z‖² = θ²
#pragma unroll
      for (int r = 0; r <= R; ++r) s2[r] = 0ull;
#pragma unroll
      for (int ch = 0; ch < CH; ++ch) {
        const int j = 4 * lane + 128 * ch;
        const ulonglong2 zz = *reinterpret_cast<const ulonglong2*>(z + j);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          s2[r] = p2_fma(sa[r][ch][0], zz.x, s2[r]);
          s2[r] = p2_fma(sa[r][ch][1], zz.y, s2[r]);
        }
        s2[R] = p2_fma(zz.x, zz.x, s2[R]);
        s2[R] = p2_fma(zz.y, zz.y, s2[R]);
      }
      float w[R + 1];
#pragma unroll
      for (int r = 0; r <= R; ++r) {
        const float2 f = p2_unpack(s2[r]);
        w[r] = f.x + f.y;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int r = 0; r <= R; ++r) w[r] += __shfl_xor_sync(0xffffffffu, w[r], o);
      }
      if (it > 0) {  // θ from the whole vector, the same in every warp of every block
        norm_of(w[R], theta, inv_theta);
        if (!(theta > 0.f)) break;  // invariant subspace
      }
      float rsq = 0.f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        w[r] = w[r] * inv_theta - theta * p[r];  // rows past nr: zero
        rsq = fmaf(w[r], w[r], rsq);
      }
      // ---- u = Σ w_i·SA_i, chunk by chunk into the warp's share
      float* wp = wpart + warp * DP;
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
        *reinterpret_cast<ulonglong2*>(wp + j) = make_ulonglong2(u0, u1);
      }
      if (lane == 0) red[warp] = rsq;
      if (!__syncthreads_and(ok)) {  // a wait of this block has run out
        left = true;
        break;
      }
#pragma unroll
      for (int q = 0; q < NG; ++q) {
        const int gq = tid + kThreads * q;
        if (DP / 4 >= kThreads || gq < DP / 4) {
          ulonglong2 a[kWarps];
#pragma unroll
          for (int v = 0; v < kWarps; ++v) a[v] = *reinterpret_cast<const ulonglong2*>(wpart + v * DP + 4 * gq);
          const P2 lo = p2_add(p2_add(p2_add(a[0].x, a[1].x), p2_add(a[2].x, a[3].x)),
                               p2_add(p2_add(a[4].x, a[5].x), p2_add(a[6].x, a[7].x)));
          const P2 hi = p2_add(p2_add(p2_add(a[0].y, a[1].y), p2_add(a[2].y, a[3].y)),
                               p2_add(p2_add(a[4].y, a[5].y), p2_add(a[6].y, a[7].y)));
          const float2 l = p2_unpack(lo), h = p2_unpack(hi);
          st_async_f4(u_dst[q] + 4u * DP * par, make_float4(l.x, l.y, h.x, h.y), u_bar[q]);
        }
      }
      if (warp == kWarps - 1 && lane < CL)
        st_async_f1(r_dst + 64u * par, sum_n<kWarps>(red), r_bar);
      // ---- exchange A: u on the own slice, ρ²
      if (!mbar_wait_cluster(barA, par)) ok = false;
      if (tid == 0) mbar_arrive_expect_tx(barA, bytesA);
      P2 us[NQ][2];
      if (slice_warp) {  // u on the slice: ranks in order, then the lanes of a group
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          ulonglong2 a[S::RPL];
#pragma unroll
          for (int e = 0; e < S::RPL; ++e)
            a[e] = *reinterpret_cast<const ulonglong2*>(u_src + DP * par + e * S::COLS + 4 * kThreads * q);
          us[q][0] = a[0].x;
          us[q][1] = a[0].y;
#pragma unroll
          for (int e = 1; e < S::RPL; ++e) {
            us[q][0] = p2_add(us[q][0], a[e].x);
            us[q][1] = p2_add(us[q][1], a[e].y);
          }
          if (!sums) us[q][0] = us[q][1] = 0ull;
#pragma unroll
          for (int o = S::NGS; o < 32; o <<= 1) {
            us[q][0] = p2_add(us[q][0], __shfl_xor_sync(0xffffffffu, us[q][0], o));
            us[q][1] = p2_add(us[q][1], __shfl_xor_sync(0xffffffffu, us[q][1], o));
          }
        }
      }
      float inv_rho;
      norm_of(sum_n<CL>(rbuf + 16 * par), rho, inv_rho);
      float4 vo[NQ];
      if (slice_warp) {  // θ v := SAᵀp − ρ v on the slice, SAᵀp = u/ρ
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          const float2 ul = p2_unpack(us[q][0]), uh = p2_unpack(us[q][1]);
          vo[q] = make_float4(zo[q].x * inv_theta, zo[q].y * inv_theta, zo[q].z * inv_theta, zo[q].w * inv_theta);
          zo[q].x = ul.x * inv_rho - rho * vo[q].x;
          zo[q].y = ul.y * inv_rho - rho * vo[q].y;
          zo[q].z = uh.x * inv_rho - rho * vo[q].z;
          zo[q].w = uh.y * inv_rho - rho * vo[q].w;
          if (sends) {
#pragma unroll
            for (int e = 0; e < S::SPL; ++e) {
              const uint32_t to = (uint32_t)(sh * S::SPL + e);
              st_async_f4(mapa_u32(z_src + 16u * kThreads * q, to), zo[q], mapa_u32(a_barB, to));
            }
          }
        }
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
          for (int q = 0; q < NQ; ++q) {
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
          for (int q = 0; q < NQ; ++q) {
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
      // ---- exchange B: θv (also awaited before leaving: nothing may
      // still be on its way to a block that exits)
      if (!mbar_wait_cluster(barB, par)) ok = false;
      if (tid == 0) mbar_arrive_expect_tx(barB, bytesB);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) continue;  // to the block's next barrier, which sends every warp out
      if (!(t >= P.eps && k < P.max_passes && rho > 0.f)) break;  // the same in every block
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
  if (rep == 0 && hsh == 0) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const float xv[4] = {xs[q].x, xs[q].y, xs[q].z, xs[q].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = (int)rank * S::COLS + 4 * (gsl + kThreads * q) + e;
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

// Rows per warp of the kernels: all steps for one block; only the upper half
// for more (fewer rows would have fitted half the blocks).
constexpr int reg_step(int ch) { return ch <= 2 ? 4 : (ch <= 4 ? 2 : 1); }
constexpr int reg_max(int ch) { return ch == 16 ? 2 : 5 * reg_step(ch); }

template <int CL, int CH>
RegKernel reg_kernel_rows(int r) {
  constexpr int st = reg_step(CH);
  const size_t smem = RegShape<CL, CH>::bytes;
  if constexpr (CH == 16) {
    if constexpr (CL == 1) {
      if (r <= 1) return {(const void*)aab_reg_kernel<CL, CH, 1>, smem};
    }
    return {(const void*)aab_reg_kernel<CL, CH, 2>, smem};
  } else {
    if constexpr (CL == 1) {
      if (r <= st) return {(const void*)aab_reg_kernel<CL, CH, st>, smem};
      if (r <= 2 * st) return {(const void*)aab_reg_kernel<CL, CH, 2 * st>, smem};
    }
    if (r <= 3 * st) return {(const void*)aab_reg_kernel<CL, CH, 3 * st>, smem};
    if (r <= 4 * st) return {(const void*)aab_reg_kernel<CL, CH, 4 * st>, smem};
    return {(const void*)aab_reg_kernel<CL, CH, 5 * st>, smem};
  }
}

template <int CL>
RegKernel reg_kernel_cl(int m, int dp) {
  const int ch = (dp + 127) / 128, chp = ch <= 2 ? 2 : (ch <= 4 ? 4 : (ch <= 8 ? 8 : 16));
  const int r = ((m + CL - 1) / CL + kWarps - 1) / kWarps;
  if (r > reg_max(chp)) return {nullptr, 0};
  switch (chp) {
    case 2: return reg_kernel_rows<CL, 2>(r);
    case 4: return reg_kernel_rows<CL, 4>(r);
    case 8: return reg_kernel_rows<CL, 8>(r);
    default: return reg_kernel_rows<CL, 16>(r);
  }
}

}  // namespace
}  // namespace aabk
}  // namespace mihs
