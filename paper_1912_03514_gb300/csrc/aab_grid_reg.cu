// AAb_Solver (Algorithm 5, Section 3.6) fused with the heavy ball and stop
// test of Algorithm 1, for one λ, as a grid of blocks that hold SA in their
// registers: the form for sketches too large for one cluster's registers
// (3076 × 2048 takes 147 blocks of 21 rows) and for the small grids that
// mihs_sketch_set_aab asks for.
//
// Block b keeps rows [b·R, b·R + R), R ≤ 28, its warp w the columns
// 128w … 128w + 127 (and the same 1024 further on), four per lane, so that
//   * the dots w_i = SA_i·v − θ·p_i need one exchange of R partial sums per
//     warp (a transposing butterfly leaves row i's sum in lane i: 31 shuffles)
//     and then live one per lane, like p; θ² = ‖θv‖² is the 32nd of them;
//   * u = SAᵀw needs none: a lane ends with the block's share of its columns
//     and sends it to the columns' owner itself; and θv comes back to the lane
//     that multiplies with it, without shared memory or a barrier.
// What is left is the way through L2, twice a pass.  Every number travels as
// one 64-bit word {value, tag}: the reader polls the word itself until the tag
// is the pass's, so there is no barrier, no fence and no flag to wait for
// before the data (the form with two grid barriers needs a release, an
// arrival, a poll and then the loads).  30 passes at 3076 × 2048: 228 → 144 µs,
// at 1600 × 1024: 196 → 123 µs; what remains per pass is two trips store → L2
// → poll → load (≈ 1.6 K cycles each) and the block's ≈ 2.5 K cycles of work.
// Tags grow from launch to launch (`epoch`), so the words need no clearing
// between the launches of a solve; before it they are cleared.  In a solve of
// more than 2²⁰ steps the tags wrap: a word that any of those steps wrote then
// holds a newer tag, so none passes for the new one.  Every sum over blocks has a fixed order: all blocks compute
// the same scalars and take the same branches.
//
// A word is overwritten only after everyone who polls it has answered with
// something that depends on it: shares of u(k + 1) are sent after all of
// θv(k + 1) has come, which its owners send after all shares of u(k).  The ρ²
// words, which blocks without columns of their own read too, alternate.
#include "aab_kernel.cuh"

namespace mihs {

namespace {

using namespace aabk;

__device__ int g_aab_gridreg_error = 0;

constexpr uint32_t kEpochStep = 4096;  // above twice the passes of a launch (at most min(m, d) ≤ 2048)

struct GridRegParams {
  const void* SA;
  int sa_type;
  int m, d, dp;
  long long ldsa;
  int sa_vec;
  const float* sa_scale;
  int scale_ld;
  int R;               // rows per block
  int cs, cs_log2;     // columns per owner (a power of two, 4 … 256)
  int owners;          // blocks that own columns: ⌈dp/cs⌉ ≤ gridDim.x
  const float* g;
  float lambda, eps;
  int max_passes;
  float* delta;
  int* passes;
  float alpha, beta;
  float* x;
  float* x_prev;
  double* x64;
  double* x_prev64;
  float* x32_shadow;
  double alpha64, beta64;
  SolveCtl* ctl;
  float* hist;
  unsigned long long cond;
  uint32_t* epoch;            // tags used so far
  unsigned long long* rho;    // 2 × 256 words: the blocks' shares of ρ², alternating
  unsigned long long* Z;      // owners · cs words: θv
  unsigned long long* U;      // [owner][block][cs] words: shares of u
};

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

__device__ __forceinline__ unsigned long long word(float v, uint32_t tag) {
  return ((unsigned long long)tag << 32) | __float_as_uint(v);
}
__device__ __forceinline__ float value(unsigned long long w) { return __uint_as_float((uint32_t)w); }
__device__ __forceinline__ bool ready(unsigned long long w, uint32_t tag) { return (uint32_t)(w >> 32) == tag; }

// Each 64-bit word of a pair is read and written whole.
__device__ __forceinline__ void st_word(unsigned long long* p, unsigned long long a) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(a) : "memory");
}
__device__ __forceinline__ void st_words(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long a;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(a) : "l"(p) : "memory");
  return a;
}
__device__ __forceinline__ ulonglong2 ld_words(const unsigned long long* p) {
  ulonglong2 a;
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a.x), "=l"(a.y) : "l"(p) : "memory");
  return a;
}

// Bounded polling: false once the limit has passed.
struct Poll {
  uint64_t t0 = 0;
  uint32_t n = 0;
  __device__ __forceinline__ bool again() {
    if ((++n & 63u) != 0) return true;
    const uint64_t t = global_timer_ns();
    if (t0 == 0) t0 = t;
    return t - t0 <= kWaitLimitNs;
  }
};

// One lane of the warp polls one word until it carries the tag, so that the
// other lanes' loads, of as many words, start when most of them have come.
// (All lanes polling all their words from the start kept L2 busy: 30 passes
// took 177 instead of 144 µs at 3076 × 2048 and 252 instead of 125 at 2000 × 512.)
__device__ __forceinline__ void await_word(const unsigned long long* p, uint32_t tag, bool& ok) {
  if ((threadIdx.x & 31) == 0) {
    Poll poll;
    while (!ready(ld_word(p), tag)) {
      if (!poll.again()) {
        ok = false;
        break;
      }
    }
  }
  __syncwarp();
}

// VC: groups of four columns per lane (dp ≤ 1024·VC); RR: rows held (≤ 28).
template <int VC, int RR>
__global__ void __launch_bounds__(kThreads, 1) aab_gridreg_kernel(const GridRegParams P) {
  const int blk = blockIdx.x, G = gridDim.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int d = P.d, dp = P.dp;
  __shared__ __align__(16) float red[kWarps][32];      // the warps' partial dots
  __shared__ __align__(16) float wsh[kWarps][32];      // w, one copy per warp
  __shared__ __align__(16) float apart[kWarps * 256];  // partial sums of u on the own slice
  __shared__ float bsum[kWarps];
  __shared__ float scal;                 // ρ²
  SolveCtl* ctl = P.ctl;

  // The control block is written by block 0 only: at the end (every block has
  // then read it, or block 0 could not have finished a pass), or when the solve
  // stops, while others may still be reading it.  Those that see `done` leave; to
  // the others the values written are the ones that they have or compute: until
  // ‖g(0)‖ is known gnorm0 is negative, so that gnorm0_known read without the
  // gnorm0 that belongs to it counts for nothing.
  int done = 0, outer = 0, max_outer = 0, g0known = 0, phase = 1, refresh = 1, corr = 0;
  float tol = 0.f, gnorm0 = 0.f, switch_tol = 0.f;
  if (ctl != nullptr) {
    done = ctl->done;
    outer = ctl->outer;
    max_outer = ctl->max_outer;
    g0known = ctl->gnorm0_known;
    tol = ctl->tol;
    gnorm0 = ctl->gnorm0;
    phase = ctl->phase;
    switch_tol = ctl->switch_tol;
    refresh = ctl->refresh;
    corr = ctl->corr;
  }
  done = __syncthreads_or(done);  // (one decision per block)
  if (done) {
    if (P.cond != 0ull && blk == 0 && tid == 0) cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
    return;
  }
  const uint32_t base = *P.epoch;

  // Rows of SA into registers (zero past the block's rows and the columns).
  const int r0 = blk * P.R;
  const int nr = max(0, min(P.m, r0 + P.R) - r0);
  int col[VC];
#pragma unroll
  for (int v = 0; v < VC; ++v) col[v] = 1024 * v + 128 * warp + 4 * lane;
  P2 sa[RR][VC][2];
#pragma unroll
  for (int r = 0; r < RR; ++r) {
#pragma unroll
    for (int v = 0; v < VC; ++v) {
      const int j = col[v];
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < nr && j < dp) {
        const long long o = (long long)(r0 + r) * P.ldsa;
        if (P.sa_type == MIHS_SA_FP32) {
          t = load4_masked(static_cast<const float*>(P.SA) + o, j, d, P.sa_vec != 0);
        } else if (P.sa_type == MIHS_SA_BF16) {
          t = load_sa4<__nv_bfloat16>(static_cast<const __nv_bfloat16*>(P.SA) + o, j, d, true, 1.f);
        } else {
          const float sc = P.sa_scale[(size_t)((r0 + r) >> 7) * P.scale_ld + (j >> 7)];
          t = load_sa4<__nv_fp8_e4m3>(static_cast<const __nv_fp8_e4m3*>(P.SA) + o, j, d, true, sc);
        }
      }
      sa[r][v][0] = p2_pack(t.x, t.y);
      sa[r][v][1] = p2_pack(t.z, t.w);
    }
  }
  // θ₁ v = g: this lane's columns, and the own slice's column of threads < cs
  // (identical sums in every block: same data, same order)
  float gsq = 0.f;
  P2 z[VC][2];
#pragma unroll
  for (int v = 0; v < VC; ++v) {
    const float4 t = col[v] < dp ? load4_masked(P.g, col[v], d, false) : make_float4(0.f, 0.f, 0.f, 0.f);
    z[v][0] = p2_pack(t.x, t.y);
    z[v][1] = p2_pack(t.z, t.w);
    gsq = fmaf(t.x, t.x, fmaf(t.y, t.y, fmaf(t.z, t.z, fmaf(t.w, t.w, gsq))));
  }
  const bool owner = blk < P.owners;
  const int jo = blk * P.cs + tid;  // the thread's own column
  const bool own = owner && tid < P.cs && jo < dp;
  float zo = own && jo < d ? P.g[jo] : 0.f, dv = 0.f, xs = 0.f;
  const float theta1 = sqrtf(block_sum(gsq, bsum));

  if (ctl != nullptr) {  // stop test of Algorithm 1 on ‖g‖ = θ₁
    const float g0 = g0known && gnorm0 >= 0.f ? gnorm0 : theta1;
    if (P.hist != nullptr && blk == 0 && tid == 0 && outer < kHistCap) P.hist[outer] = theta1;
    const bool bad = !(theta1 <= 3.0e38f);
    // A refinement correction's gradient is approximate: it never stops the
    // solve; nor does a refinement solve's plain fp32 gradient (phase 0), whose
    // rounding floor lies above the tolerances refinement is asked for (it
    // can round to zero near the solution): only a compensated one certifies.
    const bool correction = phase == 1 && corr && !refresh;
    const bool conv = tol > 0.f && theta1 <= tol * g0 && !correction && phase != 0;
    const bool capped = outer >= max_outer;
    if (bad || conv || capped) {
      if (blk == 0 && tid == 0) {
        ctl->gnorm = theta1;
        ctl->gnorm0 = g0;
        ctl->gnorm0_known = 1;
        ctl->status = bad ? MIHS_ERR_NUMERIC : (conv ? MIHS_OK : MIHS_NOT_CONVERGED);
        ctl->done = 1;
        if (P.cond != 0ull) cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
      }
      return;
    }
  }

  const int nwc = min(kWarps, (dp + 127) >> 7);  // warps with columns
  const int pc = P.cs >> 1, pc_log2 = P.cs_log2 - 1;
  const int nq = kThreads >> pc_log2;            // readers of a column pair (cs ≤ 256: nq ≥ 2)
  const int pq = tid >> pc_log2, pp = tid & (pc - 1);
  int k = 0;
  bool ok = true, failed = false;
  if (theta1 > 0.f) {
    const float lam = P.lambda;
    float rho = 0.f, rhobar = 0.f, c = 0.f, s = 0.f, phi = 0.f, theta = theta1, inv_theta = 1.0f / theta1, p = 0.f;
    float t = __int_as_float(0x7f800000);  // +inf
    for (uint32_t it = 0;; ++it) {
      const uint32_t tag = base + 1u + it;
      // ---- θv of this pass: the lane's columns from their owners
      if (it > 0) {
        const uint32_t ztag = tag - 1u;
        Poll poll;
        if (128 * warp < dp) await_word(P.Z + 128 * warp, ztag, ok);
        for (;;) {
          ulonglong2 a[VC][2];
          bool all = true;
#pragma unroll
          for (int v = 0; v < VC; ++v) {
            if (col[v] < dp) {
              a[v][0] = ld_words(P.Z + col[v]);
              a[v][1] = ld_words(P.Z + col[v] + 2);
            } else {
              a[v][0] = a[v][1] = make_ulonglong2(word(0.f, ztag), word(0.f, ztag));
            }
          }
#pragma unroll
          for (int v = 0; v < VC; ++v) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              all = all && ready(a[v][h].x, ztag) && ready(a[v][h].y, ztag);
              z[v][h] = p2_pack(value(a[v][h].x), value(a[v][h].y));
            }
          }
          if (all) break;
          if (!poll.again()) {
            ok = false;
            break;
          }
        }
      }
      // ---- partial dots of the warp's columns, row r's sum to lane r; ‖z‖² = θ²
      // is the dot of row 31
      auto dot = [&](int r) {
        P2 acc = 0ull;
#pragma unroll
        for (int v = 0; v < VC; ++v) {
          acc = p2_fma(sa[r][v][0], z[v][0], acc);
          acc = p2_fma(sa[r][v][1], z[v][1], acc);
        }
        const float2 f = p2_unpack(acc);
        return f.x + f.y;
      };
      auto znorm = [&]() {
        P2 acc = 0ull;
#pragma unroll
        for (int v = 0; v < VC; ++v) {
          acc = p2_fma(z[v][0], z[v][0], acc);
          acc = p2_fma(z[v][1], z[v][1], acc);
        }
        const float2 f = p2_unpack(acc);
        return f.x + f.y;
      };
      // (the step over 16 lanes at once: two rows' sums become one register)
      float s0[16];
      const bool up16 = (lane & 16) != 0;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const float lo = i < RR ? dot(i < RR ? i : 0) : 0.f;
        const float hi = i == 15 ? znorm() : (i + 16 < RR ? dot(i + 16 < RR ? i + 16 : 0) : 0.f);
        s0[i] = (up16 ? hi : lo) + __shfl_xor_sync(0xffffffffu, up16 ? lo : hi, 16);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
          const float keep = up ? s0[i + o] : s0[i], send = up ? s0[i] : s0[i + o];
          s0[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      red[warp][lane] = s0[0];
      if (__syncthreads_or(!ok)) {  // a wait ran out in this block
        failed = true;
        break;
      }
      float w = 0.f;
#pragma unroll
      for (int v = 0; v < kWarps; ++v) w += v < nwc ? red[v][lane] : 0.f;
      if (it > 0) {
        norm_of(__shfl_sync(0xffffffffu, w, 31), theta, inv_theta);
        if (!(theta > 0.f)) break;  // invariant subspace: same decision everywhere
      }
      w = lane < RR ? w * inv_theta - theta * p : 0.f;  // rows past nr: zero
      wsh[warp][lane] = w;
      __syncwarp();
      if (warp == kWarps - 1) {  // ρ² share
        const float r2 = warp_sum(w * w);
        if (lane == 0) st_word(P.rho + 256 * (it & 1u) + blk, word(r2, tag));
      }
      // ---- u = Σ w_i·SA_i on the lane's columns, to their owners
      P2 u[VC][2][2];
#pragma unroll
      for (int v = 0; v < VC; ++v) u[v][0][0] = u[v][0][1] = u[v][1][0] = u[v][1][1] = 0ull;
#pragma unroll
      for (int r4 = 0; r4 < RR; r4 += 4) {
        const float4 w4 = *reinterpret_cast<const float4*>(&wsh[warp][r4]);
        const P2 wr[4] = {p2_pack(w4.x, w4.x), p2_pack(w4.y, w4.y), p2_pack(w4.z, w4.z), p2_pack(w4.w, w4.w)};
#pragma unroll
        for (int e = 0; e < 4 && r4 + e < RR; ++e) {
#pragma unroll
          for (int v = 0; v < VC; ++v) {
            u[v][0][e & 1] = p2_fma(sa[r4 + e][v][0], wr[e], u[v][0][e & 1]);
            u[v][1][e & 1] = p2_fma(sa[r4 + e][v][1], wr[e], u[v][1][e & 1]);
          }
        }
      }
#pragma unroll
      for (int v = 0; v < VC; ++v) {
        if (col[v] < dp) {
          const int o = col[v] >> P.cs_log2;
          unsigned long long* dst = P.U + ((size_t)o * G + blk) * P.cs + (col[v] & (P.cs - 1));
          const float2 a0 = p2_unpack(u[v][0][0]), a1 = p2_unpack(u[v][0][1]);
          const float2 b0 = p2_unpack(u[v][1][0]), b1 = p2_unpack(u[v][1][1]);
          st_words(dst, word(a0.x + a1.x, tag), word(a0.y + a1.y, tag));
          st_words(dst + 2, word(b0.x + b1.x, tag), word(b0.y + b1.y, tag));
        }
      }
      // ---- the owners: u on the own slice from all blocks; the last warp of
      // every block: ρ² (in the same rounds of loads)
      {
        float2 a = make_float2(0.f, 0.f);
        float r2 = 0.f;
        const unsigned long long* src = P.U + (size_t)blk * G * P.cs + 2 * pp;
        const int ng = owner && blk * P.cs + 2 * pp < dp ? G : 0;  // (the last owner's slice may be cut)
        const unsigned long long* rsrc = P.rho + 256 * (it & 1u);
        bool want_rho = warp == kWarps - 1;
        const int pw = 2 * (32 * warp & (pc - 1));  // the warp's first pair
        if (owner && blk * P.cs + pw < dp) await_word(P.U + ((size_t)blk * G + G - 1) * P.cs + pw, tag, ok);
        for (int b0 = pq; b0 < ng || want_rho; b0 += 8 * nq) {
          Poll poll;
          ulonglong2 v[8];
          unsigned long long r[8];
          for (;;) {
            bool all = true;
#pragma unroll
            for (int e = 0; e < 8; ++e)
              v[e] = b0 + e * nq < ng ? ld_words(src + (size_t)(b0 + e * nq) * P.cs)
                                      : make_ulonglong2(word(0.f, tag), word(0.f, tag));
            if (want_rho) {
#pragma unroll
              for (int e = 0; e < 8; ++e)
                r[e] = lane + 32 * e < G ? ld_word(rsrc + lane + 32 * e) : word(0.f, tag);
#pragma unroll
              for (int e = 0; e < 8; ++e) all = all && ready(r[e], tag);
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) all = all && ready(v[e].x, tag) && ready(v[e].y, tag);
            if (all) break;
            if (!poll.again()) {
              ok = false;
              break;
            }
          }
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            a.x += value(v[e].x);
            a.y += value(v[e].y);
          }
          if (want_rho) {
#pragma unroll
            for (int e = 0; e < 8; ++e) r2 += value(r[e]);
            want_rho = false;
          }
        }
        // the readers of a pair within the warp, then one sum per warp (or per
        // reader, for pairs wider than a warp) to shared memory
        __syncwarp();
        if (owner) {
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            if (o >= pc) {
              a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
              a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
            }
          }
          if (pc >= 32 || lane < pc)
            *reinterpret_cast<float2*>(&apart[(pc >= 32 ? pq : warp) * P.cs + 2 * pp]) = a;
        }
        if (warp == kWarps - 1) {
          r2 = warp_sum(r2);
          if (lane == 0) scal = r2;
        }
      }
      if (__syncthreads_or(!ok)) {
        failed = true;
        break;
      }
      float inv_rho;
      norm_of(scal, rho, inv_rho);
      const float vo = zo * inv_theta;
      if (owner && tid < P.cs) {  // θ v := SAᵀp − ρ v on the slice, SAᵀp = u/ρ (whole warps, cs ≥ 32; else part of warp 0)
        float us = 0.f;
        const int np = pc >= 32 ? nq : kWarps;
        for (int q = 0; q < np; ++q) us += apart[q * P.cs + tid];
        zo = jo < d ? us * inv_rho - rho * vo : 0.f;
        if (own) st_word(P.Z + jo, word(zo, tag));
      }
      // ---- the recursion's scalars and the slice of d and x, while θv travels
      if (it == 0) {
        rhobar = sqrtf(rho * rho + lam);
        c = rho / rhobar;
        s = sqrtf(lam) / rhobar;
        phi = theta1 / rhobar;
        dv = vo * (1.0f / rhobar);
        xs = phi * dv;
      } else {
        // Eldén's rotation of √λ, the φ recursion and the forward substitution
        const float lambar = sqrtf(lam + (s * theta) * (s * theta));
        const float thetabar = c * theta;
        rhobar = sqrtf(rho * rho + lambar * lambar);
        const float inv_rhobar = 1.0f / rhobar;
        c = rho * inv_rhobar;
        s = lambar * inv_rhobar;
        phi = -phi * thetabar * inv_rhobar;
        dv = (vo - thetabar * dv) * inv_rhobar;
        xs = fmaf(phi, dv, xs);
        t = fabsf(phi * rhobar) / theta1;
        ++k;
      }
      p = w * inv_rho;
      if (!(t >= P.eps && k < P.max_passes && rho > 0.f)) break;  // the same in every block
    }
  }
  if (!(theta1 > 0.f)) {
    // Nothing to do, but block 0 may write the control block only once every
    // block has read it.
    if (tid == 0) st_word(P.rho + blk, word(0.f, base + 1u));
    if (blk == 0) {
      Poll poll;
      for (int b = tid; b < G && ok; b += kThreads)
        while (!ready(ld_word(P.rho + b), base + 1u))
          if (!poll.again()) {
            ok = false;
            break;
          }
    }
    failed = __syncthreads_or(!ok) != 0;
  }
  // (all that write it write the same; it wraps at 2³²)
  if (tid == 0 && (failed || blk == 0)) atomicExch(P.epoch, base + kEpochStep);
  if (failed) {
    if (tid == 0) {
      atomicExch(&g_aab_gridreg_error, MIHS_ERR_TIMEOUT);
      if (ctl != nullptr) {
        ctl->status = MIHS_ERR_TIMEOUT;
        ctl->done = 1;
      }
      if (P.cond != 0ull) cudaGraphSetConditional((cudaGraphConditionalHandle)P.cond, 0u);
    }
    return;
  }

  // Outputs on the owned column slice: Δ and the heavy ball.
  if (own && jo < d) {
    const int j = jo;
    if (P.delta != nullptr) P.delta[j] = xs;
    if (P.x != nullptr) {
      const float xj = P.x[j], xp = P.x_prev[j];
      P.x[j] = xj + P.alpha * xs + P.beta * (xj - xp);
      P.x_prev[j] = xj;
    }
    if (P.x64 != nullptr) {
      const double xj = P.x64[j], xp = P.x_prev64[j];
      const double xn = xj + P.alpha64 * (double)xs + P.beta64 * (xj - xp);
      P.x64[j] = xn;
      P.x_prev64[j] = xj;
      if (P.x32_shadow != nullptr) P.x32_shadow[j] = (float)xn;
    }
  }
  if (blk == 0 && tid == 0) {
    if (P.passes != nullptr) *P.passes = k;
    if (ctl != nullptr) {
      refine_step_update(ctl, phase, refresh, corr, theta1, g0known ? gnorm0 : theta1, tol, switch_tol);
      ctl->outer = outer + 1;
      ctl->inner_total += k;
      ctl->gnorm = theta1;
      if (!g0known) {
        ctl->gnorm0 = theta1;
        ctl->gnorm0_known = 1;
      }
    }
  }
}

using GridRegFn = void (*)(const GridRegParams);

// Rows of SA held, the smallest that fits: a pass costs what is held, not what
// is used.  At one group of columns up to 28 rows, the most that the 32 lanes of
// the dots and groups of four rows leave room for (30 passes, 1000 columns: 120 µs
// with 3040 rows, 20 a block, 129 with 3041 in the kernel of 28).  At two, 24 rows
// spill 0.5 KB a thread and 21 0.2 KB: 2048 columns take 141 µs with 2433 to 3192
// rows (17 to 21 a block), 178 with 3193; in the shared-memory form 220, 228 and
// 232, and 983 with 3600 rows, which are past its shared memory.
GridRegFn gridreg_kernel(int dp, int rows) {
  if (dp > 1024) {
    if (rows <= 8) return aab_gridreg_kernel<2, 8>;
    if (rows <= 16) return aab_gridreg_kernel<2, 16>;
    if (rows <= 21) return aab_gridreg_kernel<2, 21>;
    return aab_gridreg_kernel<2, 24>;
  }
  if (rows <= 8) return aab_gridreg_kernel<1, 8>;
  if (rows <= 16) return aab_gridreg_kernel<1, 16>;
  if (rows <= 20) return aab_gridreg_kernel<1, 20>;
  return aab_gridreg_kernel<1, 28>;
}

constexpr size_t kRhoWords = 512, kMaxSlice = 256;

}  // namespace

size_t aab_gridreg_ws_bytes(int d) {
  const size_t dp = (size_t)round_up(d, 4) + kMaxSlice;
  return 256 + 8 * (kRhoWords + dp + dp * (size_t)num_sms());
}

int aab_gridreg_device_error(int* code) {
  int v = 0, z = 0;
  MIHS_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_aab_gridreg_error, sizeof(int)));
  if (v != 0) MIHS_CUDA_TRY(cudaMemcpyToSymbol(g_aab_gridreg_error, &z, sizeof(int)));
  *code = v;
  return MIHS_OK;
}

int launch_aab_gridreg(const AabLaunch& a, int blocks, void* ws, cudaStream_t s) {
  const int dp = (int)round_up(a.d, 4);
  const int R = (a.m + blocks - 1) / blocks;
  const int G = (a.m + R - 1) / R;
  if (R > (dp > 1024 ? 24 : 28) || G > 256) return MIHS_ERR_UNSUPPORTED;
  GridRegParams P = {};
  P.cs = 4;
  P.cs_log2 = 2;
  while ((int64_t)P.cs * G < dp) {
    P.cs <<= 1;
    ++P.cs_log2;
  }
  if (P.cs > (int)kMaxSlice) return MIHS_ERR_UNSUPPORTED;
  P.owners = (dp + P.cs - 1) / P.cs;
  const GridRegFn fn = gridreg_kernel(dp, R);
  int per_sm = 0;
  MIHS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kThreads, 0));
  if (per_sm < 1 || G > per_sm * num_sms()) return MIHS_ERR_UNSUPPORTED;  // all blocks resident
  P.SA = a.SA;
  P.sa_type = a.sa_type;
  P.m = a.m;
  P.d = a.d;
  P.dp = dp;
  P.ldsa = a.ldsa;
  P.sa_vec = (a.ldsa % 4 == 0 && (reinterpret_cast<uintptr_t>(a.SA) & 15u) == 0) ? 1 : 0;
  P.sa_scale = a.sa_type == MIHS_SA_FP8E4M3 ? a.sa_scale : nullptr;
  P.scale_ld = (dp + 127) / 128;
  P.R = R;
  P.g = a.g;
  P.lambda = a.lambda;
  P.eps = a.eps;
  P.max_passes = a.max_passes;
  P.delta = a.delta;
  P.passes = a.passes;
  P.alpha = a.alpha;
  P.beta = a.beta;
  P.x = a.x;
  P.x_prev = a.x_prev;
  P.x64 = a.x64;
  P.x_prev64 = a.x_prev64;
  P.x32_shadow = a.x32_shadow;
  P.alpha64 = a.alpha64;
  P.beta64 = a.beta64;
  P.ctl = a.ctl;
  P.hist = a.hist;
  P.cond = a.cond;
  P.epoch = static_cast<uint32_t*>(ws);
  P.rho = reinterpret_cast<unsigned long long*>(static_cast<char*>(ws) + 256);
  P.Z = P.rho + kRhoWords;
  P.U = P.Z + dp + kMaxSlice;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  timing_begin(kTimerAab, s);
  MIHS_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, P));
  timing_end(kTimerAab, s);
  count_launch();
  return MIHS_OK;
}

}  // namespace mihs
