// Gradient A-pass for a λ-path: G[l] = Aᵀ(b − A·X[l]) for up to 16 iterates
// X[l] (one per λ_l) in ONE pass over A (Algorithm 1's gradient step, run for
// every λ of the path at once; A, b and the sketch are shared by the path,
// only λ, the iterate and β/α differ).  Streaming A once for 16 iterates
// turns the pass from HBM-bound (1 FMA per 4 bytes, two for the pass) into
// FP32-bound (32 FMAs per element).
//
// Both contractions, R = A·Xᵀ and G += Rᵀ·A, run over the same columns of A: a
// lane keeps 8 columns (4 up to d = 128) of KI iterates of X and of G in
// registers and takes 2 rows of A at a time, which it reads from shared memory
// once for both.  FMAs are packed over column pairs (f32x2): half the issue
// slots.  The 2·KI sums of 2 rows are added over the lanes in 2·KI exchanges (9
// for KI = 4).  So that a lane keeps and sends the same registers as all others,
// it holds the two rows in the order of its lane bit 4 and the iterates with
// their halves swapped by lane bit 3 (X, G and r alike).
//
// Work split: CW warps side by side cover the columns (d ≤ 256·CW), kh warps the
// iterates, KI each (groups past nl are not computed); these CW·kh warps are a
// team, and the block's teams take stages of 4 rows in turn, each from a ring of
// its own, which its warps fill in turn with bulk copies (a warp for that alone
// would cost the others registers).  The CW warps of the same iterates add their
// sums through shared memory behind one barrier of their own, which they reach
// with the G of the two rows before still to be added between their exchanges
// and the barrier, so the exchange hides under FMAs.
//
// KI = 8 halves the reads of A and r per FMA, but its 250 registers leave two
// warps per scheduler; KI = 4 has four.  With 16 iterates KI = 4 took 103 µs and
// KI = 8 80 (65536×512, this kernel alone); with up to 4 it is 53 against 62 for
// the whole call, half of the other being zeros.  Hence KI = 4 for nl ≤ 4.
//
// What bounds it now: latency.  FMAs fill 40 % of their pipe at two warps per
// scheduler; shared memory is a third busy.  Before, X and r were read from
// shared memory for every row by all threads, which the block crossed two
// barriers per 16 rows for, whatever nl.  Whole call, before → after, with 16 / 8 /
// 4 iterates: 65536×512 101 → 91 / 61 / 57 µs, 65536×1024 153 → 151 / 100 / –,
// 60000×700 140 → 134 / 83 / 67, 200000×129 141 → 127 / 81 / 68, 100000×256
// 96 → 76 / 51 / 45, 262144×64 114 → 100 / 66 / 49.  Column warps cover 256 columns
// and iterates go by 8, so just past such a step half of both is padding: there,
// with more than 8 iterates, the form of apass_path_smem.cu is the faster one.
//
// Per-block column sums go to partials[block][l][j]; a finalize kernel adds
// them in a fixed order and subtracts λ_l·X[l].
#include "internal.h"

namespace mihs {

namespace {

constexpr int kL = 16;        // iterates per pass
constexpr int kStageRows = 4;
constexpr int kMaxStages = 16;  // per team
constexpr int kRefillLag = 2;   // a stage is filled again two stages after it was read
constexpr int kRingBytes = 192 << 10;  // three stages a team at least, which the lag needs
constexpr int kPathMaxD = 1024;

__device__ int g_apass_path_error = 0;

__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Warps that an SM holds: X and G of 8 iterates and 8 columns leave two per
// scheduler (of 4 columns: three), of 4 iterates four.
__host__ __device__ constexpr int path_max_warps(int ki, int ni) { return ki == 4 ? 16 : ni == 1 ? 12 : 8; }

// Floats of the rings, which are reused for the sums over the teams; then come
// the warps' sums of two pairs of rows, their residuals of two, the barriers.
__host__ __device__ inline size_t path_ring_floats(int teams, int its, int dpad, int stages) {
  const size_t ring = (size_t)teams * stages * kStageRows * dpad, red = (size_t)teams * its * dpad;
  return ring > red || teams == 1 ? ring : red;
}

__host__ inline size_t path_smem_bytes(int teams, int warps, int its, int dpad, int stages) {
  return 4 * (path_ring_floats(teams, its, dpad, stages) + 128 * (size_t)warps) + 16 * (size_t)teams * stages;
}

template <int KI, int CW, int NI>
__global__ void __launch_bounds__(path_max_warps(KI, NI) * 32, 1)
apass_path_kernel(const float* __restrict__ A, int n, int d, long long lda, const float* __restrict__ b,
                  const float* __restrict__ X, long long ldx, int nl, float* __restrict__ partials, int dpad,
                  int rows_per_cta, int kh, int stages, const int* __restrict__ all_done) {
  if (all_done != nullptr && *all_done) return;  // every λ of the path has stopped
  const int team_warps = CW * kh, teams = path_max_warps(KI, NI) / team_warps, warps = teams * team_warps;
  extern __shared__ __align__(128) float sm[];
  float* ring = sm;                                               // [team][stage][4 rows][dpad]
  float* psum = sm + path_ring_floats(teams, KI * kh, dpad, stages);  // [2][warp][32]
  float* res = psum + 2 * warps * 32;                             // [warp][2][row][iterate][2 copies]
  uint64_t* bars = reinterpret_cast<uint64_t*>(res + 2 * warps * 32);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long r0 = (long long)blockIdx.x * rows_per_cta;
  const int nr = (int)max(0LL, min((long long)n - r0, (long long)rows_per_cta));  // the block's rows
  const int nst = (nr + kStageRows - 1) / kStageRows;
  A += r0 * lda;
  if (b != nullptr) b += r0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < teams * stages; ++s) {
      mbar_init(&bars[2 * s], 1);                   // full
      mbar_init(&bars[2 * s + 1], team_warps);   // empty
    }
    fence_mbar_init();
  }
  __syncthreads();

  const int team = warp / team_warps, wt = warp % team_warps;
  const int quarter = wt / CW, cw = wt % CW;
  // the team's stages are team, team + kTeams, … of the block's, in its own ring
  const int mine = nst > team ? (nst - team + teams - 1) / teams : 0;
  float* tring = ring + (size_t)team * stages * kStageRows * dpad;
  uint64_t* tbars = bars + 2 * team * stages;
  // the four rows of stage q into a slot: lanes 0–3 copy one each
  auto fill = [&](int q, int slot) {
    const int row0 = (team + q * teams) * kStageRows;
    const int rows = min(kStageRows, nr - row0);
    uint64_t* bar = &tbars[2 * slot];
    if (lane == 0) mbar_arrive_expect_tx(bar, (uint32_t)rows * (uint32_t)dpad * 4u);
    __syncwarp();
    if (lane < rows)
      bulk_copy_g2s(tring + (slot * kStageRows + lane) * dpad, A + (long long)(row0 + lane) * lda,
                    (uint32_t)dpad * 4u, bar);
  };
  if (wt == 0)
    for (int q = 0; q < min(mine, stages); ++q) fill(q, q);
  const int l0 = quarter * KI;
  int col[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) col[i] = (cw * NI + i) * 128 + 4 * lane;
  const int fr = lane >> 4, fk = (lane & 8) != 0 ? KI / 2 : 0;  // this lane's order of rows and iterates
  unsigned long long x2[NI][2][KI], g2[NI][2][KI];  // column pairs; iterate l0 + (k ^ fk)
#pragma unroll
  for (int i = 0; i < NI; ++i)
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int k = 0; k < KI; ++k) {
        const int j = col[i] + 2 * p, l = l0 + (k ^ fk);
        const float* xr = X + (long long)l * ldx + j;
        x2[i][p][k] = pack2(l < nl && j < d ? xr[0] : 0.f, l < nl && j + 1 < d ? xr[1] : 0.f);
        g2[i][p][k] = 0ull;
      }
  // some lane of the warp has the last, partial group of columns
  const bool ragged = (d & 3) != 0 && d > cw * NI * 128 && d < (cw + 1) * NI * 128;
  float* rw = res + warp * 64;                   // [2][row][iterate][2 copies]
  rw[32 + lane] = 0.f;
  unsigned long long a2[2][2][NI][2];            // [rows 0–1 or 2–3 of the stage][row ^ fr][..][column pair]
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int i = 0; i < NI; ++i) a2[u][r][i][0] = a2[u][r][i][1] = 0ull;
  // Offsets of this lane's rows of a pair in A, and of its rows and halves in r.
  const int arow[2] = {fr * dpad, (1 - fr) * dpad};
  const float* rrow[2][2];
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int h = 0; h < 2; ++h) rrow[r][h] = rw + 2 * KI * (r ^ fr) + 2 * ((h * KI / 2) ^ fk);
  // G += of one of the two rows in a2[u] for one half of the iterates
  auto add_g = [&](int u, int r, int h) {
#pragma unroll
    for (int k2 = 0; k2 < KI / 2; k2 += 2) {
      const int k = h * KI / 2 + k2;
      const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(rrow[r][h] + 32 * u + 2 * k2);
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        g2[i][0][k] = fma2(a2[u][r][i][0], v.x, g2[i][0][k]);
        g2[i][1][k] = fma2(a2[u][r][i][1], v.x, g2[i][1][k]);
        g2[i][0][k + 1] = fma2(a2[u][r][i][0], v.y, g2[i][0][k + 1]);
        g2[i][1][k + 1] = fma2(a2[u][r][i][1], v.y, g2[i][1][k + 1]);
      }
    }
  };
  // b of this lane's row of either pair of a stage, a stage ahead
  float bn[2];
  auto load_b = [&](int row) {
    bn[0] = b != nullptr && row < nr ? __ldg(b + row) : 0.f;
    bn[1] = b != nullptr && row + 2 < nr ? __ldg(b + row + 2) : 0.f;
  };
  load_b(team * kStageRows + fr);
  __syncwarp();

  bool dead = false;  // a wait ran out: keep to the barriers, wait no more
  int s = 0, turn = 0;  // slot; the warp of the team that fills
  uint32_t ph = 0;
  for (int q = 0; q < mine; ++q) {
    const int row0 = (team + q * teams) * kStageRows;
    const int rows = min(kStageRows, nr - row0);
    const float bv[2] = {bn[0], bn[1]};
    load_b(row0 + teams * kStageRows + fr);
    if (lane == 0 && b != nullptr && row0 + 128 < nr) asm volatile("prefetch.global.L2 [%0];" ::"l"(b + row0 + 128));
    if (!dead && !mbar_wait(&tbars[2 * s], ph, kWaitLimitNs)) {
      atomicExch(&g_apass_path_error, MIHS_ERR_TIMEOUT);
      dead = true;
    }
    __syncwarp();
    const float* st = tring + s * kStageRows * dpad;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float* su = st + 2 * u * dpad;
      // Columns from d on stay zero, whatever the memory behind a row holds.
      if (rows == kStageRows) {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int i = 0; i < NI; ++i)
            if (col[i] < d) {
              const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(su + arow[r] + col[i]);
              a2[u][r][i][0] = v.x;
              a2[u][r][i][1] = v.y;
            }
      } else {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            ulonglong2 v = make_ulonglong2(0ull, 0ull);
            if (2 * u + (r ^ fr) < rows && col[i] < d)
              v = *reinterpret_cast<const ulonglong2*>(su + arow[r] + col[i]);
            a2[u][r][i][0] = v.x;
            a2[u][r][i][1] = v.y;
          }
      }
      if (ragged) {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            const float2 lo = unpack2(a2[u][r][i][0]), hi = unpack2(a2[u][r][i][1]);
            a2[u][r][i][0] = pack2(lo.x, col[i] + 1 < d ? lo.y : 0.f);
            a2[u][r][i][1] = pack2(col[i] + 2 < d ? hi.x : 0.f, col[i] + 3 < d ? hi.y : 0.f);
          }
      }
      if (u == 1) {
        __syncwarp();
        if (lane == 0) mbar_arrive(&tbars[2 * s + 1]);  // the stage is in registers
        if (q >= kRefillLag && q - kRefillLag + stages < mine && wt == turn) {
          // the slot of stage q − 2, once the whole team has read it
          const bool wrapped = s < kRefillLag;
          const int old = wrapped ? s - kRefillLag + stages : s - kRefillLag;
          if (!dead && !mbar_wait(&tbars[2 * old + 1], wrapped ? ph ^ 1u : ph, kWaitLimitNs)) {
            atomicExch(&g_apass_path_error, MIHS_ERR_TIMEOUT);
            dead = true;
          }
          if (!__any_sync(0xffffffffu, dead)) fill(q - kRefillLag + stages, old);
        }
        if (++turn == team_warps) turn = 0;
      }
      // R over this lane's columns
      float p[2 * KI];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        unsigned long long t[KI];
#pragma unroll
        for (int k = 0; k < KI; ++k) t[k] = mul2(a2[u][r][0][0], x2[0][0][k]);
#pragma unroll
        for (int k = 0; k < KI; ++k) t[k] = fma2(a2[u][r][0][1], x2[0][1][k], t[k]);
        if constexpr (NI == 2) {
#pragma unroll
          for (int k = 0; k < KI; ++k) t[k] = fma2(a2[u][r][1][0], x2[1][0][k], t[k]);
#pragma unroll
          for (int k = 0; k < KI; ++k) t[k] = fma2(a2[u][r][1][1], x2[1][1][k], t[k]);
        }
#pragma unroll
        for (int k = 0; k < KI; ++k) {
          const float2 v = unpack2(t[k]);
          p[r * KI + k] = v.x + v.y;
        }
      }
      // over the lanes, with the G of the two rows before in between
#pragma unroll
      for (int i = 0; i < KI; ++i) p[i] += __shfl_xor_sync(0xffffffffu, p[i + KI], 16);
      add_g(u ^ 1, 0, 0);
#pragma unroll
      for (int i = 0; i < KI / 2; ++i) p[i] += __shfl_xor_sync(0xffffffffu, p[i + KI / 2], 8);
      add_g(u ^ 1, 0, 1);
#pragma unroll
      for (int h = 4, w = KI / 4; w >= 1; h >>= 1, w >>= 1) {
        const bool up = (lane & h) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
          const float send = up ? p[i] : p[i + w], keep = up ? p[i + w] : p[i];
          p[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
      }
      float t = p[0];
      if constexpr (KI == 4) t += __shfl_xor_sync(0xffffffffu, t, 2);
      t += __shfl_xor_sync(0xffffffffu, t, 1);  // lane: row lane / 16, iterate lane / (16 / KI) mod KI
      float* ps = psum + (u * warps + warp - cw) * 32 + lane;
      if constexpr (CW > 1) ps[cw * 32] = t;
      add_g(u ^ 1, 1, 0);
      add_g(u ^ 1, 1, 1);
      if constexpr (CW > 1) {
        // over the column warps, in their order; two buffers, so one barrier per exchange
        named_sync(1 + team * kh + quarter, CW * 32);
        t = 0.f;
#pragma unroll
        for (int w = 0; w < CW; ++w) t += ps[w * 32];
      }
      // KI = 8: one copy per lane; KI = 4: the same from two lanes
      rw[32 * u + (KI == 8 ? lane : 2 * (lane >> 2) + (lane & 1))] = 2 * u + fr < rows ? bv[u] - t : 0.f;
      __syncwarp();
    }
    if (++s == stages) {
      s = 0;
      ph ^= 1u;
    }
  }
  add_g(1, 0, 0);
  add_g(1, 0, 1);
  add_g(1, 1, 0);
  add_g(1, 1, 1);
  // No copy may be in flight when the block ends (none is, unless a wait ran out).
  if (wt == 0)
    for (int q = max(0, mine - stages); q < mine; ++q)
      mbar_wait(&tbars[2 * (q % stages)], (uint32_t)(q / stages) & 1u, kWaitLimitNs / 8);

  // Sum over the teams (fixed order) through the ring's memory, then write.
  float* out = partials + (size_t)blockIdx.x * kL * dpad;
  float* red = ring;  // [team][4·kh][dpad]
  named_sync(15, warps * 32);  // every stage has been read
#pragma unroll
  for (int i = 0; i < NI; ++i)
#pragma unroll
    for (int k = 0; k < KI; ++k)
      if (col[i] < dpad) {
        const float2 lo = unpack2(g2[i][0][k]), hi = unpack2(g2[i][1][k]);
        float* dst = (teams == 1 ? out : red + (size_t)team * kh * KI * dpad) + (size_t)(l0 + (k ^ fk)) * dpad + col[i];
        *reinterpret_cast<float4*>(dst) = make_float4(lo.x, lo.y, hi.x, hi.y);
      }
  if (teams > 1) {
    named_sync(15, warps * 32);
    for (int i = threadIdx.x; i < kh * KI * dpad; i += warps * 32) {
      float t = 0.f;
      for (int q = 0; q < teams; ++q) t += red[(size_t)q * kh * KI * dpad + i];
      out[i] = t;
    }
  }
}

// G[l][j] = Σ_p partials[p][l][j] − λ_l·X[l][j] (fixed order), l < nl.  A block
// adds C columns in 256/C groups of partials.
template <int C>
__global__ void __launch_bounds__(256)
apass_path_finalize_kernel(const float* __restrict__ partials, int P, int d, int dpad, const float* __restrict__ X,
                           long long ldx, PathScalars sc, float* __restrict__ G, long long ldg,
                           const int* __restrict__ all_done) {
  if (all_done != nullptr && *all_done) return;
  const int l = blockIdx.y;
  if (l >= sc.nl) return;
  constexpr int NG = 256 / C;
  __shared__ float red[NG][C + 1];
  const int c = threadIdx.x % C, grp = threadIdx.x / C;
  const int col = blockIdx.x * C + c;
  float s = 0.f;
  if (col < d) {
#pragma unroll 8
    for (int p = grp; p < P; p += NG) s += partials[((size_t)p * kL + l) * dpad + col];
  }
  red[grp][c] = s;
  __syncthreads();
  float t = 0.f;
  int j;
  if constexpr (C == 8) {  // one warp per column
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    j = lane == 0 ? blockIdx.x * C + warp : d;
    t = warp_sum(red[lane][warp]);
  } else {
    j = grp == 0 ? col : d;
    if (grp == 0) {
#pragma unroll
      for (int k = 0; k < NG; ++k) t += red[k][c];
    }
  }
  if (j < d) G[(long long)l * ldg + j] = t - (X != nullptr ? sc.lam[l] * X[(long long)l * ldx + j] : 0.f);
}

}  // namespace

int apass_path_num_partials(int64_t n) {
  const int64_t by_rows = (n + 15) / 16;  // at least four stages per block
  int64_t P = num_sms();
  if (P > by_rows) P = by_rows;
  return (int)(P < 1 ? 1 : P);
}

int apass_path_max_d() { return kPathMaxD; }

namespace {

struct PathKernel {
  const void* fn;
  int cw, max_warps;
};

template <int KI>
PathKernel path_kernel_for(int64_t dpad) {
  if (dpad <= 128) return {(const void*)&apass_path_kernel<KI, 1, 1>, 1, path_max_warps(KI, 1)};
  if (dpad <= 256) return {(const void*)&apass_path_kernel<KI, 1, 2>, 1, path_max_warps(KI, 2)};
  if (dpad <= 512) return {(const void*)&apass_path_kernel<KI, 2, 2>, 2, path_max_warps(KI, 2)};
  if (dpad <= 768) return {(const void*)&apass_path_kernel<KI, 3, 2>, 3, path_max_warps(KI, 2)};
  return {(const void*)&apass_path_kernel<KI, 4, 2>, 4, path_max_warps(KI, 2)};
}

// More than eight iterates at widths just past one of the register form's steps
// (both sides of the lines stand in apass_path_smem.cu), and rows enough for the
// block's start, which fills X's 16 rows of shared memory.
bool path_in_smem(int64_t n, int64_t dpad, int nl) {
  if (nl <= 8) return false;
  if (dpad > 256 && dpad <= 384) return n >= 12288;
  return dpad > 512 && (dpad <= 640 || (dpad <= 832 && n >= 32768));
}

}  // namespace

int launch_apass_path(const float* A, int64_t n, int64_t d, int64_t lda, const float* b, const float* X,
                      int64_t ldx, int nl, float* partials, const int* all_done, cudaStream_t s) {
  const int64_t dpad = apass_dpad(d);
  if (d > kPathMaxD || nl < 1 || nl > kL) {
    set_error("path A-pass: d=%lld (max %d) or nl=%d (1..%d) unsupported", (long long)d, kPathMaxD, nl, kL);
    return MIHS_ERR_UNSUPPORTED;
  }
  if (path_in_smem(n, dpad, nl)) return launch_apass_path_smem(A, n, d, lda, b, X, ldx, nl, partials, all_done, s);
  const int P = apass_path_num_partials(n);
  const int rows_per_cta = (int)round_up((n + P - 1) / P, kStageRows);
  const int its = nl <= 4 ? 4 : 8;
  const PathKernel k = its == 4 ? path_kernel_for<4>(dpad) : path_kernel_for<8>(dpad);
  int kh = (nl + its - 1) / its;
  const int teams = k.max_warps / (k.cw * kh), warps = teams * k.cw * kh;
  int stages = (int)(kRingBytes / (kStageRows * dpad * 4) / teams);
  if (stages > kMaxStages) stages = kMaxStages;
  const size_t smem = path_smem_bytes(teams, warps, its * kh, (int)dpad, stages);
  MIHS_CUDA_TRY(cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  int n32 = (int)n, d32 = (int)d, dp32 = (int)dpad;
  long long lda64 = lda, ldx64 = ldx;
  void* args[] = {(void*)&A, &n32, &d32, &lda64, (void*)&b, (void*)&X, &ldx64, &nl,
                  (void*)&partials, &dp32, (void*)&rows_per_cta, &kh, &stages, (void*)&all_done};
  timing_begin(kTimerApassPath, s);
  MIHS_CUDA_TRY(cudaLaunchKernel(k.fn, dim3(P), dim3(warps * 32), args, smem, s));
  timing_end(kTimerApassPath, s);
  count_launch();
  return MIHS_OK;
}

int launch_apass_path_finalize(const float* partials, int P, int64_t d, const float* X, int64_t ldx,
                               const PathScalars& sc, float* G, int64_t ldg, const int* all_done,
                               cudaStream_t s) {
  // 32 columns read whole sectors; 8 spread few sums over more SMs
  const int c = (d + 31) / 32 * sc.nl >= num_sms() ? 32 : 8;
  auto kern = c == 32 ? apass_path_finalize_kernel<32> : apass_path_finalize_kernel<8>;
  kern<<<dim3((unsigned)((d + c - 1) / c), (unsigned)sc.nl), 256, 0, s>>>(partials, P, (int)d, (int)apass_dpad(d), X,
                                                                          ldx, sc, G, ldg, all_done);
  MIHS_CHECK_LAUNCH();
  count_launch();
  return MIHS_OK;
}

int apass_path_device_error(int* code) {
  int v = 0, z = 0;
  MIHS_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_apass_path_error, sizeof(int)));
  MIHS_CUDA_TRY(cudaMemcpyToSymbol(g_apass_path_error, &z, sizeof(int)));
  int w = 0;
  const int rc = apass_path_smem_device_error(&w);
  if (rc) return rc;
  *code = v ? v : w;
  return MIHS_OK;
}

}  // namespace mihs
