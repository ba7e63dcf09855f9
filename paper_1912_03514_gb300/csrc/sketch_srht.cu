// Subsampled randomized Hadamard transform (Lemma 3, case iii):
//     SA = √(n_p/m) · P · (H_{n_p}/√n_p) · D · A = (1/√m) · P · H_{n_p} · D · A,
// n_p = 2^⌈log₂ n⌉ with A zero-padded, D = diag(±1), P = m rows of H_{n_p}
// sampled uniformly with replacement.
//
// Only the m sampled rows of H·D·A are needed.  With n_p = B·(n_p/B) the
// Sylvester matrix factors as H_{n_p} = H_{n_p/B} ⊗ H_B, so for a sampled row
// r = (r_hi, r_lo):
//     (H·D·A)[r] = Σ_blk (−1)^popc(r_hi ∧ blk) · (H_B · D·A[blk·B : (blk+1)·B])[r_lo].
// (For n_p < B the rows past n_p are zero and r_hi = 0: the same formula.)
// Blocks that lie wholly in the zero padding (rows ≥ n) add nothing and are
// skipped.
//
// srht_kernel: B = 1024 rows × 16 columns per unit, 256 threads, two columns
// per thread.  A thread loads its 32 rows straight from global memory (64
// registers; 64-byte segments, 64 KB in flight per block and two blocks per
// SM, so no shared-memory ring and no producer are needed), transforms the
// high five bits of the row index, passes through shared memory once,
// transforms the low five, and adds the signed sampled rows into accumulators
// held in registers (kAccMax·32 samples per block) and, past those, in shared
// memory (kExtra more).  Only what exceeds both takes a second block over the
// same, L2-resident, rows.  All additions are packed pairs (f32x2: half the issue
// slots of scalar ones).
//
// What bounds it: the shared-memory and load pipe (3500 wavefronts per unit, a
// third of them the 64-byte segments of the loads) is busy 58 % of the time on
// an SM with two blocks, the FP32 pipe 30 %, HBM 37 %; the phases of a unit
// follow one another, and only the other block of the SM fills the gaps.  The
// next unit's loads are issued before the samples are gathered (307 → 295 µs),
// and slices have one range more where blocks are left (→ 267 µs).
// 200000×1000, m = 600: 390 → 267 µs a sketch.  The form it replaces (512 × 32
// units through a TMA ring, one column per lane, accumulators in shared
// memory) executed 2.3 times the instructions (214 M against 95 M).  With more
// samples, that form → this one: 262144×1024 to 641 rows 506 → 334 µs, 1000
// 864 → 394, 1240 974 → 545, 1281 (two blocks) 990 → 718, 3076 3038 → 1480; a
// block of its own for each 640 samples took 654 µs at 641 and 700 rows.
#include <cmath>

#include "internal.h"

namespace mihs {

namespace {

constexpr int kW = 16;          // columns per slice
constexpr int kThreads = 256;   // 8 lanes per row × 32 row classes
constexpr int kB = 1024;        // rows per unit: 32 × 32
constexpr int kLB = 10;
constexpr int kAccMax = 20;     // sampled rows per thread: 40 of the 128 registers of two blocks per SM
// More sampled rows whose sums a block keeps in shared memory: at 72 bytes each as
// many as leave room for two blocks per SM.
constexpr int kExtra = 600;
// Accepted m for n ≥ 1024, the interface's own limit from its first form on: six
// times the widest matrix, past any sketch in use (m ≤ n bounds it below that).
constexpr int kMaxM = 12672;
// Row r of a unit starts at float 16·r + 16·(r/32): the 64-byte shift every 32
// rows keeps the second stage's reads (rows 32 apart) free of bank conflicts.
constexpr int kYFloats = kB * kW + (kB / 32) * kW;
__host__ __device__ constexpr int y_off(int r) { return kW * r + kW * (r >> 5); }

// signs[w] bit t = 1 when D_{32w+t} = −1 (counter (j,0,2,0), w0 odd), one warp
// per word; rows[i] = ⌊w0 / 2^(32−L)⌋ from counter (i,0,3,0).
__global__ void srht_prep_kernel(int n, int m, int L, uint32_t k0, uint32_t k1,
                                 uint32_t* __restrict__ signs, int* __restrict__ rows) {
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t neg = 0;
  if (idx < n) neg = philox4x32_10(make_uint4((uint32_t)idx, 0u, kTagSrhtSigns, 0u), k0, k1).x & 1u;
  const uint32_t word = __ballot_sync(0xffffffffu, neg);
  if ((threadIdx.x & 31) == 0 && idx < n) signs[idx >> 5] = word;
  if (idx < m) {
    const uint4 w = philox4x32_10(make_uint4((uint32_t)idx, 0u, kTagSrhtRows, 0u), k0, k1);
    rows[idx] = L > 0 ? (int)(w.x >> (32 - L)) : 0;
  }
}

// Two fp32 columns in one 64-bit register pair.
typedef unsigned long long P2;
__device__ __forceinline__ P2 p2_add(P2 a, P2 b) {
  P2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ P2 p2_sub(P2 a, P2 b) {
  P2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// (x, y & ymask) with both signs flipped when bit 31 of f is set.
__device__ __forceinline__ P2 p2_flip(uint2 v, uint32_t f, uint32_t ymask = 0xffffffffu) {
  const uint32_t s = f & 0x80000000u;
  P2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(v.x ^ s), "r"((v.y & ymask) ^ s));
  return d;
}

__device__ __forceinline__ void fwht32(P2 (&x)[32]) {
#pragma unroll
  for (int h = 1; h < 32; h <<= 1) {
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      if ((i & h) == 0) {
        const P2 a = x[i], b = x[i + h];
        x[i] = p2_add(a, b);
        x[i + h] = p2_sub(a, b);
      }
    }
  }
}

struct SrhtArgs {
  const float* A;
  int n, d;
  long long lda;
  int m, mc;            // sampled rows, and those of one block (blockIdx.x % zc)
  int zc;
  int nblk;             // ⌈n/B⌉
  int ks, wide, ncs;    // ranges of units per slice: ks + 1 for slices < wide, ks for the others (of ncs)
  const uint32_t* signs;
  const int* rows;
  float* out;           // [range][m][ldo]
  long long ldo;
  float scale;          // 1 for partial sums
};

// The thread's 32 rows t + 32k of unit rows rbase …, columns c and c + 1.  Lanes
// past the last column read the first one: nothing of theirs is stored.  With odd
// d the last column's pair is read whole (8-byte aligned, so it lies in the page
// of its first half) and the half past the row masked by the caller: a load of
// its own for that lane made every block of the last slice, and with it the
// kernel, a sixth slower.
__device__ __forceinline__ void load_rows(const SrhtArgs& a, long long rbase, int t, int c, uint2 (&v)[32]) {
  const int col = c < a.d ? c : 0;
  long long step = 32 * (long long)sizeof(float) * a.lda;
  asm volatile("" : "+l"(step));  // (32 precomputed row offsets would take 64 registers)
  if (rbase + kB <= a.n) {
    const char* src = reinterpret_cast<const char*>(a.A + (rbase + t) * a.lda + col);
#pragma unroll
    for (int k = 0; k < 32; ++k) {
      v[k] = __ldg(reinterpret_cast<const uint2*>(src));
      src += step;
    }
  } else {
    // The last rows of A: eight loads at a time, from clamped rows and without
    // branches between them.
    const char* src = reinterpret_cast<const char*>(a.A + min(rbase + t, (long long)a.n - 1) * a.lda + col);
#pragma unroll
    for (int k8 = 0; k8 < 32; k8 += 8) {
#pragma unroll
      for (int k = k8; k < k8 + 8; ++k) {
        v[k] = __ldg(reinterpret_cast<const uint2*>(src));
        if (rbase + t + 32 * (k + 1) < a.n) src += step;
      }
#pragma unroll
      for (int k = k8; k < k8 + 8; ++k)
        if (rbase + t + 32 * k >= a.n) v[k] = make_uint2(0u, 0u);
      asm volatile("" ::: "memory");
    }
  }
}

template <int ACC, bool EXTRA>
__global__ void __launch_bounds__(kThreads, 2) srht_kernel(const SrhtArgs a) {
  extern __shared__ float4 smem4[];
  float* Y = reinterpret_cast<float*>(smem4);                  // kYFloats
  int* off = reinterpret_cast<int*>(Y + kYFloats);             // ACC·32: byte offset of row r_lo in Y
  int2* xoff = reinterpret_cast<int2*>(off + ACC * 32);        // EXTRA: {offset, r_hi} of the samples past ACC·32
  P2* xacc = reinterpret_cast<P2*>(xoff + (EXTRA ? a.mc - ACC * 32 : 0));  // … × 8 column pairs: their sums
  const int tid = threadIdx.x, lane = tid & 31;
  const int cl = tid & 7, t = tid >> 3;                        // column pair, row class
  // Slices with the longer ranges come first: two of them never share an SM.
  const int z = (int)(blockIdx.x % a.zc);
  int w = (int)(blockIdx.x / a.zc), slice, range, ranges;
  if (w < (a.ncs - a.wide) * a.ks) {
    slice = a.wide + w % (a.ncs - a.wide);
    range = w / (a.ncs - a.wide);
    ranges = a.ks;
  } else {
    w -= (a.ncs - a.wide) * a.ks;
    slice = w % a.wide;
    range = w / a.wide;
    ranges = a.ks + 1;
  }
  const int i0 = z * a.mc, i1 = min(a.m, i0 + a.mc);
  const int c = slice * kW + 2 * cl;
  const int b0 = (int)((long long)range * a.nblk / ranges);
  const int b1 = (int)((long long)(range + 1) * a.nblk / ranges);

  // Sample q·32 + t of the block belongs to this thread's class t (slot q):
  // its offset in Y from shared memory, its r_hi for the signs of slots
  // 8j + cl in a register of lane cl of the class.
  for (int e = tid; e < ACC * 32; e += kThreads) {
    const int i = i0 + e;
    off[e] = i < i1 ? 4 * y_off(a.rows[i] & (kB - 1)) : 0;
  }
  const int nx = EXTRA ? max(0, i1 - i0 - ACC * 32) : 0;
  if (EXTRA) {
    for (int e = tid; e < nx; e += kThreads) {
      const int r = a.rows[i0 + ACC * 32 + e];
      xoff[e] = make_int2(4 * y_off(r & (kB - 1)), r >> kLB);
    }
    for (int e = t; e < nx; e += 32) xacc[8 * e + cl] = 0ull;  // (read and added to by this thread only)
  }
  constexpr int NJ = (ACC + 7) / 8;
  int rhi[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const int i = i0 + (8 * j + cl) * 32 + t;
    rhi[j] = i < i1 ? a.rows[i] >> kLB : 0;
  }
  P2 acc[ACC];
#pragma unroll
  for (int q = 0; q < ACC; ++q) acc[q] = 0ull;
  const char* Yc = reinterpret_cast<const char*>(Y) + 8 * cl;
  const int nwords = (a.n + 31) >> 5;
  const uint32_t ymask = c + 1 < a.d ? 0xffffffffu : 0u;

  uint2 v[32];
  for (int blk = b0 - 1; blk < b1; ++blk) {
    if (blk >= b0) {
    P2 x[32];
    // D: word k of the unit's 32 sign words covers rows 32k … 32k + 31, row
    // t + 32k is bit t of word k; bit k of `neg` = its sign.
    const int wi = blk * (kB / 32) + lane;
    const uint32_t sw = wi < nwords ? __ldg(a.signs + wi) : 0u;
    uint32_t neg = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uint32_t bal = __ballot_sync(0xffffffffu, (sw >> ((t & ~3) + r)) & 1u);
      if ((t & 3) == r) neg = bal;
    }
#pragma unroll
    for (int k = 0; k < 32; ++k) x[k] = p2_flip(v[k], neg << (31 - k), ymask);
    fwht32(x);  // the high five bits of the row
    __syncthreads();  // the previous unit's sampled rows have been read
    P2* Yt = reinterpret_cast<P2*>(Y + y_off(t) + 2 * cl);
#pragma unroll
    for (int k = 0; k < 32; ++k) Yt[k * (y_off(32) / 2)] = x[k];
    __syncthreads();
    P2* Yu = reinterpret_cast<P2*>(Y + y_off(32 * t) + 2 * cl);
#pragma unroll
    for (int k = 0; k < 32; ++k) x[k] = Yu[k * (kW / 2)];
    fwht32(x);  // the low five bits
#pragma unroll
    for (int k = 0; k < 32; ++k) Yu[k * (kW / 2)] = x[k];
    }
    // The next unit's rows travel while the samples are gathered.
    if (blk + 1 < b1) {
      load_rows(a, (long long)(blk + 1) * kB, t, c, v);
    } else {  // (the old values must not stay live beside the transform's)
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] = make_uint2(0u, 0u);
    }
    if (blk < b0) continue;
    __syncthreads();
    // Sampled row r takes entry r_lo of this block's transform with the sign
    // (−1)^popc(r_hi ∧ blk): lane cl finds the signs of slots 8j + cl, a ballot
    // hands them to the class's other lanes.
    uint32_t sg[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j)
      sg[j] = __ballot_sync(0xffffffffu, __popc(rhi[j] & blk) & 1) >> (lane & 24);
#pragma unroll
    for (int q = 0; q < ACC; ++q) {
      const uint2 y = *reinterpret_cast<const uint2*>(Yc + off[q * 32 + t]);
      acc[q] = p2_add(acc[q], p2_flip(y, sg[q >> 3] << (31 - (q & 7))));
    }
    if (EXTRA) {
#pragma unroll 4
      for (int e = t; e < nx; e += 32) {
        const int2 o = xoff[e];
        const uint2 y = *reinterpret_cast<const uint2*>(Yc + o.x);
        xacc[8 * e + cl] = p2_add(xacc[8 * e + cl], p2_flip(y, (uint32_t)__popc(o.y & blk) << 31));
      }
    }
  }
  float* out = a.out + (long long)range * a.m * a.ldo;
#pragma unroll
  for (int q = 0; q < ACC; ++q) {
    const int i = i0 + q * 32 + t;
    float2 v2;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v2.x), "=f"(v2.y) : "l"(acc[q]));
    if (i < i1) {
      float* o = out + (long long)i * a.ldo + c;
      if (c < a.d) o[0] = v2.x * a.scale;
      if (c + 1 < a.d) o[1] = v2.y * a.scale;
    }
  }
  if (EXTRA) {
    for (int e = t; e < nx; e += 32) {
      const float2 v2 = *reinterpret_cast<const float2*>(xacc + 8 * e + cl);
      float* o = out + (long long)(i0 + ACC * 32 + e) * a.ldo + c;
      if (c < a.d) o[0] = v2.x * a.scale;
      if (c + 1 < a.d) o[1] = v2.y * a.scale;
    }
  }
}

// SA[i][c] = scale · Σ_k part[k][i][c] in order of k (one range more in the slices < wide).
__global__ void __launch_bounds__(256) srht_reduce_kernel(const float* __restrict__ part, int ks, int wide, int m, int d,
                                                          long long ldp, float scale, float* __restrict__ SA,
                                                          long long ldsa) {
  const int c = blockIdx.x * 256 + threadIdx.x, i = blockIdx.y;
  if (c >= d) return;
  float s = 0.f;
  const int ranges = ks + (c / kW < wide ? 1 : 0);
#pragma unroll 4
  for (int k = 0; k < ranges; ++k) s += part[((long long)k * m + i) * ldp + c];
  SA[(long long)i * ldsa + c] = s * scale;
}

using KernelFn = void (*)(const SrhtArgs);

KernelFn pick_kernel(int acc) {
  if (acc <= 4) return srht_kernel<4, false>;
  if (acc <= 8) return srht_kernel<8, false>;
  if (acc <= 12) return srht_kernel<12, false>;
  if (acc <= 16) return srht_kernel<16, false>;
  if (acc <= kAccMax) return srht_kernel<kAccMax, false>;
  return srht_kernel<kAccMax, true>;
}
int acc_slots(int acc) { return acc <= 16 ? (acc + 3) / 4 * 4 : kAccMax; }

}  // namespace

int sketch_srht(const float* A, int64_t n, int64_t d, int64_t lda, int64_t m, uint64_t seed,
                float* SA, int64_t ldsa, cudaStream_t s) {
  int L = 0;
  while ((1LL << L) < n) ++L;
  if (n >= kB && m > kMaxM) {
    set_error("srht: m=%lld is beyond %d", (long long)m, kMaxM);
    return MIHS_ERR_UNSUPPORTED;
  }
  const int nblk = (int)((n + kB - 1) / kB);
  const int ncs = (int)((d + kW - 1) / kW);
  // Samples per block: as many as the registers hold, evenly cut.
  const int per_block = kAccMax * 32 + kExtra;
  const int zc = (int)((m + per_block - 1) / per_block);
  const int mc = (int)round_up((m + zc - 1) / zc, 32);
  // The blocks of one column slice share its units.  All slices are walked in
  // step (neighbours read the two halves of a 128-byte line within a short
  // time: cut into equal ranges out of step instead, DRAM traffic doubled and
  // 200000×1000 took 398 µs), and two blocks per SM are resident: ks ranges
  // per slice and one more in as many slices as there are blocks left.
  const int64_t resident = 2LL * num_sms() / zc;
  int64_t ks = resident / ncs, wide = resident % ncs;
  if (ks < 1) ks = 1, wide = 0;
  if (ks >= nblk) ks = nblk, wide = 0;
  const int64_t ranges = ks + (wide > 0 ? 1 : 0);

  StreamScratch scratch;
  const size_t nwords = (size_t)(n + 31) / 32;
  const int64_t ldp = round_up(d, 4);
  const size_t part_floats = ranges > 1 ? (size_t)ranges * m * ldp : 0;
  int rc = scratch.alloc(sizeof(float) * part_floats + sizeof(uint32_t) * nwords + sizeof(int) * (size_t)m, s);
  if (rc) return rc;
  float* part = static_cast<float*>(scratch.p);
  uint32_t* signs = reinterpret_cast<uint32_t*>(part + part_floats);
  int* rows = reinterpret_cast<int*>(signs + nwords);
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  const int64_t most = n > m ? n : m;
  srht_prep_kernel<<<(unsigned)((most + 255) / 256), 256, 0, s>>>((int)n, (int)m, L, k0, k1, signs, rows);
  MIHS_CHECK_LAUNCH();

  SrhtArgs a;
  a.A = A;
  a.n = (int)n;
  a.d = (int)d;
  a.lda = lda;
  a.m = (int)m;
  a.mc = mc;
  a.zc = zc;
  a.nblk = nblk;
  a.ks = (int)ks;
  a.wide = (int)wide;
  a.ncs = ncs;
  a.signs = signs;
  a.rows = rows;
  const float scale = (float)(1.0 / std::sqrt((double)m));
  a.out = ranges > 1 ? part : SA;
  a.ldo = ranges > 1 ? ldp : ldsa;
  a.scale = ranges > 1 ? 1.f : scale;
  const int acc = mc / 32;
  const KernelFn fn = pick_kernel(acc);
  const size_t extra = acc > kAccMax ? (size_t)(mc - kAccMax * 32) : 0;
  const size_t smem = sizeof(float) * kYFloats + sizeof(int) * 32 * (size_t)acc_slots(acc) +
                      (sizeof(int2) + sizeof(float) * kW) * extra;
  MIHS_CUDA_TRY(cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  fn<<<(unsigned)((ncs * ks + wide) * zc), kThreads, smem, s>>>(a);
  MIHS_CHECK_LAUNCH();
  count_launch(2);
  if (ranges > 1) {
    srht_reduce_kernel<<<dim3((unsigned)((d + 255) / 256), (unsigned)m), 256, 0, s>>>(
        part, (int)ks, (int)wide, (int)m, (int)d, ldp, scale, SA, ldsa);
    MIHS_CHECK_LAUNCH();
    count_launch();
  }
  return MIHS_OK;
}

}  // namespace mihs
