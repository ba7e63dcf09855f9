// Sparse embedding with one ±1 per column (Lemma 3, case i; "CountSketch"):
//     SA[h(j), :] += s(j) · A[j, :],   j = 0 … n−1.
//
// Instead of scattering rows of A into SA with atomics, the rows are bucketed
// by h once (a counting sort of n 32-bit keys: ~12 B/row of extra traffic) and
// thread blocks then own output rows h and stream their rows of A in
// ascending j.  A is read exactly once, in coalesced segments, no atomic
// touches SA, and the sum order is fixed, so SA is bit-reproducible.
//
// Counting sort: the n rows are cut into at most kMaxChunks chunks, one block
// each, which counts its rows per bucket in shared memory and stores the m
// counts; the scatter pass reads every chunk's counts, so that a block knows
// where its rows of each bucket begin without a global atomic, and the chunk
// boundaries inside a bucket are known too (`start`).  At 262144×1024, m = 588:
// 4 µs to count and 11 µs to scatter, where one global counter per bucket took
// 34 and 35 µs (446 atomics on each of 588 words, ≈ 76 ns apiece).  With more
// buckets every block reads more counts and fewer rows meet on a global counter,
// which then is the cheaper: above kHistMaxM, or up to 4096 where a bucket has no
// more than 64 rows (chunk counts / global counters: 262144×1024 to 2048 rows 202 /
// 214 µs, to 4096 209 / 204, to 8192 243 / 214; 262144×64 to 3000 72 / 77,
// 100000×200 to 3000 67 / 64).
#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace mihs {

namespace {

constexpr int kMaxChunks = 64;     // the scatter pass reads chunks × m counts in every block
constexpr int kChunkRows = 2048;   // fewest rows worth a chunk
constexpr int kHistMaxM = 2560;    // bucket counters of a chunk in shared memory (10 KB)
constexpr int kSortThreads = 1024;
constexpr int kGatherThreads = 256;
constexpr int kSortCap = 8192;  // bucket entries sorted in shared memory
// Rows loaded before they are added (16-byte loads in flight per thread):
// 4 left the gather bound by load latency (55 % of DRAM bandwidth).
constexpr int kRowsInFlight = 8;

// h(j) = ⌊w0·m/2³²⌋, s(j) = + if w1 even; Philox counter (j, 0, 1, 0).  The
// sign travels in bit 31.
__device__ __forceinline__ int cs_code(int j, uint32_t m, uint32_t k0, uint32_t k1) {
  const uint4 w = philox4x32_10(make_uint4((uint32_t)j, 0u, kTagCountSketch, 0u), k0, k1);
  const int h = (int)(((uint64_t)w.x * m) >> 32);
  return h | ((w.y & 1u) ? (int)0x80000000 : 0);
}

// Counts of one chunk: code[j] for its rows and hist[chunk][h].
__global__ void __launch_bounds__(kSortThreads)
cs_count_kernel(int n, int m, int rows, uint32_t k0, uint32_t k1, int* __restrict__ code, int* __restrict__ hist) {
  extern __shared__ int cnt[];
  for (int h = threadIdx.x; h < m; h += kSortThreads) cnt[h] = 0;
  __syncthreads();
  const long long j1 = min((long long)n, (long long)(blockIdx.x + 1) * rows);
  for (long long j = (long long)blockIdx.x * rows + threadIdx.x; j < j1; j += kSortThreads) {
    const int c = cs_code((int)j, (uint32_t)m, k0, k1);
    code[j] = c;
    atomicAdd(cnt + (c & 0x7fffffff), 1);
  }
  __syncthreads();
  for (int h = threadIdx.x; h < m; h += kSortThreads) hist[(size_t)blockIdx.x * m + h] = cnt[h];
}

// start[chunk][h] = where the chunk's rows of bucket h begin in the list, and
// list[...] = j | (sign << 31) for its rows (the order inside a chunk's share
// of a bucket is fixed later).  Every block sums all chunks' counts itself:
// chunks · m words from L2 instead of one more launch.
__global__ void __launch_bounds__(kSortThreads)
cs_scatter_kernel(int n, int m, int rows, const int* __restrict__ code, const int* __restrict__ hist,
                  int* __restrict__ start, int* __restrict__ list) {
  extern __shared__ int cursor[];
  __shared__ int wsum[kSortThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int chunks = gridDim.x, mine = blockIdx.x;
  // The chunk's first codes, loaded while the counts are summed.
  const long long j0 = (long long)mine * rows + threadIdx.x;
  const long long j1 = min((long long)n, (long long)(mine + 1) * rows);
  constexpr int kAhead = 4;
  int ahead[kAhead];
#pragma unroll
  for (int u = 0; u < kAhead; ++u) ahead[u] = j0 + u * kSortThreads < j1 ? __ldg(code + j0 + u * kSortThreads) : 0;
  int carry = 0;
  for (int base = 0; base < m; base += kSortThreads) {
    const int h = base + threadIdx.x;
    int total = 0, before = 0;
    if (h < m) {
      for (int c0 = 0; c0 < chunks; c0 += 32) {  // 32 loads in flight
        int v[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) v[u] = c0 + u < chunks ? __ldg(hist + (size_t)(c0 + u) * m + h) : 0;
#pragma unroll
        for (int u = 0; u < 32; ++u) {
          total += v[u];
          before += c0 + u < mine ? v[u] : 0;
        }
      }
    }
    int inc = total;  // inclusive scan over the block's buckets
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int pre = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kSortThreads / 32; ++w) {
      const int t = wsum[w];
      pre += w < warp ? t : 0;
      all += t;
    }
    if (h < m) {
      const int pos = carry + pre + inc - total + before;
      cursor[h] = pos;
      start[(size_t)mine * m + h] = pos;
    }
    carry += all;
    __syncthreads();
  }
  auto place = [&](long long j, int c) {
    const int pos = atomicAdd(cursor + (c & 0x7fffffff), 1);
    list[pos] = (int)j | (c & (int)0x80000000);
  };
#pragma unroll
  for (int u = 0; u < kAhead; ++u)
    if (j0 + u * kSortThreads < j1) place(j0 + u * kSortThreads, ahead[u]);
  for (long long j = j0 + kAhead * kSortThreads; j < j1; j += kSortThreads) place(j, code[j]);
}

// More than kHistMaxM buckets: one global counter per bucket (few rows share one).
__global__ void cs_hash_global_kernel(int n, uint32_t m, uint32_t k0, uint32_t k1, int* __restrict__ code,
                                      int* __restrict__ counts) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int c = cs_code(j, m, k0, k1);
  code[j] = c;
  atomicAdd(counts + (c & 0x7fffffff), 1);
}

// Exclusive scan of counts[0..m) → start, cursor (one block).
__global__ void __launch_bounds__(1024) cs_scan_kernel(const int* __restrict__ counts, int m, int* __restrict__ start,
                                                       int* __restrict__ cursor) {
  __shared__ int buf[1024];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < m; base += 1024) {
    const int i = base + threadIdx.x;
    const int v = i < m ? counts[i] : 0;
    buf[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {  // Hillis–Steele inclusive scan
      const int t = threadIdx.x >= o ? buf[threadIdx.x - o] : 0;
      __syncthreads();
      buf[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < m) {
      const int ex = carry + buf[threadIdx.x] - v;
      start[i] = ex;
      cursor[i] = ex;
    }
    __syncthreads();
    if (threadIdx.x == 1023) carry += buf[1023];
    __syncthreads();
  }
}

__global__ void cs_scatter_global_kernel(int n, const int* __restrict__ code, int* __restrict__ cursor,
                                         int* __restrict__ list) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int c = code[j];
  const int pos = atomicAdd(cursor + (c & 0x7fffffff), 1);
  list[pos] = j | (c & (int)0x80000000);
}

__device__ __forceinline__ int entry_row(int e) { return e & 0x7fffffff; }
__device__ __forceinline__ float entry_sign(int e) { return e < 0 ? -1.f : 1.f; }

// One block per (chunk range z, output row h, column slice of 4·CT columns):
// sort its list entries by j, then Σ s(j) A[j] over them.  The 256 threads are
// CT column groups (16 bytes each) × 256/CT row groups, which take every
// 256/CT-th entry and are added in order at the end.
//
// Memory-bound: 4·n·d bytes.  Two things cost beyond them.  A row is read in
// one piece where a block is wide enough (CT covers d up to 1024 columns): at
// 262144×1024 slices of 64 / 128 / 256 / 512 / 1024 columns took 311 / 233 /
// 200 / 184 / 171 µs, the random row segments costing DRAM locality.  And one
// block per bucket, all 588 resident at once, ran as long as the fullest
// bucket (180 µs); a bucket cut into chunk ranges (ks = 3 there) ends evenly:
// 171 µs, 6.28 TB/s, 0.93 of the measured copy.
//
// RAGGED: the last group of a row is read whole too; its columns past the row are
// the row's padding and never stored.  With a load of its own for it, 262144×1021
// to 588 rows took 239 µs against 200, 100000×203 57 against 47.  That load costs
// little where the row's last warp holds few groups, see the launch.  More blocks per
// SM read more rows at once and cost DRAM locality: this kernel needs 40 registers,
// which leave six where wide rows take four (262144×1021 with six 222 µs); the other
// one's branch, never taken otherwise, makes it 63 and so four (262144×1024 193 µs,
// without the branch and with six blocks 222).
template <int CT, bool WHOLE, bool RAGGED>
__global__ void __launch_bounds__(kGatherThreads)
cs_gather_kernel(const float* __restrict__ A, int n, int d, long long lda, const int* __restrict__ start,
                 const int* __restrict__ list, int m, int chunks, int ks, int slices, float* __restrict__ out,
                 long long ldo, int vec_out) {
  constexpr int RG = kGatherThreads / CT;
  __shared__ int keys[kSortCap];
  __shared__ float4 red[RG > 1 ? kGatherThreads : 1];
  // (32-bit arithmetic: buckets of a few rows end soon after it)
  const unsigned zh = blockIdx.x / (unsigned)slices;
  const int slice0 = (int)(blockIdx.x - zh * (unsigned)slices);
  const int z = (int)(zh / (unsigned)m), h = (int)(zh - (unsigned)z * (unsigned)m);
  const int z0 = z * chunks / ks, z1 = (z + 1) * chunks / ks;
  const int beg = start[(size_t)z0 * m + h];
  const int end = z1 < chunks ? start[(size_t)z1 * m + h] : (h + 1 < m ? start[h + 1] : n);
  const int cnt = end - beg;
  const bool sorted = cnt <= kSortCap;
  if (sorted) {
    int np2 = 1;
    while (np2 < cnt) np2 <<= 1;
    for (int e = threadIdx.x; e < np2; e += kGatherThreads) keys[e] = e < cnt ? list[beg + e] : 0x7fffffff;
    __syncthreads();
    // bitonic sort by row index (bit 31 carries the sign, so sort on j)
    for (int k = 2; k <= np2; k <<= 1) {
      for (int jj = k >> 1; jj > 0; jj >>= 1) {
        for (int e = threadIdx.x; e < np2; e += kGatherThreads) {
          const int p = e ^ jj;
          if (p > e) {
            const int a = keys[e], b = keys[p];
            const bool up = (e & k) == 0;
            const bool gt = (a & 0x7fffffff) > (b & 0x7fffffff);
            if (gt == up) {
              keys[e] = b;
              keys[p] = a;
            }
          }
        }
        __syncthreads();
      }
    }
  }
  const int ct = threadIdx.x % CT, rg = threadIdx.x / CT;
  auto sum_slice = [&](int slice) {
    const int col = 4 * (slice * CT + ct);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (col < d) {
      const bool full = col + 4 <= d;
      auto load = [&](int en) {
        const float* row = A + (long long)entry_row(en) * lda + col;
        if (RAGGED || full) return __ldcs(reinterpret_cast<const float4*>(row));
        return make_float4(row[0], col + 1 < d ? row[1] : 0.f, col + 2 < d ? row[2] : 0.f, 0.f);
      };
      auto add = [&](int en, const float4& a) {
        const float sg = entry_sign(en);
        acc.x = fmaf(sg, a.x, acc.x);
        acc.y = fmaf(sg, a.y, acc.y);
        acc.z = fmaf(sg, a.z, acc.z);
        acc.w = fmaf(sg, a.w, acc.w);
      };
      int e = rg;
      for (; e + (kRowsInFlight - 1) * RG < cnt; e += kRowsInFlight * RG) {
        int en[kRowsInFlight];
        float4 a[kRowsInFlight];
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u) en[u] = sorted ? keys[e + u * RG] : list[beg + e + u * RG];
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u) a[u] = load(en[u]);
#pragma unroll
        for (int u = 0; u < kRowsInFlight; ++u) add(en[u], a[u]);
      }
      for (; e < cnt; e += RG) {
        const int en = sorted ? keys[e] : list[beg + e];
        add(en, load(en));
      }
    }
    if constexpr (RG > 1) {
      red[threadIdx.x] = acc;
      __syncthreads();
      if (rg != 0) return;
#pragma unroll
      for (int g = 1; g < RG; ++g) {
        const float4 b = red[g * CT + ct];
        acc.x += b.x;
        acc.y += b.y;
        acc.z += b.z;
        acc.w += b.w;
      }
    }
    if (col >= d) return;
    float* o = out + ((long long)z * m + h) * ldo + col;
    if (col + 4 <= d && vec_out) {
      *reinterpret_cast<float4*>(o) = acc;
    } else {
      o[0] = acc.x;
      if (col + 1 < d) o[1] = acc.y;
      if (col + 2 < d) o[2] = acc.z;
      if (col + 3 < d) o[3] = acc.w;
    }
  };
  if constexpr (WHOLE) {  // all slices of the bucket (RG = 1: no barrier in a slice)
    for (int slice = 0; slice * 4 * CT < d; ++slice) sum_slice(slice);
  } else {
    sum_slice(slice0);
  }
}

// SA[h][c] = Σ_z part[z][h][c] in order of z.
__global__ void cs_reduce_kernel(const float* __restrict__ part, int ks, int m, int d, int dp, float* __restrict__ SA,
                                 long long ldsa) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x, h = blockIdx.y;
  if (c >= d) return;
  float s = 0.f;
  for (int z = 0; z < ks; ++z) s += part[((size_t)z * m + h) * dp + c];
  SA[(long long)h * ldsa + c] = s;
}

}  // namespace

int sketch_countsketch(const float* A, int64_t n, int64_t d, int64_t lda, int64_t m,
                       uint64_t seed, float* SA, int64_t ldsa, cudaStream_t s) {
  const bool chunked = m <= kHistMaxM || (m <= 4096 && n > 64 * m);
  int64_t chunks = 1, rows = n;
  if (chunked) {
    chunks = (n + kChunkRows - 1) / kChunkRows;
    if (chunks > kMaxChunks) chunks = kMaxChunks;
    rows = round_up((n + chunks - 1) / chunks, 32);
    chunks = (n + rows - 1) / rows;
  }
  // Column groups per block: the whole row up to 1024 columns (see the gather).
  const int64_t groups = (d + 3) / 4;
  int ct = 16;
  while (ct < 256 && ct < groups) ct *= 2;
  int slices = (int)((groups + ct - 1) / ct);
  // Chunk ranges per bucket: few and full buckets are cut so that two waves of
  // blocks (8 per SM) share the work and a block's entries can be sorted, as
  // long as a part still has 24 rows (32768×512 to 1024 rows: 47 µs cut into parts
  // of 16, 41 whole), or, up to three blocks per SM, eight for each thread to keep
  // in flight (8783×515 to 120 rows: 28 µs in parts of 15 to 18, 32 in parts of 24).
  int64_t units = m * slices;
  const int64_t per_bucket = (n + m - 1) / m;
  const int64_t least = kRowsInFlight * (kGatherThreads / ct);
  int64_t ks = (8LL * num_sms() + units - 1) / units;
  int64_t most = per_bucket / (least > 24 ? least : 24);
  const int64_t few = std::min<int64_t>((3LL * num_sms() + units - 1) / units, per_bucket / least);
  if (most < few) most = few;
  if (ks > most) ks = most;
  const int64_t need = (per_bucket + kSortCap / 2 - 1) / (kSortCap / 2);
  if (ks < need) ks = need;
  if (ks > chunks) ks = chunks;
  if (ks < 1) ks = 1;
  // of as many chunks each (five chunks in four parts take as long as in three), but
  // within the two waves: past them blocks that end early make room for the next, and
  // more parts only cost (158618×256 to 32 rows: 38 uneven parts 58 µs, 64 even ones 66;
  // 120000×256 to 64 rows, 19 and 20: 49.5 and 51.4).
  const int64_t even = (chunks + chunks / ks - 1) / (chunks / ks);
  if (even > ks && even <= per_bucket / least && units * even <= 8LL * num_sms()) ks = even;
  // Buckets enough for two waves by themselves: a block sorts its bucket once for
  // all slices of the row (50000×1500 to 20000 rows: 187 µs against 238).
  const bool whole = slices > 1 && m * ks >= 16LL * num_sms();
  if (whole) {
    units = m;
    slices = 1;
  }

  StreamScratch scratch;
  const int64_t dp = round_up(d, 4);
  // part[ks][m][dp] when ks > 1, code[n], list[n], hist/counts[chunks][m], start[chunks][m], cursor[m]
  const size_t part_floats = ks > 1 ? (size_t)ks * m * dp : 0;
  const size_t bytes = sizeof(float) * part_floats +
                       sizeof(int) * ((size_t)2 * n + 2 * (size_t)chunks * m + (chunked ? 0 : (size_t)m));
  int rc = scratch.alloc(bytes, s);
  if (rc) return rc;
  float* part = static_cast<float*>(scratch.p);
  int* code = reinterpret_cast<int*>(part + part_floats);
  int* list = code + n;
  int* hist = list + n;
  int* start = hist + (size_t)chunks * m;
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  if (chunked) {
    const size_t smem = sizeof(int) * (size_t)m;
    cs_count_kernel<<<(unsigned)chunks, kSortThreads, smem, s>>>((int)n, (int)m, (int)rows, k0, k1, code, hist);
    MIHS_CHECK_LAUNCH();
    cs_scatter_kernel<<<(unsigned)chunks, kSortThreads, smem, s>>>((int)n, (int)m, (int)rows, code, hist, start, list);
    MIHS_CHECK_LAUNCH();
    count_launch(2);
  } else {
    int* cursor = start + m;
    const int nb = (int)((n + 255) / 256);
    MIHS_CUDA_TRY(cudaMemsetAsync(hist, 0, sizeof(int) * (size_t)m, s));
    cs_hash_global_kernel<<<nb, 256, 0, s>>>((int)n, (uint32_t)m, k0, k1, code, hist);
    MIHS_CHECK_LAUNCH();
    cs_scan_kernel<<<1, 1024, 0, s>>>(hist, (int)m, start, cursor);
    MIHS_CHECK_LAUNCH();
    cs_scatter_global_kernel<<<nb, 256, 0, s>>>((int)n, code, cursor, list);
    MIHS_CHECK_LAUNCH();
    count_launch(3);
  }
  float* out = ks > 1 ? part : SA;
  const long long ldo = ks > 1 ? (long long)dp : (long long)ldsa;
  const int vec_out = ldo % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
  const unsigned grid = (unsigned)(units * ks);
  auto pick = [&](auto ragged) {
    constexpr bool R = decltype(ragged)::value;
    return whole       ? cs_gather_kernel<256, true, R>
           : ct == 256 ? cs_gather_kernel<256, false, R>
           : ct == 128 ? cs_gather_kernel<128, false, R>
           : ct == 64  ? cs_gather_kernel<64, false, R>
           : ct == 32  ? cs_gather_kernel<32, false, R>
                       : cs_gather_kernel<16, false, R>;
  };
  // A load of its own for the last group is the better where the last warp of a row of
  // more than 256 columns holds three groups or fewer: 668734×389 to 120 rows 238 µs
  // against 296 read whole, 504123×517 to 502 265 against 287, 402061×650 254 against 282;
  // with five and more, and in narrower rows, it is not (66971×545 to 502 72 against 63),
  // nor where a block that walks all slices comes to these groups as a slice of their own
  // (152409×1030 to 3000 rows 204 against 183).
  const int64_t last = groups % 32;
  const bool alone = whole && groups % ct == last;
  const bool ragged = d % 4 != 0 && (groups <= 64 || last == 0 || last > 3 || alone);
  auto kern = ragged ? pick(std::true_type{}) : pick(std::false_type{});
  // (16 KB more than the sort's 32 leave four blocks per SM.  Six / four: 481882×542 to
  // 502 rows 266 / 289 µs, 51545×710 59 / 60, 368179×710 272 / 242, 24614×850 45 / 43,
  // 307680×850 262 / 221.)
  const int64_t four_from = groups > 192 ? 64 : groups > 150 ? 256 : INT64_MAX >> 20;
  const size_t idle = ragged && ct == 256 && n * lda * 4 > (four_from << 20) ? 16384 : 0;
  kern<<<grid, kGatherThreads, idle, s>>>(A, (int)n, (int)d, (long long)lda, start, list, (int)m, (int)chunks, (int)ks,
                                       slices, out, ldo, vec_out);
  MIHS_CHECK_LAUNCH();
  count_launch();
  if (ks > 1) {
    cs_reduce_kernel<<<dim3((unsigned)((d + 127) / 128), (unsigned)m), 128, 0, s>>>(part, (int)ks, (int)m, (int)d,
                                                                                    (int)dp, SA, (long long)ldsa);
    MIHS_CHECK_LAUNCH();
    count_launch();
  }
  return MIHS_OK;
}

}  // namespace mihs
