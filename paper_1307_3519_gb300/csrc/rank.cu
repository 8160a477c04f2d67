// rank.cu -- per-trait average-rank transform (section "Input data": ranks per
// trait row; section "Handling tied data": average ranks for ties and the factor
// sum(t^3 - t); section "Handling missing values": NaN samples are left out).
//
// One warp per trait.  The row's present values are sorted as integers (a bitonic
// network over the warp's registers) into shared memory, and each present sample k
// finds lo = #{j present: x_j < x_k} and, where the row has ties, eq = #{j present: x_j
// == x_k} (k itself included) by binary search, so 2 * average rank = 2 lo + eq + 1,
// exactly.  The stored value is the centred integer a = 2 lo + eq - K = 2 rank - (K + 1),
// |a| <= K-1, which FP16 holds exactly for K <= 512 (integers up to 2048 are exact).
// The run containing k has length eq, so sum_k (eq_k^2 - 1) = sum_runs (t^3 - t).
#include "common.cuh"

namespace krux {

namespace {
constexpr int kRankWarps = 8;

// Tie factor C = 1 - sum(t^3-t)/(K^3-K) and the trait constants of the scan:
// H = 3/(K(K+1)C) * sum_i D_i^2/N_i, so cfac = 3/(K(K+1)C) and the fast-test
// bound tau = K(K+1)C/3; degenerate traits (K < 2 or C = 0) get cfac 0, tau +inf.
// With M = K^3 - K - sum(t^3-t) (an exact integer), K(K+1)C = M/(K-1): cfac is one
// correctly rounded FP64 division, 3(K-1)/M, and tau an FP32 one.
__device__ __forceinline__ void trait_consts(int K, long long tie, float &tau, double &cfac) {
  const long long M = K >= 2 ? (long long)K * K * K - K - tie : 0;
  if (M > 0) {
    cfac = 3.0 * (double)(K - 1) / (double)M;
    tau = (float)M / (float)(3 * (K - 1));
  } else {
    cfac = 0.0;
    tau = __int_as_float(0x7f800000);  // +inf: never a hit
  }
}

// A value as an integer of the same order: -0.0 as +0.0, NaN after everything.
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t b = __float_as_uint(x);
  if (x != x) return 0xffffffffu;
  if (x == 0.f) return 0x80000000u;
  return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}

// Sorts 32 E values, element lane * E + i in v[i] (bitonic network; strides below E stay
// in the lane).
template <int E>
__device__ __forceinline__ void warp_sort(uint32_t (&v)[E], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= E) {  // the partner is another lane's element i
        const bool low = ((lane & (j / E)) == 0) == (((lane * E) & k) == 0);
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, v[i], j / E);
          v[i] = low ? min(v[i], o) : max(v[i], o);
        }
      } else {
#pragma unroll
        for (int i = 0; i < E; ++i) {
          if (i & j) continue;
          const uint32_t a = min(v[i], v[i | j]), b = max(v[i], v[i | j]);
          const bool up = k < E ? (i & k) == 0 : ((lane * E) & k) == 0;
          v[i] = up ? a : b;
          v[i | j] = up ? b : a;
        }
      }
    }
  }
}

// E values per lane (32 E >= N).  The O(N^2) count of smaller and equal values that this
// replaces took 884 us for 15,000 x 500, 163 for 15,000 x 200 and 69 for 20,000 x 102;
// the network and the searches 100, 38 and 27.  The block's first warp writes the FP64 constants of
// its rows together (FP64 issue is slow on this part); rows past T are padding: zero
// ranks, never a hit.
template <int E>
__global__ void __launch_bounds__(kRankWarps * 32)
rank_kernel(const float *__restrict__ expr, int T, int N, int64_t ld, int Np, int rows_pad, RankDev r) {
  __shared__ uint32_t sorted[kRankWarps][32 * E];
  __shared__ int sK[kRankWarps], stie[kRankWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * kRankWarps + warp;
  int K = 0, tie = 0;
  if (t < T) {
    const float *row = expr + (int64_t)t * ld;
    uint32_t own[E], v[E];
    int nan_seen = 0;
#pragma unroll
    for (int i = 0; i < E; ++i) {  // sample 32 i + lane
      const int k = 32 * i + lane;
      const float x = k < N ? row[k] : __int_as_float(0x7fc00000);
      own[i] = order_key(x);
      v[i] = own[i];
      // the NaN samples, in sample order
      const bool isn = k < N && x != x;
      const unsigned bn = __ballot_sync(0xffffffffu, isn);
      if (isn) r.nan_idx[(int64_t)t * N + nan_seen + __popc(bn & ((1u << lane) - 1u))] = (uint16_t)k;
      nan_seen += __popc(bn);
    }
    K = N - nan_seen;
    warp_sort<E>(v, lane);
    uint32_t *a = sorted[warp];
#pragma unroll
    for (int i = 0; i < E; ++i) a[lane * E + i] = v[i];
    __syncwarp();
    // ties among the present values
    bool same = false;
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int p = 32 * i + lane;
      same |= p + 1 < K && a[p] == a[p + 1];
    }
    const bool ties = __any_sync(0xffffffffu, same);
#pragma unroll
    for (int i = 0; i < E; ++i) {
      const int k = 32 * i + lane;
      const bool present = own[i] != 0xffffffffu;
      int lo = 0, hi = 0;
#pragma unroll
      for (int step = 16 * E; step > 0; step >>= 1)
        if (a[lo + step - 1] < own[i]) lo += step;
      hi = lo + 1;
      if (ties) {
        hi = lo;  // (own[i] itself lies at lo, so hi ends beyond it)
#pragma unroll
        for (int step = 16 * E; step > 0; step >>= 1)
          if (hi + step <= 32 * E && a[hi + step - 1] <= own[i]) hi += step;
        if (hi < 32 * E && a[hi] <= own[i]) ++hi;
      }
      const int eq = present ? hi - lo : 0;
      if (!present) lo = 0;
      const int c = present ? 2 * lo + eq - K : 0;
      if (k < N) {
        r.lo[(int64_t)t * N + k] = (uint16_t)lo;
        r.eq[(int64_t)t * N + k] = (uint16_t)eq;
        tie += present ? eq * eq - 1 : 0;
      }
      if (k < Np) {
        r.A[(int64_t)t * Np + k] = __int2half_rn(c);
        if (r.At) r.At[tiled_index(t, k, Np)] = __int2half_rn(c);
      }
    }
    tie = (int)__reduce_add_sync(0xffffffffu, (unsigned)tie);
    if (lane == 0) {
      r.tie[t] = tie;
      r.K[t] = K;
      r.nan_cnt[t] = (uint16_t)nan_seen;
      // the tile's traits with NaN (low 16 bits) and with more than kNanCMax (high)
      if (nan_seen > 0) atomicAdd(&r.tile_nan[t / kTileM], 1u + (nan_seen > kNanCMax ? 1u << 16 : 0u));
    }
  } else if (t < rows_pad) {
    for (int k = lane; k < Np; k += 32) {
      r.A[(int64_t)t * Np + k] = __int2half_rn(0);
      if (r.At) r.At[tiled_index(t, k, Np)] = __int2half_rn(0);
    }
    if (lane == 0) r.nan_cnt[t] = 0;
  }
  if (lane == 0) {
    sK[warp] = K;
    stie[warp] = tie;
  }
  __syncthreads();
  if (warp == 0 && lane < kRankWarps) {
    const int q = blockIdx.x * kRankWarps + lane;
    if (q < rows_pad) trait_consts(sK[lane], (long long)stie[lane], r.tau[q], r.cfac[q]);
  }
}

// out[p][row][k] = A[row][perm_p[k]] for k < N (padding columns stay 0): the
// rank matrix of the expression with its sample columns permuted (ranks, tie
// sums and K are invariant under a column permutation).  One block per 32 rows, its
// rows staged in shared memory once for all permutations; a thread gathers 8
// consecutive samples and stores 16 bytes, in either layout.  Bound by the stores
// (72 MB for 16 x 20,000 x 102: 110 us with one 2-byte element per thread).
constexpr int kPermRows = 32;
template <bool kTiled>
__global__ void __launch_bounds__(256)
permute_rows_kernel(const __half *__restrict__ A, __half *__restrict__ out, int rows_pad, int Np,
                    int N, const int32_t *__restrict__ perms, int P, unsigned int *status) {
  __shared__ __align__(16) __half rows[kPermRows * kMaxN];
  __shared__ __align__(16) int32_t perm[kMaxN];
  const int row0 = blockIdx.x * kPermRows;  // (rows_pad is a multiple of 128)
  const int per_row = Np / 8;
  for (int i = threadIdx.x; i < kPermRows * per_row; i += blockDim.x)
    reinterpret_cast<uint4 *>(rows)[i] = reinterpret_cast<const uint4 *>(A + (int64_t)row0 * Np)[i];
  for (int p = blockIdx.y; p < P; p += gridDim.y) {
    __syncthreads();
    for (int k = threadIdx.x; k < Np; k += blockDim.x) {
      int32_t src = -1;
      if (k < N) {
        src = perms[(int64_t)p * N + k];
        if (src < 0 || src >= N) {
          if (status != nullptr) atomicOr(status, kDevBadPerm);
          src = -1;
        }
      }
      perm[k] = src;
    }
    __syncthreads();
    __half *o = out + (int64_t)p * rows_pad * Np;
    for (int i = threadIdx.x; i < kPermRows * per_row; i += blockDim.x) {
      // tiled: consecutive threads take the halves and rows of one atom
      const int r = kTiled ? (i >> 1) % kPermRows : i / per_row;
      const int q = kTiled ? 2 * (i / (2 * kPermRows)) + (i & 1) : i - r * per_row;
      __align__(16) __half v[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int32_t src = perm[8 * q + j];
        v[j] = src >= 0 ? rows[r * Np + src] : __int2half_rn(0);
      }
      const int64_t at = kTiled ? tiled_index(row0 + r, 8 * q, Np) : (int64_t)(row0 + r) * Np + 8 * q;
      *reinterpret_cast<uint4 *>(o + at) = *reinterpret_cast<const uint4 *>(v);
    }
  }
}
// inv[q][perms[q][k]] = k (entries outside 0..N-1 are skipped; the row gather
// reports them).
__global__ void invert_perms_kernel(const int32_t *__restrict__ perms, int P, int N,
                                    int32_t *__restrict__ inv) {
  const int64_t total = (int64_t)P * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(i / N), k = (int)(i % N);
    const int32_t v = perms[i];
    if (v >= 0 && v < N) inv[(int64_t)q * N + v] = k;
  }
}

__global__ void permute_nan_idx_kernel(const uint16_t *__restrict__ nan_cnt,
                                       const uint16_t *__restrict__ nan_idx, int T, int N,
                                       const int32_t *__restrict__ inv, int P,
                                       uint16_t *__restrict__ out) {
  const int64_t total = (int64_t)P * T * N;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(i % N);
    const int64_t qt = i / N;
    const int t = (int)(qt % T);
    const int q = (int)(qt / T);
    if (j < nan_cnt[t]) out[i] = (uint16_t)inv[(int64_t)q * N + nan_idx[(int64_t)t * N + j]];
  }
}
}  // namespace

// Per-trait constants of the padding rows of the last 128-trait tile: never a hit.
__global__ void pad_traits_kernel(int T, int rows_pad, float *tau, double *cfac, uint16_t *nan_cnt) {
  const int t = T + blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= rows_pad) return;
  tau[t] = __int_as_float(0x7f800000);
  cfac[t] = 0.0;
  nan_cnt[t] = 0;
}

cudaError_t launch_pad_traits(int T, int rows_pad, float *tau, double *cfac, uint16_t *nan_cnt,
                              cudaStream_t s) {
  if (rows_pad <= T) return cudaSuccess;
  pad_traits_kernel<<<1, 128, 0, s>>>(T, rows_pad, tau, cfac, nan_cnt);
  return cudaGetLastError();
}

cudaError_t launch_rank(const float *expr, int T, int N, int64_t ld, int Np, int rows_pad,
                        const RankDev &r, cudaStream_t s) {
  const int grid = (rows_pad + kRankWarps - 1) / kRankWarps;
  if (N <= 32) rank_kernel<1><<<grid, kRankWarps * 32, 0, s>>>(expr, T, N, ld, Np, rows_pad, r);
  else if (N <= 64) rank_kernel<2><<<grid, kRankWarps * 32, 0, s>>>(expr, T, N, ld, Np, rows_pad, r);
  else if (N <= 128) rank_kernel<4><<<grid, kRankWarps * 32, 0, s>>>(expr, T, N, ld, Np, rows_pad, r);
  else if (N <= 256) rank_kernel<8><<<grid, kRankWarps * 32, 0, s>>>(expr, T, N, ld, Np, rows_pad, r);
  else rank_kernel<16><<<grid, kRankWarps * 32, 0, s>>>(expr, T, N, ld, Np, rows_pad, r);
  return cudaGetLastError();
}

cudaError_t launch_invert_perms(const int32_t *perms, int P, int N, int32_t *inv, cudaStream_t s) {
  const int64_t total = (int64_t)P * N;
  if (total == 0) return cudaSuccess;
  int grid = (int)((total + 255) / 256);
  if (grid > 152 * 4) grid = 152 * 4;
  invert_perms_kernel<<<grid, 256, 0, s>>>(perms, P, N, inv);
  return cudaGetLastError();
}

cudaError_t launch_permute_nan_idx(const uint16_t *nan_cnt, const uint16_t *nan_idx, int T, int N,
                                   const int32_t *inv, int P, uint16_t *out, cudaStream_t s) {
  const int64_t total = (int64_t)P * T * N;
  if (total == 0) return cudaSuccess;
  int grid = (int)((total + 255) / 256);
  if (grid > 152 * 16) grid = 152 * 16;
  permute_nan_idx_kernel<<<grid, 256, 0, s>>>(nan_cnt, nan_idx, T, N, inv, P, out);
  return cudaGetLastError();
}

cudaError_t launch_permute_rows(const __half *A, __half *out, int rows_pad, int Np, int N,
                                const int32_t *perms, int P, bool tiled, unsigned int *status,
                                cudaStream_t s) {
  if (P <= 0 || rows_pad <= 0) return cudaSuccess;
  const dim3 grid((unsigned)(rows_pad / kPermRows), (unsigned)(P < 8 ? P : 8));
  if (tiled) permute_rows_kernel<true><<<grid, 256, 0, s>>>(A, out, rows_pad, Np, N, perms, P, status);
  else permute_rows_kernel<false><<<grid, 256, 0, s>>>(A, out, rows_pad, Np, N, perms, P, status);
  return cudaGetLastError();
}

}  // namespace krux

// ---------------------------------------------------------------------------
// Ranks of every trait over the samples left after dropping a missing-genotype
// pattern (section "Handling missing values": a new expression matrix with the
// samples of the pattern removed, re-ranked).  No re-sort: for present samples,
// x_q < x_k exactly when lo_q < lo_k and x_q == x_k exactly when lo_q == lo_k,
// so lo' = lo - #{q dropped, present, lo_q < lo_k} and
// eq' = eq - #{q dropped, present, lo_q == lo_k}.
//
// With K' the present samples left, the centred rank 2 lo' + eq' - K' is the old one less
// sum_q sign(lo_k - lo_q) over the dropped present samples q: small integers, exact in
// FP16, so a bucket costs four packed operations per two samples and dropped sample.
//
// One warp per trait row and kRerankChunk buckets of a run (buckets of one base rank set;
// grid.y = chunk of buckets): the row's lo and centred ranks are read once, into
// registers (lane l owns samples 4l..4l+3 of every 128), lo also into the warp's
// shared-memory copy (where the dropped samples' values are looked up); the chunk's job
// fields are staged in shared memory.  Lane b counts bucket b's K at the start and turns
// it and the tie sum (zero for a row without ties, whose tie pass is left out) into the
// FP64 constants at the end, all buckets of the chunk at once.  Issue-bound: 200 buckets
// of 5,000 x 102 took 282 us with lo, eq and the tie sum updated as 32-bit integers and
// four conversions per lane, now 136 (229 MB written).
namespace krux {
namespace {
constexpr int kRerankWarps = 8;
constexpr int kRerankChunk = 16;            // buckets per warp
constexpr int kRerankDrops = 1024;          // drop-list entries staged per block

struct RerankOut {  // a bucket's outputs and drop list, staged per block
  __half *A;
  float *tau;
  double *cfac;
  int32_t drop_off, n_drop;
};

// kPasses = ceil(Np / 128) passes of 4 samples per lane (the row in registers).
template <int kPasses>
__global__ void __launch_bounds__(kRerankWarps * 32, kPasses == 1 ? 5 : (kPasses == 2 ? 2 : 1))
rerank_kernel(const RerankJob *__restrict__ jobs, int n_jobs_all, const int32_t *__restrict__ drops,
              int tiled) {
  __shared__ uint32_t srow[kRerankWarps][kMaxN];  // lo of the warp's row as FP16, twice; ~0: absent
  __shared__ RerankOut sj[kRerankChunk];
  __shared__ int32_t sdrop[kRerankDrops];          // the chunk's drop lists, when they fit
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int jbase = blockIdx.y * kRerankChunk;
  const int n_jobs = min(kRerankChunk, n_jobs_all - jbase);
  if (threadIdx.x < n_jobs) {
    const RerankJob &J = jobs[jbase + threadIdx.x];
    sj[threadIdx.x] = RerankOut{J.A, J.tau, J.cfac, J.drop_off, J.n_drop};
  }
  __syncthreads();
  // the chunk's drop lists lie back to back in `drops`
  const int d0 = sj[0].drop_off;
  const int nd = sj[n_jobs - 1].drop_off + sj[n_jobs - 1].n_drop - d0;
  const bool staged = nd <= kRerankDrops;
  if (staged)
    for (int i = threadIdx.x; i < nd; i += blockDim.x) sdrop[i] = drops[d0 + i];
  __syncthreads();
  const RerankJob &J0 = jobs[0];  // every job of the run has this base and shape
  const int N = J0.N, Np = J0.Np, T = J0.T, rows_pad = J0.rows_pad;
  const int t = blockIdx.x * kRerankWarps + warp;
  if (t >= rows_pad) return;  // whole warps leave; no block barrier follows
  if (t >= T) {  // padding row: zeros, never a hit
    for (int j = 0; j < n_jobs; ++j) {
      const RerankOut &J = sj[j];
      for (int k = lane; k < Np; k += 32)
        J.A[tiled ? tiled_index(t, k, Np) : (int64_t)t * Np + k] = __int2half_rn(0);
      if (lane == 0) {
        J.tau[t] = __int_as_float(0x7f800000);
        J.cfac[t] = 0.0;
      }
    }
    return;
  }
  const uint16_t *lo = J0.base.lo + (int64_t)t * N;
  const uint16_t *eq = J0.base.eq + (int64_t)t * N;
  const int K0 = J0.base.K[t];
  const auto dup = [](int x) {
    const uint32_t h = (uint32_t)__half_as_ushort(__int2half_rn(x));
    return h | (h << 16);
  };
  for (int k = lane; k < N; k += 32) srow[warp][k] = eq[k] > 0 ? dup(lo[k]) : 0xffffffffu;
  __half2 av[kPasses][2], lv[kPasses][2];  // the samples' centred ranks and lo
  uint32_t pm[kPasses][2];                 // 0xffff where the sample is present
  bool ties = false;
#pragma unroll
  for (int ps = 0; ps < kPasses; ++ps)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int a[2], l[2];
      pm[ps][h] = 0u;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int k = 128 * ps + 4 * lane + 2 * h + i;
        const int e = k < N ? (int)eq[k] : 0;
        l[i] = e > 0 ? (int)lo[k] : 0;
        a[i] = e > 0 ? 2 * l[i] + e - K0 : 0;
        if (e > 0) pm[ps][h] |= 0xffffu << (16 * i);
        ties = ties || e > 1;
      }
      av[ps][h] = __halves2half2(__int2half_rn(a[0]), __int2half_rn(a[1]));
      lv[ps][h] = __halves2half2(__int2half_rn(l[0]), __int2half_rn(l[1]));
    }
  ties = __any_sync(0xffffffffu, ties);
  __syncwarp();
  int myK = K0, mytie = 0;  // bucket lane's, for the constants
  if (lane < n_jobs) {
    const int32_t *dl = staged ? sdrop + (sj[lane].drop_off - d0) : drops + sj[lane].drop_off;
    for (int d = 0; d < sj[lane].n_drop; ++d) myK -= srow[warp][dl[d]] != 0xffffffffu;
  }
  const __half2 one = __float2half2_rn(1.f), minus = __float2half2_rn(-1.f);
  const int64_t at0 = tiled ? tiled_index(t, 4 * lane, Np) : (int64_t)t * Np + 4 * lane;
  const int64_t step = tiled ? 8 * 2048 : 128;  // 128 samples on
  for (int j = 0; j < n_jobs; ++j) {
    const RerankOut &J = sj[j];
    const int n_drop = J.n_drop;
    const int32_t *dl = staged ? sdrop + (J.drop_off - d0) : drops + J.drop_off;
    __half2 x[kPasses][2];
    uint32_t m[kPasses][2];
#pragma unroll
    for (int ps = 0; ps < kPasses; ++ps)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        x[ps][h] = av[ps][h];
        m[ps][h] = pm[ps][h];
      }
    for (int d = 0; d < n_drop; ++d) {
      const int q = dl[d];
      const uint32_t w = srow[warp][q];
      if (w == 0xffffffffu) continue;  // (the dropped sample has no value)
      const __half2 lq = *reinterpret_cast<const __half2 *>(&w);
#pragma unroll
      for (int ps = 0; ps < kPasses; ++ps) {
        const unsigned int r = (unsigned int)(q - 128 * ps - 4 * lane);
        const uint32_t left = (r & 1u) ? 0x0000ffffu : 0xffff0000u;
        if (r < 2u) m[ps][0] &= left;
        if ((r & ~1u) == 2u) m[ps][1] &= left;
#pragma unroll
        for (int h = 0; h < 2; ++h)
          x[ps][h] = __hsub2(x[ps][h], __hmin2(__hmax2(__hsub2(lv[ps][h], lq), minus), one));
      }
    }
#pragma unroll
    for (int ps = 0; ps < kPasses; ++ps)
      if (128 * ps + 4 * lane < Np) {
        uint2 v;
        v.x = *reinterpret_cast<const uint32_t *>(&x[ps][0]) & m[ps][0];
        v.y = *reinterpret_cast<const uint32_t *>(&x[ps][1]) & m[ps][1];
        *reinterpret_cast<uint2 *>(J.A + at0 + ps * step) = v;
      }
    if (ties) {  // sum over the samples left of eq'^2 - 1
      int tie = 0;
#pragma unroll
      for (int ps = 0; ps < kPasses; ++ps)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = 128 * ps + 4 * lane + i;
          if (!((m[ps][i >> 1] >> (16 * (i & 1))) & 1u)) continue;
          int e = (int)eq[k];
          for (int d = 0; e > 1 && d < n_drop; ++d) e -= srow[warp][dl[d]] == srow[warp][k];
          tie += e * e - 1;
        }
      tie = (int)__reduce_add_sync(0xffffffffu, (unsigned)tie);
      if (lane == j) mytie = tie;
    }
  }
  if (lane < n_jobs) {  // the chunk's FP64 constants, one bucket per lane
    float tau;
    double cfac;
    trait_consts(myK, (long long)mytie, tau, cfac);
    sj[lane].tau[t] = tau;
    sj[lane].cfac[t] = cfac;
  }
}
}  // namespace

// One launch per run of buckets with the same base rank set (hjobs: the host copy
// of the device table djobs).  tiled: the matrices in the plain forms' layout.
cudaError_t launch_rerank_buckets(const RerankJob *djobs, const RerankJob *hjobs,
                                  const int32_t *drops, int n_jobs, bool tiled, cudaStream_t s) {
  for (int j0 = 0; j0 < n_jobs;) {
    int j1 = j0 + 1;
    while (j1 < n_jobs && hjobs[j1].base.lo == hjobs[j0].base.lo) ++j1;
    const int rows_pad = hjobs[j0].rows_pad;
    const dim3 grid((unsigned)((rows_pad + kRerankWarps - 1) / kRerankWarps),
                    (unsigned)((j1 - j0 + kRerankChunk - 1) / kRerankChunk));
    const int Np = hjobs[j0].Np;
    if (Np <= 128)
      rerank_kernel<1><<<grid, kRerankWarps * 32, 0, s>>>(djobs + j0, j1 - j0, drops, tiled);
    else if (Np <= 256)
      rerank_kernel<2><<<grid, kRerankWarps * 32, 0, s>>>(djobs + j0, j1 - j0, drops, tiled);
    else
      rerank_kernel<4><<<grid, kRerankWarps * 32, 0, s>>>(djobs + j0, j1 - j0, drops, tiled);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    j0 = j1;
  }
  return cudaSuccess;
}
}  // namespace krux
