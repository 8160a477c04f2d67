// pack.cu -- genotype packing (section "Calculation of the Kruskal-Wallis test
// statistic by matrix multiplication": the index matrices I_i(m,k) = [G(m,k) = i]
// and the group sizes N_i(m) = sum_k I_i(m,k)).
//
// Two rows per SNP are enough: with centred ranks the three rank sums satisfy D_0 + D_1 +
// D_2 = 0.  The packed operand is FP16 in chunks of 64 SNPs of 128 rows.  For the general
// forms rows [0,64) are I_0 and [64,128) I_1, each Np samples long; for the plain forms
// they are the weighted rows P and Q (PqCoef), in tiles (tiled_index).
#include <algorithm>

#include "common.cuh"

namespace krux {

namespace {
constexpr int kPackWarps = 8;

// Missing-genotype pre-pass: flags SNPs with a -1 code, appends (index, sample
// bitmask) of each such SNP, and reports codes outside {-1, 0..max_code}.
__global__ void __launch_bounds__(kPackWarps * 32)
missing_scan_kernel(const int8_t *__restrict__ geno, int64_t ldg, int N, int64_t snp_begin,
                    int64_t n_snps, int max_code, unsigned int *n_missing, int64_t *miss_idx,
                    uint64_t *miss_mask, unsigned int *status) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * kPackWarps + warp;
  if (j >= n_snps) return;
  const int8_t *g = geno + (snp_begin + j) * ldg;
  uint32_t words[kMaxN / 32];
  bool any = false, bad = false;
#pragma unroll
  for (int w = 0; w < kMaxN / 32; ++w) {
    words[w] = 0u;
    if (w * 32 < N) {  // warp-uniform
      const int k = w * 32 + lane;
      const int code = k < N ? (int)g[k] : 0;
      bad |= (code < -1 || code > max_code);
      words[w] = __ballot_sync(0xffffffffu, code == -1);
      any |= words[w] != 0u;
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kDevBadCode);
  if (!any) return;
  unsigned int slot = 0;
  if (lane == 0) slot = atomicAdd(n_missing, 1u);
  slot = __shfl_sync(0xffffffffu, slot, 0);
  if (lane == 0) miss_idx[slot] = snp_begin + j;
  if (lane < kMaxN / 64) {
    const uint64_t m = (uint64_t)words[2 * lane] | ((uint64_t)words[2 * lane + 1] << 32);
    miss_mask[(int64_t)slot * (kMaxN / 64) + lane] = m;
  }
}

// The same pre-pass for rows stored back to back (ldg == N), which is the usual
// layout: the block is read as a flat byte array with 16-byte loads, every byte
// checked four at a time; a -1 sets the bit of its SNP in `flags` (rare), a code
// outside {-1, 0..max_code} sets kDevBadCode.  base = row 0 of the range, nbytes
// = rows * N.
__device__ __forceinline__ void missing_word(uint32_t x, int64_t o, int N, uint32_t mc4,
                                             uint32_t *flags, bool &bad) {
  uint32_t ff = __vcmpeq4(x, 0xffffffffu);
  bad |= (__vcmpgtu4(x, mc4) & ~ff) != 0u;
  while (ff != 0u) {
    const int byte = (__ffs(ff) - 1) >> 3;
    const int64_t snp = (o + byte) / N;
    atomicOr(&flags[snp >> 5], 1u << (snp & 31));
    ff &= ~(0xffu << (8 * byte));
  }
}

__global__ void __launch_bounds__(256)
missing_flag_kernel(const int8_t *__restrict__ base, int64_t nbytes, int N, int max_code,
                    uint32_t *flags, unsigned int *status) {
  const uint32_t mc4 = (uint32_t)max_code * 0x01010101u;
  const int64_t head = std::min<int64_t>((16 - (int64_t)((uintptr_t)base & 15)) & 15, nbytes);
  const int64_t words = (nbytes - head) / 16;
  const int64_t tail0 = head + 16 * words;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (int64_t i = tid; i < words; i += nthreads) {
    const uint4 v = *reinterpret_cast<const uint4 *>(base + head + 16 * i);
    const int64_t o = head + 16 * i;
    missing_word(v.x, o, N, mc4, flags, bad);
    missing_word(v.y, o + 4, N, mc4, flags, bad);
    missing_word(v.z, o + 8, N, mc4, flags, bad);
    missing_word(v.w, o + 12, N, mc4, flags, bad);
  }
  // the unaligned head and the tail, one byte per thread
  const int64_t extra = head + (nbytes - tail0);
  if (tid < extra) {
    const int64_t o = tid < head ? tid : tail0 + (tid - head);
    const int code = base[o];
    if (code == -1) {
      const int64_t snp = o / N;
      atomicOr(&flags[snp >> 5], 1u << (snp & 31));
    }
    bad |= code < -1 || code > max_code;
  }
  if (bad) atomicOr(status, kDevBadCode);
}

// The flagged SNPs (bit j of flags: SNP snp_begin + j) appended as (index, sample
// bitmask), one warp per flag word.
__global__ void __launch_bounds__(256)
missing_collect_kernel(const int8_t *__restrict__ geno, int64_t ldg, int N, int64_t snp_begin,
                       int64_t n_snps, const uint32_t *__restrict__ flags, unsigned int *n_missing,
                       int64_t *miss_idx, uint64_t *miss_mask) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * 8 + warp;
  if (w * 32 >= n_snps) return;
  uint32_t bits = flags[w];
  while (bits != 0u) {
    const int bit = __ffs(bits) - 1;
    bits &= bits - 1u;
    const int64_t j = w * 32 + bit;
    const int8_t *g = geno + (snp_begin + j) * ldg;
    uint32_t words[kMaxN / 32];
#pragma unroll
    for (int q = 0; q < kMaxN / 32; ++q) {
      words[q] = 0u;
      if (q * 32 < N) {  // warp-uniform
        const int k = q * 32 + lane;
        words[q] = __ballot_sync(0xffffffffu, k < N && g[k] == -1);
      }
    }
    unsigned int slot = 0;
    if (lane == 0) slot = atomicAdd(n_missing, 1u);
    slot = __shfl_sync(0xffffffffu, slot, 0);
    if (lane == 0) miss_idx[slot] = snp_begin + j;
    if (lane < kMaxN / 64) {
      const uint64_t m = (uint64_t)words[2 * lane] | ((uint64_t)words[2 * lane + 1] << 32);
      miss_mask[(int64_t)slot * (kMaxN / 64) + lane] = m;
    }
  }
}

// ---- device-side grouping of the flagged SNPs by missing-sample pattern ----------
// (section "Handling missing values": one matrix per pattern).  An open-addressing
// table over 64-bit hashes of the sample masks (0 = empty slot) finds each pattern's
// bucket; every member's mask is then compared with its bucket representative's
// (a hash collision is reported, and the host groups on its own instead).
__device__ __forceinline__ uint64_t pattern_hash(const uint64_t *m) {
  uint64_t h = 0x9e3779b97f4a7c15ull;
#pragma unroll
  for (int w = 0; w < kMaxN / 64; ++w) h = (h ^ m[w]) * 0x100000001b3ull;
  return (h ^ (h >> 29)) | 1ull;
}

__global__ void pattern_insert_kernel(const unsigned int *__restrict__ n_missing,
                                      const uint64_t *__restrict__ mask,
                                      unsigned long long *tab_hash, int *tab_rep, int64_t cap,
                                      int *slot_of) {
  const int64_t m = *n_missing;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long h = pattern_hash(mask + i * (kMaxN / 64));
    int64_t t = (int64_t)(h & (unsigned long long)(cap - 1));
    for (int64_t probe = 0; probe < cap; ++probe) {  // the table has room for every mask
      const unsigned long long prev = atomicCAS(tab_hash + t, 0ull, h);
      if (prev == 0ull || prev == h) {
        atomicMin(tab_rep + t, (int)i);
        slot_of[i] = (int)t;
        break;
      }
      t = (t + 1) & (cap - 1);
    }
  }
}

// Numbers the occupied slots (bucket ids) and copies each bucket's representative
// mask out.
__global__ void pattern_number_kernel(const unsigned long long *__restrict__ tab_hash,
                                      const int *__restrict__ tab_rep, int64_t cap, int *tab_id,
                                      unsigned int *n_buckets, const uint64_t *__restrict__ mask,
                                      uint64_t *bucket_mask) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < cap;
       t += (int64_t)gridDim.x * blockDim.x) {
    if (tab_hash[t] == 0ull) continue;
    const int id = (int)atomicAdd(n_buckets, 1u);
    tab_id[t] = id;
    const int rep = tab_rep[t];
#pragma unroll
    for (int w = 0; w < kMaxN / 64; ++w)
      bucket_mask[(int64_t)id * (kMaxN / 64) + w] = mask[(int64_t)rep * (kMaxN / 64) + w];
  }
}

// Bucket of every flagged SNP, bucket sizes and first SNPs, and the check of every
// mask against its bucket's.
__global__ void pattern_count_kernel(const unsigned int *__restrict__ n_missing,
                                     const int *__restrict__ slot_of, const int *__restrict__ tab_id,
                                     const uint64_t *__restrict__ mask,
                                     const uint64_t *__restrict__ bucket_mask,
                                     const int64_t *__restrict__ miss_idx, int *bucket_of,
                                     unsigned int *count, unsigned long long *first,
                                     unsigned int *status) {
  const int64_t m = *n_missing;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int b = tab_id[slot_of[i]];
    bucket_of[i] = b;
    atomicAdd(count + b, 1u);
    atomicMin(first + b, (unsigned long long)miss_idx[i]);
    bool same = true;
#pragma unroll
    for (int w = 0; w < kMaxN / 64; ++w)
      same = same && mask[i * (kMaxN / 64) + w] == bucket_mask[(int64_t)b * (kMaxN / 64) + w];
    if (!same) atomicOr(status, kDevHashCollision);
  }
}

// Writes every flagged SNP into its bucket's list (offset[b] .. + count[b]).
__global__ void pattern_scatter_kernel(const unsigned int *__restrict__ n_missing,
                                       const int *__restrict__ bucket_of,
                                       const int64_t *__restrict__ offset,
                                       const int64_t *__restrict__ miss_idx, unsigned int *fill,
                                       int64_t *list) {
  const int64_t m = *n_missing;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int b = bucket_of[i];
    list[offset[b] + atomicAdd(fill + b, 1u)] = miss_idx[i];
  }
}

// The rows without a missing code, in order: one block scans the per-word counts of
// the flag bits, then every word writes its complete rows.
__global__ void __launch_bounds__(1024)
complete_offsets_kernel(const uint32_t *__restrict__ flags, int64_t n_snps, int64_t *woff) {
  __shared__ int64_t part[1024];
  const int64_t nw = (n_snps + 31) / 32;
  const int64_t per = (nw + 1023) / 1024;
  const int64_t w0 = threadIdx.x * per, w1 = w0 + per < nw ? w0 + per : nw;
  int64_t sum = 0;
  for (int64_t w = w0; w < w1; ++w) {
    const int64_t left = n_snps - 32 * w;
    const int valid = left < 32 ? (int)left : 32;
    const uint32_t vm = valid >= 32 ? 0xffffffffu : (1u << valid) - 1u;
    sum += __popc(~flags[w] & vm);
  }
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int d = 1; d < 1024; d <<= 1) {  // inclusive scan of the partial sums
    const int64_t v = threadIdx.x >= (unsigned)d ? part[threadIdx.x - d] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t run = threadIdx.x ? part[threadIdx.x - 1] : 0;
  for (int64_t w = w0; w < w1; ++w) {
    woff[w] = run;
    const int64_t left = n_snps - 32 * w;
    const int valid = left < 32 ? (int)left : 32;
    const uint32_t vm = valid >= 32 ? 0xffffffffu : (1u << valid) - 1u;
    run += __popc(~flags[w] & vm);
  }
  if (threadIdx.x == 1023) woff[nw] = part[1023];
}

__global__ void complete_scatter_kernel(const uint32_t *__restrict__ flags,
                                        const int64_t *__restrict__ woff, int64_t snp_begin,
                                        int64_t n_snps, int64_t *list) {
  const int64_t nw = (n_snps + 31) / 32;
  for (int64_t w = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; w < nw;
       w += (int64_t)gridDim.x * blockDim.x) {
    const int64_t left = n_snps - 32 * w;
    const int valid = left < 32 ? (int)left : 32;
    uint32_t bits = ~flags[w] & (valid >= 32 ? 0xffffffffu : (1u << valid) - 1u);
    int64_t o = woff[w];
    while (bits) {
      const int j = __ffs((int)bits) - 1;
      bits &= bits - 1u;
      list[o++] = snp_begin + 32 * w + j;
    }
  }
}

// Flag bits of the flagged SNPs (the pre-pass that produces no flag array).
__global__ void flags_from_idx_kernel(const unsigned int *__restrict__ n_missing,
                                      const int64_t *__restrict__ miss_idx, int64_t snp_begin,
                                      uint32_t *flags) {
  const int64_t m = *n_missing;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = miss_idx[i] - snp_begin;
    atomicOr(flags + (j >> 5), 1u << (j & 31));
  }
}

// Metadata of SNP slot jj of a chunk: group sizes, df and the coefficients of the
// hot test (zero for an excluded SNP: one with a missing code outside its bucket).
__device__ __forceinline__ void write_meta(ChunkMeta &m, int jj, int n0, int n1, int n2,
                                           bool excluded, int64_t snp_out, float rh1, float rh2,
                                           int signed_df1, int linear, float rl) {
  const int groups = (n0 > 0) + (n1 > 0) + (n2 > 0);
  const int df = groups > 0 ? groups - 1 : 0;
  float al = 0.f, be = 0.f, ga = 0.f;
  if (linear) {
    // dosage regression (parametric comparison): rl (2 S_0 + S_1)^2 / S_gg,
    // S_gg = sum over samples of (g - mean g)^2
    const int K = n0 + n1 + n2;
    const float gs = (float)n1 + 2.f * (float)n2;
    const float sgg = K > 0 ? (float)n1 + 4.f * (float)n2 - gs * gs / (float)K : 0.f;
    if (df > 0 && !excluded && sgg > 0.5f / (float)(K > 0 ? K : 1)) {
      al = 4.f * rl / sgg;
      be = 0.5f;
    }
  } else if (df > 0 && !excluded) {
    // sum_i D_i^2 / N_i with D_2 = -(u + v):  (r0 + r2) u^2 + 2 r2 u v + (r1 + r2) v^2
    //   = alpha (u + beta v)^2 + gamma v^2,  alpha = r0 + r2, beta = r2 / alpha,
    //   gamma = r1 + r2 r0 / alpha   (empty groups have r_i = 0).  FP32 is enough:
    // these only feed the thresholded test, whose band is rechecked in FP64.
    const float q0 = n0 ? 1.f / (float)n0 : 0.f, q1 = n1 ? 1.f / (float)n1 : 0.f,
                q2 = n2 ? 1.f / (float)n2 : 0.f;
    const float a = q0 + q2;
    const float rh = (df == 1 ? rh1 : rh2) * ((signed_df1 && df == 1) ? -1.f : 1.f);
    al = a * rh;
    be = q2 / a;
    ga = (q1 + q2 * q0 / a) * rh;
  }
  m.alpha[jj] = al;
  m.beta[jj] = be;
  m.gamma[jj] = ga;
  m.snp[jj] = excluded ? -1 : (int32_t)snp_out;
  m.n[0][jj] = (uint16_t)n0;
  m.n[1][jj] = (uint16_t)n1;
  m.n[2][jj] = (uint16_t)n2;
  m.df[jj] = (uint8_t)df;
}

// Weights of one SNP's packed rows in the plain forms (see ChunkMeta), and the
// group order they stand for.
struct PqCoef {
  uint32_t w0, w1;          // ChunkMeta's pq0, pq1
  float a0, a1, g;          // the weights as FP32
  int na, nb, nl;           // sizes of groups a, b and of the group left out
};
// x > 0 rounded up / to nearest at `bits` significant bits (exponent of x)
__device__ __forceinline__ float round_up_bits(float x, int bits) {
  const uint32_t m = (1u << (24 - bits)) - 1u;
  return __uint_as_float((__float_as_uint(x) + m) & ~m);
}
__device__ __forceinline__ PqCoef pq_coef(int n0, int n1, int n2, bool excluded, float rh1,
                                          float rh2, int bits) {
  PqCoef c;
  c.w0 = 0u;
  c.w1 = 1u << 18;  // a = 0, b = 1
  c.a0 = c.a1 = c.g = 0.f;
  // L: a largest group; b: a smallest one; a: the third
  const int n[3] = {n0, n1, n2};
  const int L = n0 >= n1 && n0 >= n2 ? 0 : (n1 >= n2 ? 1 : 2);
  const int x = L == 0 ? 1 : 0, y = L == 2 ? 1 : 2;
  const int nx = x == 0 ? n[0] : n[1], ny = y == 1 ? n[1] : n[2];
  const int b = nx <= ny ? x : y, a = nx <= ny ? y : x;
  c.nb = min(nx, ny);
  c.na = max(nx, ny);
  c.nl = max(n0, max(n1, n2));
  const int groups = (n0 > 0) + (n1 > 0) + (n2 > 0);
  if (groups < 2 || excluded) return c;
  // (a two-group SNP has b empty and D_b = 0: its a and L carry the form)
  const float rh = groups == 2 ? rh1 : rh2;
  const float qa = 1.f / (float)c.na, qb = c.nb > 0 ? 1.f / (float)c.nb : 0.f, ql = 1.f / (float)c.nl;
  const float s = qa + ql;
  const float alpha = s * rh, beta = ql / s;
  const float step = exp2f((float)-bits);
  // A0^2 >= alpha (1 + step), A1 = A0 (beta + d) with |d| <= 2^-bits: the largest of
  // alpha w^2 - A0^2 (w + d v)^2 over w is alpha d^2 (1 + 1/eta) v^2, eta = A0^2 / alpha
  // - 1 >= step; G^2 takes that on top of gamma (1e-5: FP32 rounding of all this)
  c.a0 = round_up_bits(sqrtf(alpha * (1.f + step)) * 1.00001f, bits);
  const uint32_t e = (__float_as_uint(c.a0) >> 23) & 255u;
  const float ulp = __uint_as_float((e - (uint32_t)(bits - 1)) << 23);  // A0's last place
  c.a1 = rintf(c.a0 * beta / ulp) * ulp;
  const float d = fabsf(c.a1 / c.a0 - beta) + 1e-6f;
  const float gamma = (qb + ql * qa / s) * rh;
  c.g = round_up_bits(sqrtf(gamma + alpha * d * d * (1.f + 1.f / step)) * 1.00001f, bits);
  c.w0 = (uint32_t)__half_as_ushort(__float2half_rn(c.a0)) |
         ((uint32_t)__half_as_ushort(__float2half_rn(c.a1)) << 16);
  c.w1 = (uint32_t)__half_as_ushort(__float2half_rn(c.g)) | ((uint32_t)a << 16) | ((uint32_t)b << 18);
  return c;
}

// The regression's only row: sqrt(alpha) (D_0 + D_1 / 2), Q = 0 (see write_meta).
__device__ __forceinline__ PqCoef pq_coef_linear(int n0, int n1, int n2, bool excluded, float rl) {
  PqCoef c{};
  c.w1 = 1u << 18;
  const int K = n0 + n1 + n2;
  const float gs = (float)n1 + 2.f * (float)n2;
  const float sgg = K > 0 ? (float)n1 + 4.f * (float)n2 - gs * gs / (float)K : 0.f;
  if (excluded || !(sgg > 0.5f / (float)(K > 0 ? K : 1))) return c;
  c.a0 = round_up_bits(sqrtf(4.f * rl / sgg) * 1.00001f, 10);
  c.w0 = (uint32_t)__half_as_ushort(__float2half_rn(c.a0)) |
         ((uint32_t)__half_as_ushort(__float2half_rn(0.5f * c.a0)) << 16);
  return c;
}

// Weights of one marker's four packed rows in the plain form (up to five groups).  With
// the groups by size, the largest left out and g_0 >= g_1 >= .. the others, the
// quadratic form sum_i D_i^2 / N_i / h_df has the Cholesky factor
//   P_i = l_i D_{g_i} + c_i sum_{k > i} D_{g_k},
//   l_i = sqrt(r_i + rho_i), c_i = rho_i / l_i, rho_0 = r_largest, rho_{i+1} = rho_i r_i / l_i^2
// (r = 1 / (N h_df)); empty groups have no row.  Rows are scaled by 1 + 4 * 2^-bits and
// rounded as PqCoef's: A_i upwards, C_i on A_i's grid.  The grid error of row i is at
// most 2^-bits l_i |sum_{k > i} D| <= 2^-bits sqrt(2 (3 - i)) times the form's root (l_i^2
// <= 2 r_i <= 2 r_k), 3.5 * 2^-bits over the rows, so sum P_i^2 never falls below the
// form (and exceeds it by about 20 * 2^-bits at most).
struct PqCoefM {
  uint32_t w[kMaxCodeM], order;
};
__device__ __forceinline__ PqCoefM pq_coef_multi(const int (&n)[kMaxCodeM + 1], bool excluded,
                                                 const float *rh, int bits) {
  PqCoefM c{};
  // codes by size, largest first (selection: five entries)
  int ord[kMaxCodeM + 1], sz[kMaxCodeM + 1];
#pragma unroll
  for (int i = 0; i <= kMaxCodeM; ++i) {
    ord[i] = i;
    sz[i] = n[i];
  }
#pragma unroll
  for (int i = 0; i < kMaxCodeM; ++i)
#pragma unroll
    for (int k = i + 1; k <= kMaxCodeM; ++k)
      if (sz[k] > sz[i]) {
        const int a = sz[i], b = ord[i];
        sz[i] = sz[k];
        ord[i] = ord[k];
        sz[k] = a;
        ord[k] = b;
      }
  int groups = 0;
#pragma unroll
  for (int i = 0; i <= kMaxCodeM; ++i) groups += n[i] > 0;
#pragma unroll
  for (int i = 0; i < kMaxCodeM; ++i) c.order |= (uint32_t)ord[i + 1] << (3 * i);
  c.order |= (uint32_t)ord[0] << 12;
  if (groups < 2 || excluded) return c;
  const float h = rh[groups - 2];
  float rho = h / (float)sz[0];
  const float up = (1.f + 4.f * exp2f((float)-bits)) * 1.00001f;
#pragma unroll
  for (int i = 0; i < kMaxCodeM; ++i) {
    if (sz[i + 1] == 0) break;
    const float r = h / (float)sz[i + 1];
    const float l2 = r + rho;
    const float a = round_up_bits(sqrtf(l2) * up, bits);
    const uint32_t e = (__float_as_uint(a) >> 23) & 255u;
    const float ulp = __uint_as_float((e - (uint32_t)(bits - 1)) << 23);
    const float cc = rintf(a * (rho / l2) / ulp) * ulp;
    c.w[i] = (uint32_t)__half_as_ushort(__float2half_rn(a)) |
             ((uint32_t)__half_as_ushort(__float2half_rn(cc)) << 16);
    rho = rho * r / l2;
  }
  return c;
}

// The plain form's coefficient sets of SNP slot jj for traits with NaN samples:
// set s takes the quadratic form from group sizes max(N_i - C, 1), C = nan_set_c(s)
// (an empty group stays empty), with the threshold of the smallest df the pair can
// keep (1/h_1 when some group may vanish).  For a trait with c <= C NaN samples it
// bounds the pair's exact sum_i D_i^2 / N_i' / h_df' from above, whichever groups the
// NaN samples fall in.  It is written on the accumulators: D_b = Q / G and D_a =
// (P - A1 D_b) / A0 turn alpha (D_a + beta D_b)^2 + gamma D_b^2 into
// alpha / A0^2 (P + (beta A0 - A1) / G Q)^2 + gamma / G^2 Q^2.
__device__ __forceinline__ void write_coef_nan(void *block, int jj, const PqCoef &w, float rh1,
                                               float rh2) {
#pragma unroll
  for (int si = 0; si < kNanSets; ++si) {
    const int c = nan_set_c(si);
    float al = 0.f, be = 0.f, ga = 0.f;
    if (w.a0 > 0.f) {  // two groups or more: groups a and L are not empty
      const int sure = (w.na > c) + (w.nb > c) + (w.nl > c);  // groups no c NaN samples can empty
      const float rh = sure >= 3 ? rh2 : rh1;
      const float qa = 1.f / (float)max(w.na - c, 1),
                  qb = w.nb ? 1.f / (float)max(w.nb - c, 1) : 0.f,
                  ql = 1.f / (float)max(w.nl - c, 1);
      const float a = qa + ql;
      al = a * rh / (w.a0 * w.a0);
      be = (ql / a * w.a0 - w.a1) / w.g;
      ga = (qb + ql * qa / a) * rh / (w.g * w.g);
    }
    CoefSet *cs = coef_set(block, si);
    cs->alpha[jj] = al;
    cs->beta[jj] = be;
    cs->gamma[jj] = ga;
  }
}

// Packs SNP slot j (one warp; j may be the padding of the last chunk).  SNP j is
// snp_list[j] if a list is given, else snp_begin + j.  SNPs that carry a missing
// code are packed with zero coefficients here (they are scanned in their
// missing-pattern bucket, where the rank set excludes those samples and the -1
// entries simply pack as 0 in both indicators).
__device__ __forceinline__ void pack_slot(const int8_t *__restrict__ geno, int64_t ldg, int N,
                                          int Np, const int64_t *__restrict__ snp_list,
                                          int64_t snp_begin, int64_t n_snps, int64_t j,
                                          int64_t snp_out_base, float rh1, float rh2,
                                          int allow_missing, int signed_df1,
                                          __half *__restrict__ B, ChunkMeta *__restrict__ meta,
                                          unsigned int *status, int linear, float rl, int lane) {
  const int64_t c = j / kChunkSnps;
  const int jj = (int)(j % kChunkSnps);
  __half *r0 = B + (c * kChunkRows + jj) * Np;
  __half *r1 = B + (c * kChunkRows + kChunkSnps + jj) * Np;
  ChunkMeta &m = meta[c];
  const __half one = __int2half_rn(1), zero = __int2half_rn(0);
  if (j >= n_snps) {
    for (int k = lane; k < Np; k += 32) {
      r0[k] = zero;
      r1[k] = zero;
    }
    if (lane == 0) {
      m.alpha[jj] = 0.f;
      m.beta[jj] = 0.f;
      m.gamma[jj] = 0.f;
      m.snp[jj] = -1;
      m.n[0][jj] = m.n[1][jj] = m.n[2][jj] = 0;
      m.df[jj] = 0;
    }
    return;
  }
  const int64_t s = snp_list ? snp_list[j] : snp_begin + j;
  const int8_t *g = geno + s * ldg;
  int n0 = 0, n1 = 0, n2 = 0;
  bool miss = false, bad = false;
  for (int k = lane; k < Np; k += 32) {
    const int code = k < N ? (int)g[k] : -1;
    r0[k] = code == 0 ? one : zero;
    r1[k] = code == 1 ? one : zero;
    n0 += code == 0;
    n1 += code == 1;
    n2 += code == 2;
    if (k < N) {
      miss |= code == -1;
      bad |= (code < -1 || code > 2);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    n0 += __shfl_xor_sync(0xffffffffu, n0, o);
    n1 += __shfl_xor_sync(0xffffffffu, n1, o);
    n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  }
  miss = __any_sync(0xffffffffu, miss);
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    if (bad) atomicOr(status, kDevBadCode);
    if (miss && !allow_missing) atomicOr(status, kDevMissing);
    write_meta(m, jj, n0, n1, n2, miss && !allow_missing, snp_out_base + s, rh1, rh2, signed_df1,
               linear, rl);
  }
}

// One warp per packed SNP slot of one SNP set.
__global__ void __launch_bounds__(kPackWarps * 32)
pack_kernel(const int8_t *__restrict__ geno, int64_t ldg, int N, int Np,
            const int64_t *__restrict__ snp_list, int64_t snp_begin, int64_t n_snps,
            int64_t n_slots, int64_t snp_out_base, float rh1, float rh2, int allow_missing,
            int signed_df1, __half *__restrict__ B, ChunkMeta *__restrict__ meta,
            unsigned int *status, int linear, float rl) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * kPackWarps + warp;
  if (j >= n_slots) return;
  pack_slot(geno, ldg, N, Np, snp_list, snp_begin, n_snps, j, snp_out_base, rh1, rh2,
            allow_missing, signed_df1, B, meta, status, linear, rl, lane);
}

// Last job whose first flattened unit is at or below x (x below the total).
__device__ __forceinline__ int find_job(const PackJob *__restrict__ jobs, int n_jobs, int64_t x,
                                        bool halves) {
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((halves ? jobs[mid].half0 : jobs[mid].slot0) <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// Four codes starting at byte offset o of the staged rows (any alignment).
__device__ __forceinline__ uint32_t stage_word(const uint8_t *st, int o) {
  const uint32_t *w = reinterpret_cast<const uint32_t *>(st + (o & ~3));
  return __funnelshift_r(w[0], w[1], 8 * (o & 3));
}
// Bytes 0..3 of a 0x00 / 0xff byte mask as two FP16 pairs holding the pair v where set.
__device__ __forceinline__ uint2 mask_to_halves(uint32_t m, uint32_t v) {
  return make_uint2(__byte_perm(m, 0u, 0x1100) & v, __byte_perm(m, 0u, 0x3322) & v);
}

// Shared-memory bytes of one warp's staged rows: a row of N codes takes
// (N + 30) / 16 * 16 bytes (16-byte granules around it, wherever it starts), and a
// batch holds 32, 16 or 8 rows.
constexpr int kStageBytes = 8 * ((kMaxN + 30) / 16 * 16);
static_assert(kStageBytes >= 32 * 128 && kStageBytes >= 16 * 256, "8, 16 and 32 rows fit");

// 16 bytes at p (aligned) into shared memory; only bytes in [lo, hi) may be read.
__device__ __forceinline__ void stage_granule(uint8_t *d, const int8_t *p, const int8_t *lo,
                                              const int8_t *hi) {
  if (p >= lo && p + 16 <= hi) {
    *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<const uint4 *>(p);
  } else {  // it crosses the matrix's first or last byte
    for (int b = 0; b < 16; ++b)
      if (p + b >= lo && p + b < hi) d[b] = (uint8_t)p[b];
  }
}

// All SNP sets of a call in one launch (rank-sum form): one warp per 32 flattened
// slots (half a chunk; every job spans whole chunks).  The warp stages batches of
// genotype rows in shared memory with 16-byte loads (any row order, alignment and
// leading dimension), counts the groups of each row (32 / batch lanes per row),
// derives the rows' weights (ChunkMeta: 0/1 indicators or the plain forms' P and Q
// rows), and writes both packed rows with 16-byte stores.  Bound by the stores (4 Np
// bytes per SNP against N read): one pass over the genotypes per SNP, so the group
// sizes are known before the rows that are scaled by them are written.
// kMulti: markers with up to five groups in the plain form's layout (chunks of 32 SNPs,
// four rows each).
struct RecipH {
  float r[4];  // 1 / h_df
};
template <bool kMulti>
__global__ void __launch_bounds__(kPackWarps * 32)
pack_batch_kernel(const PackJob *__restrict__ jobs, int n_jobs, int64_t total_slots, RecipH rh,
                  int signed_df1, unsigned int *status) {
  const float rh1 = rh.r[0], rh2 = rh.r[1];
  __shared__ __align__(16) uint8_t stage[kPackWarps][kStageBytes + 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t x0 = ((int64_t)blockIdx.x * kPackWarps + warp) * 32;
  if (x0 >= total_slots) return;
  const PackJob &J = jobs[find_job(jobs, n_jobs, x0, false)];
  const int64_t j0 = x0 - J.slot0;  // a multiple of 32
  const int N = J.N, Np = J.Np, bits = J.pq_bits;
  const int64_t ldg = J.ldg;
  const int8_t *__restrict__ geno = J.geno;
  const int8_t *lo_end = J.geno_lo, *hi_end = J.geno_hi;
  uint8_t *st = stage[warp];
  const int pitch = (N + 30) / 16 * 16, cpr = pitch / 16;
  const int lgr = pitch <= 128 ? 5 : (pitch <= 256 ? 4 : 3);
  const int R = 1 << lgr, L = 32 >> lgr;  // rows per batch, lanes per row
  const int per_row = Np / 8;
  // t / per_row and t / cpr for t < 1024 as multiplications (divisors up to 66)
  const uint32_t inv_row = (65536u + (uint32_t)per_row - 1u) / (uint32_t)per_row;
  const uint32_t inv_cpr = (65536u + (uint32_t)cpr - 1u) / (uint32_t)cpr;
  // consecutive rows are staged as the one span they form, others row by row
  const bool span = J.snp_list == nullptr && (int64_t)R * ldg + 32 <= kStageBytes;
  constexpr int kSnps = kMulti ? kChunkSnpsM : kChunkSnps;
  const int64_t c = j0 / kSnps;
  const int jj0 = (int)(j0 % kSnps);
  ChunkMeta &m = J.meta[c];
  __half *Bc = J.B + c * kChunkRows * Np;
  bool any_bad = false, any_excl = false;
  // lane i: the genotype row of slot i (-1: padding of the last chunk)
  int64_t my_row = -1;
  if (j0 + lane < J.n_snps) my_row = J.snp_list ? J.snp_list[j0 + lane] : J.snp_begin + j0 + lane;
  for (int r0 = 0; r0 < 32; r0 += R) {
    const int64_t row0 = __shfl_sync(0xffffffffu, my_row, r0);
    if (span) {
      if (row0 >= 0) {
        const int64_t last = min((int64_t)R, J.n_snps - j0 - r0) - 1;
        const int8_t *src = geno + row0 * ldg;
        const int pad = (int)((uintptr_t)src & 15u);
        const int len = pad + (int)(last * ldg) + N;
        for (int o = 16 * lane; o < len; o += 512) stage_granule(st + o, src - pad + o, lo_end, hi_end);
      }
    } else {
      for (int t0 = 0; t0 < R * cpr; t0 += 32) {
        const int t = t0 + lane;
        const int r = (int)(((uint32_t)t * inv_cpr) >> 16), q = t - r * cpr;
        const int64_t row = __shfl_sync(0xffffffffu, my_row, (r0 + r) & 31);
        if (t < R * cpr && row >= 0) {
          const int8_t *src = geno + row * ldg;
          const int pad = (int)((uintptr_t)src & 15u);
          if (16 * q < pad + N)
            stage_granule(st + r * pitch + 16 * q, src - pad + 16 * q, lo_end, hi_end);
        }
      }
    }
    __syncwarp();
    // lanes L r .. L r + L - 1: the group sizes, missing and invalid codes of row r
    const int mr = lane >> (5 - lgr), sub = lane & (L - 1);
    const int64_t row = __shfl_sync(0xffffffffu, my_row, r0 + mr);
    int n0 = 0, n1 = 0, n2 = 0, n3 = 0, n4 = 0, nm = 0;
    const int o0 = row < 0 ? 0
                   : span  ? (int)((uintptr_t)(geno + row0 * ldg) & 15u) + mr * (int)ldg
                           : mr * pitch + (int)((uintptr_t)(geno + row * ldg) & 15u);
    if (row >= 0) {
      for (int k = 4 * sub; k < N; k += 4 * L) {
        uint32_t w = stage_word(st, o0 + k);
        const int v = min(N - k, 4);
        const uint32_t vm = v >= 4 ? 0xffffffffu : (1u << (8 * v)) - 1u;
        w = (w & vm) | (0x07070707u & ~vm);  // 7: outside every class below
        n0 += __popc(__vcmpeq4(w, 0u)) >> 3;
        n1 += __popc(__vcmpeq4(w, 0x01010101u)) >> 3;
        n2 += __popc(__vcmpeq4(w, 0x02020202u)) >> 3;
        nm += __popc(__vcmpeq4(w, 0xffffffffu)) >> 3;
        if (kMulti) {
          n3 += __popc(__vcmpeq4(w, 0x03030303u)) >> 3;
          n4 += __popc(__vcmpeq4(w, 0x04040404u)) >> 3;
        }
      }
    }
    for (int o = 1; o < L; o <<= 1) {
      n0 += __shfl_xor_sync(0xffffffffu, n0, o);
      n1 += __shfl_xor_sync(0xffffffffu, n1, o);
      n2 += __shfl_xor_sync(0xffffffffu, n2, o);
      nm += __shfl_xor_sync(0xffffffffu, nm, o);
      if (kMulti) {
        n3 += __shfl_xor_sync(0xffffffffu, n3, o);
        n4 += __shfl_xor_sync(0xffffffffu, n4, o);
      }
    }
    const bool excl = row >= 0 && nm > 0 && !J.allow_missing;
    any_bad |= row >= 0 && n0 + n1 + n2 + n3 + n4 + nm != N;
    any_excl |= excl;
    if constexpr (kMulti) {
      const int n[kMaxCodeM + 1] = {n0, n1, n2, n3, n4};
      const PqCoefM w = pq_coef_multi(n, row < 0 || excl, rh.r, bits);
      if (sub == 0) {
        ChunkMetaM &mm = reinterpret_cast<ChunkMetaM &>(m);
        const int jj = jj0 + r0 + mr;
        const int groups = (n0 > 0) + (n1 > 0) + (n2 > 0) + (n3 > 0) + (n4 > 0);
        const float h = groups > 1 && row >= 0 && !excl ? rh.r[groups - 2] : 0.f;
#pragma unroll
        for (int i = 0; i <= kMaxCodeM; ++i) {
          mm.coef[i][jj] = n[i] > 0 ? h / (float)n[i] : 0.f;
          mm.n[i][jj] = (uint16_t)n[i];
        }
        mm.snp[jj] = row < 0 || excl ? -1 : (int32_t)row;
        mm.df[jj] = (uint8_t)(groups > 0 ? groups - 1 : 0);
#pragma unroll
        for (int i = 0; i < kMaxCodeM; ++i) mm.pq[i][jj] = w.w[i];
        mm.order[jj] = w.order;
      }
      for (int t0 = 0; t0 < R * per_row; t0 += 32) {
        const int t = t0 + lane;
        const int r = (t >> 1) & (R - 1), k8 = 16 * (t >> (lgr + 1)) + 8 * (t & 1);
        const int ln = (r << (5 - lgr)) & 31;
        uint32_t wt[kMaxCodeM];
#pragma unroll
        for (int i = 0; i < kMaxCodeM; ++i) wt[i] = __shfl_sync(0xffffffffu, w.w[i], ln);
        const uint32_t order = __shfl_sync(0xffffffffu, w.order, ln);
        const int ob = __shfl_sync(0xffffffffu, row >= 0 ? o0 : -1, ln);
        if (t >= R * per_row) continue;
        uint32_t x[2] = {0x07070707u, 0x07070707u};
        if (ob >= 0) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int v = min(max(N - k8 - 4 * q, 0), 4);
            const uint32_t vm = v >= 4 ? 0xffffffffu : (1u << (8 * v)) - 1u;
            x[q] = (stage_word(st, ob + k8 + 4 * q) & vm) | (0x07070707u & ~vm);
          }
        }
        uint32_t later[2] = {0u, 0u};  // samples in groups g_k, k > i
#pragma unroll
        for (int i = kMaxCodeM - 1; i >= 0; --i) {
          const uint32_t code = ((order >> (3 * i)) & 7u) * 0x01010101u;
          const uint32_t va = __byte_perm(wt[i], 0u, 0x1010), vc = __byte_perm(wt[i], 0u, 0x3232);
          uint32_t o4[4];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const uint32_t in = __vcmpeq4(x[q], code);
            const uint2 a = mask_to_halves(in, va), b = mask_to_halves(later[q], vc);
            o4[2 * q] = a.x | b.x;
            o4[2 * q + 1] = a.y | b.y;
            later[q] |= in;
          }
          *reinterpret_cast<uint4 *>(Bc + tiled_index(kChunkSnpsM * i + jj0 + r0 + r, k8, Np)) =
              make_uint4(o4[0], o4[1], o4[2], o4[3]);
        }
      }
      __syncwarp();
      continue;
    }
    PqCoef w;
    w.w0 = 0x3c00u;  // 0/1 indicators of groups 0 and 1
    w.w1 = 0x3c00u | (1u << 18);
    if (bits > 0)
      w = J.linear ? pq_coef_linear(n0, n1, n2, row < 0 || excl, J.rl)
                   : pq_coef(n0, n1, n2, row < 0 || excl, rh1, rh2, bits);
    if (sub == 0) {
      const int jj = jj0 + r0 + mr;
      write_meta(m, jj, n0, n1, n2, row < 0 || excl, row < 0 ? 0 : row, rh1, rh2, signed_df1,
                 J.linear, J.rl);
      if (bits > 0) {
        m.pq0[jj] = w.w0;
        m.pq1[jj] = w.w1;
        const int groups = row < 0 || excl ? 0 : (n0 > 0) + (n1 > 0) + (n2 > 0);
        m.sgn[jj] = groups < 2 ? 0.f : (signed_df1 && groups == 2 ? -1.f : 1.f);
        if (J.coef_nan)
          write_coef_nan(reinterpret_cast<uint8_t *>(J.codes) + c * kCoefNanBytes, jj, w, rh1, rh2);
      }
    }
    // both packed rows: item t = row r, samples 8q .. 8q + 7; the plain forms' layout
    // is walked atom by atom, so that consecutive lanes fill consecutive rows' bytes
    for (int t0 = 0; t0 < R * per_row; t0 += 32) {
      const int t = t0 + lane;
      const int r = bits != 0 ? (t >> 1) & (R - 1) : (int)(((uint32_t)t * inv_row) >> 16);
      const int k8 = bits != 0 ? 16 * (t >> (lgr + 1)) + 8 * (t & 1) : 8 * (t - r * per_row);
      const int ln = (r << (5 - lgr)) & 31;
      const uint32_t w0 = __shfl_sync(0xffffffffu, w.w0, ln), w1 = __shfl_sync(0xffffffffu, w.w1, ln);
      const int ob = __shfl_sync(0xffffffffu, row >= 0 ? o0 : -1, ln);
      if (t >= R * per_row) continue;
      uint32_t lo = 0x03030303u, hi = 0x03030303u;  // 3: in no group
      if (ob >= 0) {
        lo = stage_word(st, ob + k8);
        hi = stage_word(st, ob + k8 + 4);
        // samples at or beyond N are padding
        const int vl = min(max(N - k8, 0), 4), vh = min(max(N - k8 - 4, 0), 4);
        const uint32_t ml = vl >= 4 ? 0xffffffffu : (1u << (8 * vl)) - 1u;
        const uint32_t mh = vh >= 4 ? 0xffffffffu : (1u << (8 * vh)) - 1u;
        lo = (lo & ml) | (0x03030303u & ~ml);
        hi = (hi & mh) | (0x03030303u & ~mh);
      }
      const uint32_t ca = ((w1 >> 16) & 3u) * 0x01010101u, cb = ((w1 >> 18) & 3u) * 0x01010101u;
      const uint32_t va = __byte_perm(w0, 0u, 0x1010), vb = __byte_perm(w0, 0u, 0x3232),
                     vg = __byte_perm(w1, 0u, 0x1010);
      const uint32_t la = __vcmpeq4(lo, ca), ha = __vcmpeq4(hi, ca);
      const uint32_t lb = __vcmpeq4(lo, cb), hb = __vcmpeq4(hi, cb);
      const uint2 p0 = mask_to_halves(la, va), p1 = mask_to_halves(lb, vb);
      const uint2 p2 = mask_to_halves(ha, va), p3 = mask_to_halves(hb, vb);
      const uint2 q0 = mask_to_halves(lb, vg), q1 = mask_to_halves(hb, vg);
      const int rp = jj0 + r0 + r, rq = kChunkSnps + rp;  // rows of the chunk
      const int64_t ap = bits != 0 ? tiled_index(rp, k8, Np) : (int64_t)rp * Np + k8;
      const int64_t aq = bits != 0 ? tiled_index(rq, k8, Np) : (int64_t)rq * Np + k8;
      *reinterpret_cast<uint4 *>(Bc + ap) = make_uint4(p0.x | p1.x, p0.y | p1.y, p2.x | p3.x, p2.y | p3.y);
      *reinterpret_cast<uint4 *>(Bc + aq) = make_uint4(q0.x, q0.y, q1.x, q1.y);
    }
    __syncwarp();
  }
  if (__any_sync(0xffffffffu, any_bad) && lane == 0) atomicOr(status, kDevBadCode);
  if (__any_sync(0xffffffffu, any_excl) && lane == 0) atomicOr(status, kDevMissing);
}

__device__ __forceinline__ uint64_t spread_bits(uint32_t v) {
  uint64_t x = v;
  x = (x | (x << 16)) & 0x0000FFFF0000FFFFull;
  x = (x | (x << 8)) & 0x00FF00FF00FF00FFull;
  x = (x | (x << 4)) & 0x0F0F0F0F0F0F0F0Full;
  x = (x | (x << 2)) & 0x3333333333333333ull;
  x = (x | (x << 1)) & 0x5555555555555555ull;
  return x;
}

// 2-bit genotype codes per chunk and sample: word [c][k][h] holds, at bits
// 2j..2j+1, the code of SNP 64c + 32h + j at sample k (0,1,2; 3 = missing or
// padding).  Used by the epilogue to drop a trait's NaN samples from N_i.  One
// warp per chunk half hw = 2c + h.
__device__ __forceinline__ void codes_half(const int8_t *__restrict__ geno, int64_t ldg, int N,
                                           int Np, const int64_t *__restrict__ snp_list,
                                           int64_t snp_begin, int64_t n_snps, int64_t hw,
                                           uint64_t *__restrict__ codes, int lane) {
  const int64_t j = hw * 32 + lane;
  const int8_t *g = nullptr;
  if (j < n_snps) g = geno + (snp_list ? snp_list[j] : snp_begin + j) * ldg;
  const int64_t c = hw >> 1;
  const int h = (int)(hw & 1);
  for (int k = 0; k < Np; ++k) {
    int code = 3;
    if (g && k < N) {
      const int v = g[k];
      code = (v >= 0 && v <= 2) ? v : 3;
    }
    const uint32_t b0 = __ballot_sync(0xffffffffu, code & 1);
    const uint32_t b1 = __ballot_sync(0xffffffffu, (code >> 1) & 1);
    if (lane == 0) codes[(c * Np + k) * 2 + h] = spread_bits(b0) | (spread_bits(b1) << 1);
  }
}

__global__ void __launch_bounds__(kPackWarps * 32)
codes_kernel(const int8_t *__restrict__ geno, int64_t ldg, int N, int Np,
             const int64_t *__restrict__ snp_list, int64_t snp_begin, int64_t n_snps,
             int64_t n_halves, uint64_t *__restrict__ codes) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t hw = (int64_t)blockIdx.x * kPackWarps + warp;  // chunk * 2 + half
  if (hw >= n_halves) return;
  codes_half(geno, ldg, N, Np, snp_list, snp_begin, n_snps, hw, codes, lane);
}

// The same for all SNP sets of a call that have codes (one warp per flattened half).
__global__ void __launch_bounds__(kPackWarps * 32)
codes_batch_kernel(const PackJob *__restrict__ jobs, int n_jobs, int64_t total_halves) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t x = (int64_t)blockIdx.x * kPackWarps + warp;
  if (x >= total_halves) return;
  const PackJob &J = jobs[find_job(jobs, n_jobs, x, true)];
  if (J.codes == nullptr || J.coef_nan) return;  // (such jobs span no halves)
  codes_half(J.geno, J.ldg, J.N, J.Np, J.snp_list, J.snp_begin, J.n_snps, x - J.half0, J.codes,
             lane);
}

// Markers with codes 0..4: one warp per packed SNP slot j of a 32-SNP chunk;
// rows 32i + jj (i = 0..3) of chunk j / 32 get I_i, the metadata the group
// sizes and coefficients (1 / N_i) / h_df (group 4's weighs (D_0+..+D_3)^2).
__global__ void __launch_bounds__(kPackWarps * 32)
pack_multi_kernel(const int8_t *__restrict__ geno, int64_t ldg, int N, int Np,
                  const int64_t *__restrict__ snp_list, int64_t snp_begin, int64_t n_snps,
                  int64_t n_slots, float rh1, float rh2, float rh3, float rh4, int allow_missing,
                  __half *__restrict__ B, ChunkMetaM *__restrict__ meta, unsigned int *status) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t j = (int64_t)blockIdx.x * kPackWarps + warp;
  if (j >= n_slots) return;
  const int64_t c = j / kChunkSnpsM;
  const int jj = (int)(j % kChunkSnpsM);
  __half *rows[kMaxCodeM];
#pragma unroll
  for (int i = 0; i < kMaxCodeM; ++i) rows[i] = B + (c * kChunkRows + kChunkSnpsM * i + jj) * Np;
  ChunkMetaM &m = meta[c];
  const __half one = __int2half_rn(1), zero = __int2half_rn(0);
  const int64_t s = j < n_snps ? (snp_list ? snp_list[j] : snp_begin + j) : -1;
  const int8_t *g = s >= 0 ? geno + s * ldg : nullptr;
  int cnt[kMaxCodeM + 1] = {0, 0, 0, 0, 0};
  bool miss = false, bad = false;
  for (int k = lane; k < Np; k += 32) {
    const int code = (g != nullptr && k < N) ? (int)g[k] : -1;
#pragma unroll
    for (int i = 0; i < kMaxCodeM; ++i) rows[i][k] = code == i ? one : zero;
#pragma unroll
    for (int i = 0; i <= kMaxCodeM; ++i) cnt[i] += code == i;
    if (g != nullptr && k < N) {
      miss |= code == -1;
      bad |= (code < -1 || code > kMaxCodeM);
    }
  }
#pragma unroll
  for (int i = 0; i <= kMaxCodeM; ++i)
    for (int o = 16; o > 0; o >>= 1) cnt[i] += __shfl_xor_sync(0xffffffffu, cnt[i], o);
  miss = __any_sync(0xffffffffu, miss);
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    if (bad) atomicOr(status, kDevBadCode);
    if (miss && !allow_missing) atomicOr(status, kDevMissing);
    int groups = 0;
#pragma unroll
    for (int i = 0; i <= kMaxCodeM; ++i) groups += cnt[i] > 0;
    const int df = groups > 0 ? groups - 1 : 0;
    const bool excluded = g == nullptr || (miss && !allow_missing);
    const float rh = df == 1 ? rh1 : df == 2 ? rh2 : df == 3 ? rh3 : rh4;
#pragma unroll
    for (int i = 0; i <= kMaxCodeM; ++i) {
      m.coef[i][jj] = (df > 0 && !excluded && cnt[i] > 0) ? rh / (float)cnt[i] : 0.f;
      m.n[i][jj] = (uint16_t)cnt[i];
    }
    m.snp[jj] = excluded ? -1 : (int32_t)s;
    m.df[jj] = (uint8_t)df;
  }
}
}  // namespace

cudaError_t launch_pack_multi(const int8_t *geno, int64_t ldg, int N, int Np,
                              const int64_t *snp_list, int64_t snp_begin, int64_t n_snps,
                              const double *h, int allow_missing, __half *B, ChunkMetaM *meta,
                              unsigned int *status, cudaStream_t s) {
  const int64_t nchunks = (n_snps + kChunkSnpsM - 1) / kChunkSnpsM;
  const int64_t n_slots = nchunks * kChunkSnpsM;
  if (n_slots == 0) return cudaSuccess;
  const int64_t grid = (n_slots + kPackWarps - 1) / kPackWarps;
  pack_multi_kernel<<<(unsigned)grid, kPackWarps * 32, 0, s>>>(
      geno, ldg, N, Np, snp_list, snp_begin, n_snps, n_slots, (float)(1.0 / h[0]),
      (float)(1.0 / h[1]), (float)(1.0 / h[2]), (float)(1.0 / h[3]), allow_missing, B, meta,
      status);
  return cudaGetLastError();
}

// Packing for the dosage regression of the parametric comparison: the same
// indicators, coefficients rl (2 S_0 + S_1)^2 / S_gg (rl = 1 / ((K-1) r_c^2)).
cudaError_t launch_pack_linear(const int8_t *geno, int64_t ldg, int N, int Np, int64_t snp_begin,
                               int64_t n_snps, double rl, __half *B, ChunkMeta *meta,
                               unsigned int *status, cudaStream_t s) {
  const int64_t nchunks = (n_snps + kChunkSnps - 1) / kChunkSnps;
  const int64_t n_slots = nchunks * kChunkSnps;
  if (n_slots == 0) return cudaSuccess;
  const int64_t grid = (n_slots + kPackWarps - 1) / kPackWarps;
  pack_kernel<<<(unsigned)grid, kPackWarps * 32, 0, s>>>(geno, ldg, N, Np, nullptr, snp_begin, n_snps,
                                                         n_slots, 0, 0.f, 0.f, 0, 0, B, meta, status,
                                                         1, (float)rl);
  return cudaGetLastError();
}

cudaError_t launch_missing_scan(const int8_t *geno, int64_t ldg, int N, int64_t snp_begin,
                                int64_t n_snps, int max_code, unsigned int *n_missing,
                                int64_t *miss_idx, uint64_t *miss_mask, unsigned int *status,
                                uint32_t *flags, cudaStream_t s) {
  if (n_snps <= 0) return cudaSuccess;
  if (flags != nullptr && ldg == N) {  // rows back to back: the flat pre-pass
    cudaError_t e = cudaMemsetAsync(flags, 0, (size_t)((n_snps + 31) / 32) * 4, s);
    if (e != cudaSuccess) return e;
    const int64_t nbytes = n_snps * (int64_t)N;
    const int64_t words = nbytes / 16 + 32;
    const int64_t blocks = std::min<int64_t>((words + 255) / 256, 152 * 16);
    missing_flag_kernel<<<(unsigned)blocks, 256, 0, s>>>(geno + snp_begin * ldg, nbytes, N,
                                                         max_code, flags, status);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int64_t fw = (n_snps + 31) / 32;
    missing_collect_kernel<<<(unsigned)((fw + 7) / 8), 256, 0, s>>>(geno, ldg, N, snp_begin, n_snps,
                                                                   flags, n_missing, miss_idx,
                                                                   miss_mask);
    return cudaGetLastError();
  }
  const int64_t grid = (n_snps + kPackWarps - 1) / kPackWarps;
  missing_scan_kernel<<<(unsigned)grid, kPackWarps * 32, 0, s>>>(geno, ldg, N, snp_begin, n_snps,
                                                                 max_code, n_missing, miss_idx,
                                                                 miss_mask, status);
  return cudaGetLastError();
}

cudaError_t launch_pack2(const int8_t *geno, int64_t ldg, int N, int Np, const int64_t *snp_list,
                         int64_t snp_begin, int64_t n_snps, int64_t snp_out_base, double h1,
                         double h2, int allow_missing, int signed_df1, __half *B,
                         ChunkMeta *meta, uint64_t *codes, unsigned int *status, cudaStream_t s) {
  const int64_t nchunks = (n_snps + kChunkSnps - 1) / kChunkSnps;
  const int64_t n_slots = nchunks * kChunkSnps;
  if (n_slots == 0) return cudaSuccess;
  const int64_t grid = (n_slots + kPackWarps - 1) / kPackWarps;
  pack_kernel<<<(unsigned)grid, kPackWarps * 32, 0, s>>>(geno, ldg, N, Np, snp_list, snp_begin,
                                                         n_snps, n_slots, snp_out_base,
                                                         (float)(1.0 / h1), (float)(1.0 / h2),
                                                         allow_missing, signed_df1, B, meta, status,
                                                         0, 0.f);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || codes == nullptr) return e;
  const int64_t n_halves = nchunks * 2;
  const int64_t grid2 = (n_halves + kPackWarps - 1) / kPackWarps;
  codes_kernel<<<(unsigned)grid2, kPackWarps * 32, 0, s>>>(geno, ldg, N, Np, snp_list, snp_begin,
                                                           n_snps, n_halves, codes);
  return cudaGetLastError();
}

cudaError_t launch_pack_batch(const PackJob *jobs, int n_jobs, int64_t total_slots,
                              int64_t total_halves, const double *h, bool multi, int signed_df1,
                              unsigned int *status, cudaStream_t s) {
  if (n_jobs <= 0) return cudaSuccess;
  if (total_slots > 0) {
    const int64_t warps = (total_slots + 31) / 32;
    const int64_t grid = (warps + kPackWarps - 1) / kPackWarps;
    RecipH rh{};
    for (int d = 0; d < (multi ? 4 : 2); ++d) rh.r[d] = (float)(1.0 / h[d]);
    if (multi)
      pack_batch_kernel<true><<<(unsigned)grid, kPackWarps * 32, 0, s>>>(jobs, n_jobs, total_slots, rh,
                                                                        signed_df1, status);
    else
      pack_batch_kernel<false><<<(unsigned)grid, kPackWarps * 32, 0, s>>>(jobs, n_jobs, total_slots, rh,
                                                                         signed_df1, status);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (total_halves > 0) {
    const int64_t grid = (total_halves + kPackWarps - 1) / kPackWarps;
    codes_batch_kernel<<<(unsigned)grid, kPackWarps * 32, 0, s>>>(jobs, n_jobs, total_halves);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

cudaError_t launch_pattern_group(const unsigned int *n_missing, const uint64_t *mask,
                                 const int64_t *miss_idx, int64_t n_snps, PatternScratch &w,
                                 unsigned int *status, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(w.tab_hash, 0, (size_t)w.cap * 8, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.tab_rep, 0x7f, (size_t)w.cap * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.n_buckets, 0, 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.count, 0, (size_t)n_snps * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.fill, 0, (size_t)n_snps * 4, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w.first, 0xff, (size_t)n_snps * 8, s);
  if (e != cudaSuccess) return e;
  const unsigned g1 = (unsigned)std::min<int64_t>((n_snps + 255) / 256, 152 * 8);
  const unsigned g2 = (unsigned)std::min<int64_t>((w.cap + 255) / 256, 152 * 8);
  pattern_insert_kernel<<<g1, 256, 0, s>>>(n_missing, mask, w.tab_hash, w.tab_rep, w.cap, w.slot_of);
  pattern_number_kernel<<<g2, 256, 0, s>>>(w.tab_hash, w.tab_rep, w.cap, w.tab_id, w.n_buckets, mask,
                                           w.bucket_mask);
  pattern_count_kernel<<<g1, 256, 0, s>>>(n_missing, w.slot_of, w.tab_id, mask, w.bucket_mask,
                                          miss_idx, w.bucket_of, w.count, w.first, status);
  return cudaGetLastError();
}

cudaError_t launch_pattern_lists(const unsigned int *n_missing, const int64_t *miss_idx,
                                 const uint32_t *flags, bool flags_ready, int64_t snp_begin,
                                 int64_t n_snps, PatternScratch &w, int64_t *bucket_list,
                                 int64_t *complete_list, cudaStream_t s) {
  const unsigned g1 = (unsigned)std::min<int64_t>((n_snps + 255) / 256, 152 * 8);
  const int64_t nw = (n_snps + 31) / 32;
  uint32_t *fl = const_cast<uint32_t *>(flags);
  if (!flags_ready) {
    cudaError_t e = cudaMemsetAsync(fl, 0, (size_t)nw * 4, s);
    if (e != cudaSuccess) return e;
    flags_from_idx_kernel<<<g1, 256, 0, s>>>(n_missing, miss_idx, snp_begin, fl);
  }
  pattern_scatter_kernel<<<g1, 256, 0, s>>>(n_missing, w.bucket_of, w.offset, miss_idx, w.fill,
                                            bucket_list);
  complete_offsets_kernel<<<1, 1024, 0, s>>>(flags, n_snps, w.woff);
  complete_scatter_kernel<<<(unsigned)std::min<int64_t>((nw + 255) / 256, 152 * 8), 256, 0, s>>>(
      flags, w.woff, snp_begin, n_snps, complete_list);
  return cudaGetLastError();
}

namespace {
// One thread per neighbouring pair of coordinates.
__global__ void order_kernel(const int64_t *__restrict__ a, int64_t n, const int64_t *__restrict__ b,
                             int64_t m, unsigned int *status) {
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i + 1 < n || i + 1 < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (i + 1 < n) bad |= a[i] > a[i + 1];
    if (i + 1 < m) bad |= b[i] > b[i + 1];
  }
  if (bad) atomicOr(status, kDevUnsorted);
}

// First index of the nondecreasing a[0..n) with a[i] >= x (or > x).
template <bool kAfter>
__device__ __forceinline__ int bound_of(const int64_t *__restrict__ a, int n, int64_t x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (kAfter ? a[mid] <= x : a[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// One warp per B tile: the range of its SNP rows (lists need not be in order), whose
// ends carry its smallest and largest coordinate, and the trait tiles within the
// window of that range.
__global__ void cis_items_kernel(const CisGroup *__restrict__ groups, int n_groups, int64_t n_tiles,
                                 const int64_t *__restrict__ snp_pos,
                                 const int64_t *__restrict__ trait_pos, int T, int64_t window,
                                 WorkItem *__restrict__ items, int32_t *__restrict__ n_items) {
  const int lane = threadIdx.x & 31;
  const int64_t x = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (x >= n_tiles) return;
  int gi = 0;
  for (int lo = 0, hi = n_groups - 1; lo < hi;) {
    const int mid = (lo + hi + 1) >> 1;
    if (groups[mid].tile0 <= x) lo = mid; else hi = mid - 1;
    gi = lo;
  }
  const CisGroup g = groups[gi];
  const int64_t b = x - g.tile0, j0 = b * g.tile_snps;
  const int64_t j1 = j0 + g.tile_snps < g.n_snps ? j0 + g.tile_snps : g.n_snps;
  int64_t first = INT64_MAX, last = -1;
  if (g.snp_list) {
    for (int64_t j = j0 + lane; j < j1; j += 32) {
      const int64_t r = g.snp_list[j];
      first = r < first ? r : first;
      last = r > last ? r : last;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const int64_t f = __shfl_xor_sync(0xffffffffu, first, o), l = __shfl_xor_sync(0xffffffffu, last, o);
      first = f < first ? f : first;
      last = l > last ? l : last;
    }
  } else if (j0 < j1) {
    first = g.snp_begin + j0;
    last = g.snp_begin + j1 - 1;
  }
  if (lane != 0 || last < 0) return;
  const int64_t lo = snp_pos[first], hi = snp_pos[last];
  // (a window that leaves the integers' range reaches to the end)
  const int t0 = lo < INT64_MIN + window ? 0 : bound_of<false>(trait_pos, T, lo - window);
  const int t1 = hi > INT64_MAX - window ? T : bound_of<true>(trait_pos, T, hi + window);
  if (t0 >= t1) return;
  WorkItem w;
  w.group = g.group;
  w.btile = (int32_t)b;
  w.step_begin = t0 / kTileM;
  w.step_end = (t1 - 1) / kTileM + 1;
  items[atomicAdd(n_items, 1)] = w;
}
}  // namespace

cudaError_t launch_cis_order(const int64_t *snp_pos, int64_t S, const int64_t *trait_pos, int T,
                             unsigned int *status, cudaStream_t s) {
  const int64_t most = S > T ? S : T;
  if (most > 1)
    order_kernel<<<(unsigned)std::min<int64_t>((most + 255) / 256, 152 * 8), 256, 0, s>>>(
        snp_pos, S, trait_pos, T, status);
  return cudaGetLastError();
}

cudaError_t launch_cis_items(const CisGroup *groups, int n_groups, int64_t n_tiles,
                             const int64_t *snp_pos, const int64_t *trait_pos, int T,
                             int64_t window, WorkItem *items, int32_t *n_items, cudaStream_t s) {
  if (n_tiles > 0)
    cis_items_kernel<<<(unsigned)((n_tiles + 7) / 8), 256, 0, s>>>(groups, n_groups, n_tiles, snp_pos,
                                                                   trait_pos, T, window, items, n_items);
  return cudaGetLastError();
}

// ---- SNP order of a permutation batch --------------------------------------
// The plain permutation forms test a 16-SNP block against one bound where its SNPs are of
// one df class, and pick a bound per SNP where they are mixed: half as many operations
// again and a shared-memory word per SNP.  So a large batch's SNPs are packed class by
// class, df-2 ones first, each class in its own order.  Three small launches: a class bit
// per SNP, the bits' prefix sums, the list.
namespace {

// Bit i of words[w]: SNP 32 w + i has exactly two genotype groups.  One warp per word.
__global__ void class_bits_kernel(const int8_t *__restrict__ geno, int64_t ldg, int N,
                                  int64_t n_snps, uint32_t *__restrict__ words, int64_t n_words) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  if (w >= n_words) return;
  const int n = (int)min((int64_t)32, n_snps - 32 * w);
  const int8_t *g = geno + 32 * w * ldg;
  uint32_t bits = 0u;
#pragma unroll 4
  for (int i = 0; i < n; ++i, g += ldg) {
    uint32_t seen = 0u;  // genotypes 0, 1, 2
    for (int k = lane; k < N; k += 32) seen |= 1u << (g[k] & 3);
    seen = __reduce_or_sync(0xffffffffu, seen) & 7u;
    bits |= (__popc(seen) == 2 ? 1u : 0u) << i;
  }
  if (lane == 0) words[w] = bits;
}

// base[w]: SNPs of the first w words with their bit set; base[n_words]: of all.
__global__ void __launch_bounds__(1024)
    class_base_kernel(const uint32_t *__restrict__ words, int64_t n_words, uint32_t *__restrict__ base) {
  __shared__ uint32_t part[32];
  __shared__ uint32_t carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0u;
  for (int64_t w0 = 0; w0 < n_words; w0 += 8 * 1024) {
    // eight words a thread
    const int64_t w = w0 + 8 * threadIdx.x;
    uint32_t c[8], sum = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      c[i] = w + i < n_words ? (uint32_t)__popc(words[w + i]) : 0u;
      sum += c[i];
    }
    uint32_t pre = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, pre, o);
      if (lane >= o) pre += y;
    }
    __syncthreads();  // (part and carry of the lap before are read)
    if (lane == 31) part[warp] = pre;
    __syncthreads();
    uint32_t before = carry;
    for (int i = 0; i < warp; ++i) before += part[i];
    uint32_t at = before + pre - sum;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (w + i < n_words) base[w + i] = at;
      at += c[i];
    }
    __syncthreads();
    if (threadIdx.x == 1023) carry = at;
  }
  __syncthreads();
  if (threadIdx.x == 0) base[n_words] = carry;
}

__global__ void class_list_kernel(const uint32_t *__restrict__ words, const uint32_t *__restrict__ base,
                                  int64_t n_words, int64_t snp_begin, int64_t n_snps,
                                  int64_t *__restrict__ list) {
  const int64_t two = n_snps - (int64_t)base[n_words];  // SNPs of the first part
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n_snps;
       j += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t word = words[j >> 5], bit = 1u << (j & 31);
    const int64_t ones = (int64_t)base[j >> 5] + __popc(word & (bit - 1u));  // set ones before j
    list[(word & bit) ? two + ones : j - ones] = snp_begin + j;
  }
}

}  // namespace

// list, words, prefix sums
size_t class_order_bytes(int64_t n_snps) {
  const int64_t n_words = (n_snps + 31) / 32;
  return (size_t)n_snps * 8 + (size_t)(2 * n_words + 1) * 4;
}
cudaError_t launch_class_order(const int8_t *geno, int64_t ldg, int N, int64_t snp_begin,
                               int64_t n_snps, void *scratch, cudaStream_t s) {
  const int64_t n_words = (n_snps + 31) / 32;
  int64_t *list = reinterpret_cast<int64_t *>(scratch);
  uint32_t *words = reinterpret_cast<uint32_t *>(list + n_snps), *base = words + n_words;
  class_bits_kernel<<<(unsigned)((n_words + 7) / 8), 256, 0, s>>>(geno + snp_begin * ldg, ldg, N, n_snps,
                                                                  words, n_words);
  class_base_kernel<<<1, 1024, 0, s>>>(words, n_words, base);
  class_list_kernel<<<(unsigned)std::min<int64_t>((n_snps + 255) / 256, 152 * 8), 256, 0, s>>>(
      words, base, n_words, snp_begin, n_snps, list);
  return cudaGetLastError();
}

}  // namespace krux
