// param.cu -- parametric comparison statistics on the same tiles (the paper
// compares kruX with matrix-eQTL's linear and ANOVA models on the same data).
//
// The contraction is the one of the Kruskal-Wallis scan with the centred ranks
// replaced by standardised values z = (x - mean) / sd (FP16, so the fused test is
// approximate): with S_i = sum of z over genotype group i,
//   ANOVA:  SS_between = sum_i S_i^2 / N_i (sum_i S_i = 0), compared with the
//           per-df bound tau_df = (K-1) F_c df / (K - 1 - df + F_c df);
//   linear: S_zg = S_1 + 2 S_2 = -(2 S_0 + S_1), compared with the bound
//           S_zg^2 >= r_c^2 S_gg (K - 1), r_c^2 = t_c^2 / (K - 2 + t_c^2).
// Every pair at or above the lower edge of a wide band is kept as a provisional
// hit; this file's finalisation recomputes each one from the caller's FP32 values
// (exact group sums, FP64 after them) and keeps those with p < P_c.
#include <atomic>

#include "common.cuh"
#include "fp64_tables.cuh"
#include "param_tails.cuh"

namespace krux {

namespace {

// The continued fraction of I_x(a, 1/2) on [0, kTabMax]: a polynomial of degree kTabDeg
// in t = (x - middle) / half width on each of kTabInts equal intervals, from the
// Chebyshev interpolation there (the nearest singularity, x = 1, lies at least eleven
// interval widths away: the terms left out are below 1e-16).  One warp per interval; a =
// (N - 2) / 2 is the only one a call needs (two genotype groups, or the regression).
constexpr int kTabInts = 128, kTabDeg = 9;
constexpr double kTabMax = 0.92;
__global__ void cf_table_kernel(double a, double *__restrict__ table) {
  const int i = threadIdx.x & 31, interval = blockIdx.x;
  const double h = 0.5 * kTabMax / kTabInts, mid = (2 * interval + 1) * h;
  constexpr int n = kTabDeg + 1;
  const double f = i < n ? ibeta_cf(a, 0.5, mid + h * cospi((i + 0.5) / n)) : 0.0;
  double c = 0.0;  // lane i: the coefficient of T_i
  for (int j = 0; j < n; ++j) c += __shfl_sync(0xffffffffu, f, j) * cospi(i * (j + 0.5) / n);
  c *= (i ? 2.0 : 1.0) / n;
  // powers of t: lane i gathers row i of the Chebyshev polynomials' coefficients
  double t0 = i == 0 ? 1.0 : 0.0, t1 = i == 1 ? 1.0 : 0.0, p = 0.0;
  for (int k = 0; k < n; ++k) {
    p += __shfl_sync(0xffffffffu, c, k) * t0;
    const double up = __shfl_up_sync(0xffffffffu, t1, 1);
    const double t2 = (i ? 2.0 * up : 0.0) - t0;
    t0 = t1;
    t1 = t2;
  }
  if (i < n) table[interval * n + i] = p;
}

// The polynomial at x, 0 < x < kTabMax.
__device__ __forceinline__ double cf_of(double x, const double *__restrict__ table) {
  const int i = min((int)((float)x * (float)(kTabInts / kTabMax)), kTabInts - 1);
  const double t = fma(x, 2.0 * kTabInts / kTabMax, -(double)(2 * i + 1));
  const double *c = table + i * (kTabDeg + 1);
  double f = c[kTabDeg];
#pragma unroll
  for (int k = kTabDeg - 1; k >= 0; --k) f = fma(f, t, c[k]);
  return f;
}

// I_x(a, 1/2) with front = 1 / (a B(a, 1/2)) and the table of its continued fraction.
__device__ __forceinline__ double half_beta(double x, double a, double front,
                                            const double *__restrict__ table) {
  if (!(x > 0.0)) return 0.0;
  if (x >= kTabMax) return ibeta(a, 0.5, x);
  return front * exp(a * log(x)) * sqrt(1.0 - x) * cf_of(x, table);
}

// What the finalisation holds in shared memory.
constexpr int kExpBitsP = 7;
struct ParamTables {
  double e[2 << kExpBitsP];        // exp_neg
  double l[3 * kLogTab];           // log_ge1
};
__device__ ParamTables c_param;
struct ParamShared {
  ParamTables t;
  double cf[kTabInts * (kTabDeg + 1)];
  double2 rcp[kMaxN + 1];          // 1 / i in two parts
};

// Place of an FP32 value in fixed point whose unit is 2^-29 of the last place of a
// value with exponent field emax: below 2^53, exact unless the value is 2^29 times
// smaller than the largest (then rounded to nearest).
__device__ __forceinline__ long long to_fixed(float x, int emax) {
  const uint32_t b = __float_as_uint(x);
  int e = (int)((b >> 23) & 255u);
  const long long m = (long long)((b & 0x7fffffu) | (e ? 0x800000u : 0u));
  if (e == 0) e = 1;
  const int sh = 29 - (emax - e);
  const long long f = sh >= 0 ? m << sh : (sh > -25 ? (m + (1ll << (-sh - 1))) >> -sh : 0ll);
  return (b >> 31) ? -f : f;
}

// One warp per trait: the row centred in 64-bit fixed point (below 2^54, so that 512
// values sum without overflow) with the FP64 sum of its squares for the finalisation,
// the standardised FP16 row of A (0 in the padding columns, in both layouts), and the
// constants the scan reads (bound 1, no NaN).  A NaN sets kDevBadCode.  The mean comes
// from the exact integer sum; only the squares need FP64, two operations a value (with
// the mean, deviations and scale in FP64, 20,000 x 102: some 200 us against 38).
__global__ void standardize_kernel(const float *__restrict__ expr, int T, int N, int64_t ld, int Np,
                                   __half *__restrict__ A, __half *__restrict__ At,
                                   long long *__restrict__ fixed, double *__restrict__ squares,
                                   float *__restrict__ tau, double *__restrict__ cfac,
                                   uint16_t *__restrict__ nan_cnt, unsigned int *status) {
  const int warp = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (warp >= T) return;
  const float *x = expr + (int64_t)warp * ld;
  int emax = 1;
  bool nan = false;
  for (int k = lane; k < N; k += 32) {
    const float v = x[k];
    nan |= v != v;
    emax = max(emax, (int)((__float_as_uint(v) >> 23) & 255u));
  }
  emax = (int)__reduce_max_sync(0xffffffffu, (unsigned)emax);
  const bool finite = emax < 255;
  long long sum = 0;
  for (int k = lane; k < N && finite; k += 32) sum += to_fixed(x[k], emax);
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const long long mid = sum / N;
  double q = 0.0;
  for (int k = lane; k < N; k += 32) {
    const long long f = finite ? to_fixed(x[k], emax) - mid : 0ll;
    fixed[(int64_t)warp * N + k] = f;
    q = fma((double)f, (double)f, q);
  }
  for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
  const float sd = sqrtf((float)q / (float)(N - 1));
  const float inv = sd > 0.f ? 1.f / sd : 0.f;
  for (int k = lane; k < Np; k += 32) {
    const float z = k < N && finite ? (float)(to_fixed(x[k], emax) - mid) * inv : 0.f;
    A[(int64_t)warp * Np + k] = __float2half_rn(z);
    At[tiled_index(warp, k, Np)] = __float2half_rn(z);
  }
  nan = __any_sync(0xffffffffu, nan);
  if (lane == 0) {
    if (nan) atomicOr(status, kDevBadCode);
    squares[warp] = q;
    // a constant row can never be significant: bound +inf
    tau[warp] = sd > 0.f ? 1.0f : __int_as_float(0x7f800000);
    cfac[warp] = 1.0;
    nan_cnt[warp] = 0;
  }
}

// Four genotype bytes at p (aligned); only bytes in [lo, hi) may be read.
__device__ __forceinline__ uint32_t geno_word(const int8_t *p, const int8_t *lo, const int8_t *hi) {
  if (p >= lo && p + 4 <= hi) return *reinterpret_cast<const uint32_t *>(p);
  uint32_t w = 0u;
  for (int b = 0; b < 4; ++b)
    if (p + b >= lo && p + b < hi) w |= (uint32_t)(uint8_t)p[b] << (8 * b);
  return w;
}

// FP64 statistic and p of every provisional hit, and the hits with p < P_c to the
// caller's lists (d0 = d1 = 0: parametric hits carry no rank sums).  Complete data:
// the total and the squares are the trait's, the group sizes come with the hit, so a
// hit needs the sums of two groups alone, taken exactly in 64-bit integers.  One
// thread per hit: four genotypes a word, the trait's row shared by the threads of one
// event.  FP64 issues at a 64th of the integer rate on this part, so what is left of it
// counts.  With rho = SS_between / SS_within and u = 1 + rho, both tails of the analysis of
// variance are powers of 1 / u: u^-((N - 3) / 2) for three groups (closed form), front u^-((N - 2)
// / 2) sqrt(rho / u) cf(1 / u) for two, so a warp of both runs one logarithm and one
// exponential, from tables; divisions by group sizes are products with reciprocals in two
// parts.  With FP64 additions, squares per hit and the continued fraction evaluated per
// hit, 1.95 M hits of 102 samples took 2.73 ms; with the library's tails, one for each
// number of groups, 0.60; now 0.35.
__global__ void __launch_bounds__(256, 4)
finalize_param_kernel(const krux_hit *__restrict__ hits, const HitAux *__restrict__ aux,
                      const unsigned long long *__restrict__ count, int64_t capacity,
                      const long long *__restrict__ fixed, const double *__restrict__ squares,
                      const int8_t *__restrict__ geno, int64_t ldg, const int8_t *__restrict__ lo,
                      const int8_t *__restrict__ hi, int N, int model, double a_half, double front,
                      const double *__restrict__ table, double pthresh, krux_hit *__restrict__ out,
                      double *__restrict__ out_stat, double *__restrict__ out_p,
                      int64_t out_capacity, unsigned long long *__restrict__ n_out) {
  extern __shared__ __align__(16) char shared[];
  ParamShared &S = *reinterpret_cast<ParamShared *>(shared);
  for (int i = threadIdx.x; i < (int)(sizeof(ParamTables) / 8); i += blockDim.x)
    reinterpret_cast<double *>(&S.t)[i] = reinterpret_cast<const double *>(&c_param)[i];
  for (int i = threadIdx.x; i < kTabInts * (kTabDeg + 1); i += blockDim.x) S.cf[i] = table[i];
  for (int i = threadIdx.x; i <= N; i += blockDim.x) {
    const double r = i ? 1.0 / (double)i : 0.0;
    S.rcp[i] = make_double2(r, i ? fma(-(double)i, r, 1.0) * r : 0.0);
  }
  __syncthreads();
  const auto over = [&](double x, int n) {  // x / n, n = 0 gives 0
    const double2 r = S.rcp[n];
    return fma(x, r.x, x * r.y);
  };
  const unsigned long long c = *count;
  const int64_t n = c < (unsigned long long)capacity ? (int64_t)c : capacity;
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) - lane; i0 < n;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i0 + lane;
    double value = 0.0, p = 1.0;
    krux_hit r{};
    if (i < n) {
      r = ld_hit(hits + i);
      const HitAux x = ld_aux(aux + i);
      const long long *f = fixed + (int64_t)r.trait * N;
      const int8_t *g = geno + (int64_t)r.snp * ldg;
      const int pad = (int)((uintptr_t)g & 3u);
      const int8_t *gp = g - pad;
      long long S0 = 0, S1 = 0, St = 0;
      uint32_t cur = geno_word(gp, lo, hi);
      for (int k = 0; k < N; k += 4) {
        gp += 4;
        const uint32_t next = k + 4 - pad < N ? geno_word(gp, lo, hi) : 0u;
        const uint32_t w = __funnelshift_r(cur, next, 8 * pad);
        cur = next;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (k + t < N) {
            const long long v = __ldg(f + k + t);
            const uint32_t code = (w >> (8 * t)) & 0xffu;
            St += v;
            if (code == 0u) S0 += v;
            if (code == 1u) S1 += v;
          }
        }
      }
      const double s[3] = {(double)S0, (double)S1, (double)(St - S0 - S1)};
      const double st = (double)St, q = squares[r.trait], K = (double)N;
      const int cnt[3] = {x.n0, x.n1, x.n2};
      if (model == 0) {  // one-way ANOVA
        int groups = 0;
        double sq = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          if (cnt[j] == 0) continue;
          ++groups;
          sq += over(s[j] * s[j], cnt[j]);
        }
        const double ssb = sq - over(st * st, N);
        const double ssw = fmax(q - sq, 0.0);
        if (groups >= 2 && N > groups) {
          if (ssw > 0.0) {
            const double rho = ssb / ssw;
            const int d2 = N - groups;
            value = rho * (groups == 3 ? 0.5 * d2 : (double)d2);
            if (!(value > 0.0)) {
              p = 1.0;
            } else if (rho < 1e-3 || rho > 1e30) {  // p near 1, or far below what FP64 holds
              p = groups == 3 ? f_tail(value, 2.0, d2) : half_beta(d2 / (d2 + value), a_half, front, S.cf);
            } else {
              const double u = 1.0 + rho;
              // log(1 + rho) in two parts (what u's rounding lost, to first order), and its
              // multiple as well: the exponent is large, p keeps its last places (from its
              // statistic to 2e-15, without this and with the library's functions 8e-15)
              double low;
              const double lu = log_ge1(u, S.t.l, low), a = 0.5 * d2, x = a * lu;
              low = fma(rho - (u - 1.0), (double)(1.f / (float)u), low);
              low = fma(a, low, fma(a, lu, -x));
              p = x < 700.0 ? exp_neg<kExpBitsP>(x, S.t.e) : exp(-x);
              p = fma(-p, low, p);
              if (groups == 2) {
                const double v = 1.0 / u;
                p = v < kTabMax ? p * (front * sqrt(rho * v) * cf_of(v, S.cf)) : ibeta(a_half, 0.5, v);
              }
            }
          } else if (ssb > 0.0) {
            value = __longlong_as_double(0x7ff0000000000000ll);
            p = 0.0;
          }
        }
      } else {  // dosage regression
        const double gs = (double)cnt[1] + 2.0 * cnt[2];
        const double gm = gs / K;
        const double sgg = (double)cnt[1] + 4.0 * cnt[2] - gs * gm;
        const double sxg = s[1] + 2.0 * s[2] - gm * st;
        const double sxx = q - st * st / K;
        if (N >= 3 && sgg > 0.0 && sxx > 0.0) {
          const double rr = sxg / sqrt(sgg * sxx);
          if (fabs(rr) < 1.0) {
            value = rr * sqrt((K - 2) / (1.0 - rr * rr));
            const double t2 = value * value;
            p = t2 > 0.0 ? half_beta((K - 2) / (K - 2 + t2), a_half, front, S.cf) : 1.0;
          } else {
            value = rr > 0 ? __longlong_as_double(0x7ff0000000000000ll)
                           : -__longlong_as_double(0x7ff0000000000000ll);
            p = 0.0;
          }
        }
      }
    }
    const bool keep = i < n && p < pthresh;
    const uint32_t bal = __ballot_sync(0xffffffffu, keep);
    if (bal == 0u) continue;
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(n_out, (unsigned long long)__popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0) + (unsigned int)__popc(bal & ((1u << lane) - 1u));
    if (keep && base < (unsigned long long)out_capacity) {
      r.d0 = 0;
      r.d1 = 0;
      st_hit(out + base, r);
      out_stat[base] = value;
      out_p[base] = p;
    }
  }
}

}  // namespace

size_t param_table_bytes() { return kTabInts * (kTabDeg + 1) * sizeof(double); }

cudaError_t launch_standardize(const float *expr, int T, int N, int64_t ld, int Np, __half *A,
                               __half *At, long long *fixed, double *squares, float *tau,
                               double *cfac, uint16_t *nan_cnt, unsigned int *status,
                               cudaStream_t s) {
  if (T <= 0) return cudaSuccess;
  const int warps_per_block = 8;
  const int grid = (T + warps_per_block - 1) / warps_per_block;
  standardize_kernel<<<grid, warps_per_block * 32, 0, s>>>(expr, T, N, ld, Np, A, At, fixed, squares,
                                                           tau, cfac, nan_cnt, status);
  return cudaGetLastError();
}

// The finalisation's table of a call: some 60 us of serial FP64 chains, on a stream of its own
// beside the scan.
cudaError_t launch_param_table(int N, double *table, cudaStream_t s) {
  cf_table_kernel<<<kTabInts, 32, 0, s>>>(0.5 * (N - 2), table);
  return cudaGetLastError();
}

cudaError_t param_prepare(cudaStream_t s) {
  static std::atomic<unsigned long long> uploaded{0};
  return once_per_device(uploaded, s, [](cudaStream_t s) {
    static const ParamTables t = [] {
      ParamTables x;
      fill_exp_table<kExpBitsP>(x.e);
      fill_log_table(x.l);
      return x;
    }();
    cudaError_t e = cudaMemcpyToSymbolAsync(c_param, &t, sizeof t, 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(finalize_param_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(ParamShared));
    return e;
  });
}

cudaError_t launch_finalize_param(const krux_hit *hits, const HitAux *aux,
                                  const unsigned long long *count, int64_t capacity,
                                  const long long *fixed, const double *squares,
                                  const int8_t *geno, int64_t ldg, const int8_t *lo,
                                  const int8_t *hi, int N, int model, const double *table,
                                  double pthresh, krux_hit *out, double *out_stat, double *out_p,
                                  int64_t out_capacity, unsigned long long *n_out, int sm_count,
                                  cudaStream_t s) {
  if (capacity <= 0) return cudaSuccess;
  int grid = sm_count * 4;
  const int64_t need = (capacity + 255) / 256;
  if (need < grid) grid = (int)need;
  // 1 / (a B(a, 1/2)), a = (N - 2) / 2, by the recurrence of the gamma function from
  // a = 1/2 (1 / (a B) = 2 / pi) or a = 1 (1/2)
  const int nu = N - 2;
  long double front = nu & 1 ? 2.0L / 3.14159265358979323846264338327950288L : 0.5L;
  // B(a + 1, 1/2) = B(a, 1/2) a / (a + 1/2): 1 / (a B) gains (a + 1/2) / (a + 1)
  for (long double a = nu & 1 ? 0.5L : 1.0L; a < 0.5L * nu - 0.25L; a += 1.0L) front *= (a + 0.5L) / (a + 1.0L);
  finalize_param_kernel<<<grid, 256, sizeof(ParamShared), s>>>(hits, aux, count, capacity, fixed, squares, geno, ldg, lo,
                                             hi, N, model, 0.5 * nu, (double)front, table, pthresh,
                                             out, out_stat, out_p, out_capacity, n_out);
  return cudaGetLastError();
}

// Host-side thresholds of the fused test.
double param_f_crit(double pthresh, double d1, double d2) {
  double lo = 0.0, hi = 1.0;
  while (f_tail(hi, d1, d2) > pthresh && hi < 1e300) hi *= 2.0;
  for (int i = 0; i < 200; ++i) {
    const double mid = 0.5 * (lo + hi);
    if (f_tail(mid, d1, d2) > pthresh) lo = mid; else hi = mid;
  }
  return 0.5 * (lo + hi);
}

double param_t_crit(double pthresh, double nu) {
  double lo = 0.0, hi = 1.0;
  while (t_tail2(hi, nu) > pthresh && hi < 1e300) hi *= 2.0;
  for (int i = 0; i < 200; ++i) {
    const double mid = 0.5 * (lo + hi);
    if (t_tail2(mid, nu) > pthresh) lo = mid; else hi = mid;
  }
  return 0.5 * (lo + hi);
}

}  // namespace krux

// Test hook: the tails above evaluated on the host (no GPU needed).
extern "C" double krux_debug_tail(int kind, double x, double d1, double d2) {
  if (kind == 0) return krux::f_tail(x, d1, d2);
  if (kind == 1) return krux::t_tail2(x, d1);
  return krux::ibeta(d1, d2, x);
}
