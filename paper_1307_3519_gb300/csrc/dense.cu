// dense.cu -- the FP64 pass of a dense output: H (Eq. 2 with the tie factor) and the
// chi-square p of every pair, from the rank sums the plain scan form wrote (section
// "P-value calculation").
//
// FP64 issues at a 64th of the FP32 rate on this part, so the pass is bound by its FP64
// operations, counted per warp: the statistic's numerator is formed in integers
// (DenseCol), exp and erfc come from tables and short polynomials (table reduction of the
// exponential as in Tang, "Table-driven implementation of the exponential function", 1989;
// erfc(sqrt x) as exp(-x) erfcx(sqrt x) with piecewise polynomials of erfcx), comparisons
// and conversions are done on the bits, and a block takes its columns by df class, so that
// a warp runs one of the two tails: about 13 FP64 operations for df 2 and 31 for df 1.
// With three FP64 divisions and the library's exp and erfc in the scan's epilogue, 1,000 x
// 20,003 x 102 took 4.35 ms; a pass of 16 and 34 operations with both classes in every
// warp 1.04 ms, this one 0.66, after 0.11 ms for the rank sums.
#include <cmath>
#include <atomic>

#include "common.cuh"
#include "fp64_tables.cuh"

namespace krux {

namespace {
constexpr int kExpBits = 12, kExpTab = 1 << kExpBits;  // 2^(-j / 4096), high and low parts
constexpr int kErfInts = 512, kErfDeg = 6;   // erfcx on [0, 6.4), intervals of 1/80
constexpr int kDenseThreads = 512;           // and columns of a block's window
__device__ double c_exp[2 * kExpTab];
__device__ double c_erfcx[kErfInts * (kErfDeg + 1)];

struct DenseTables {
  double e[2 * kExpTab];
  double f[kErfInts * (kErfDeg + 1)];
};

// A normal positive double as FP32 (truncated), and back (exact), on the bits: FP64's
// conversions issue as slowly as its arithmetic.
__device__ __forceinline__ float f32_of(double x) {
  return __uint_as_float((((uint32_t)__double2hiint(x) - 0x38000000u) << 3) |
                         ((uint32_t)__double2loint(x) >> 29));
}
__device__ __forceinline__ double f64_of(float x) {
  const uint32_t b = __float_as_uint(x);
  return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// erfc(sqrt x) = exp(-x) erfcx(sqrt x), x > 0.
__device__ __forceinline__ double erfc_sqrt(double x, const double *etab, const double *ftab) {
  const int hi = __double2hiint(x);
  if (hi >= 0x40440000 || hi < 0x39c00000) return erfc(sqrt(x));  // x >= 40, x < 2^-99
  // sqrt by two Newton steps from the FP32 reciprocal root
  const float yf = rsqrtf(f32_of(x));
  const double y = f64_of(yf), hy = f64_of(0.5f * yf);
  double z = x * y;
  z = fma(fma(-z, z, x), hy, z);
  z = fma(fma(-z, z, x), hy, z);
  const int i = (int)(f32_of(z) * 80.0f);  // (the next interval's edge may fall in this one)
  const double w = fma(f64_of((float)(2 * i + 1)), -0.00625, z);
  const double *c = ftab + i * (kErfDeg + 1);
  double f = c[kErfDeg];
#pragma unroll
  for (int j = kErfDeg - 1; j >= 0; --j) f = fma(f, w, c[j]);
  return exp_neg<kExpBits>(x, etab) * f;
}

// p within some 1e-12 of P_c: as the other forms decide it (they may differ in the last
// places, and P_c may be a p of the data).
__device__ __noinline__ double p_at_threshold(int d0, int d1, int n0, int n1, int n2, int df, double cf) {
  return kw_p64(kw_H64(d0, d1, n0, n1, n2, cf), df);
}

// One thread per packed slot: its column's entry.
__global__ void dense_cols_kernel(const GroupDesc *__restrict__ groups, int g0, int64_t snp0,
                                  DenseCol *__restrict__ col) {
  const GroupDesc &g = groups[g0 + blockIdx.y];
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= (int64_t)g.nchunks * kChunkSnps) return;
  const ChunkMeta &m = g.meta[j / kChunkSnps];
  const int jj = (int)(j % kChunkSnps);
  if (m.snp[jj] < 0) return;
  DenseCol c;
  c.n0 = m.n[0][jj];
  c.n1 = m.n[1][jj];
  c.n2 = m.n[2][jj];
  c.df = m.df[jj];
  c.pad_ = 0;
  const uint32_t p0 = max((int)c.n0, 1), p1 = max((int)c.n1, 1), p2 = max((int)c.n2, 1);
  c.a = p1 * p2;
  c.b = p0 * p2;
  c.c = p0 * p1;
  const double den = (double)c.a * (double)p0;
  c.rcp = 1.0 / den;
  c.rcp_lo = fma(-den, c.rcp, 1.0) * c.rcp;
  c.group = g0 + (int)blockIdx.y;
  c.snp = m.snp[jj];
  col[m.snp[jj] - snp0] = c;
}

// Work items: a window of kDenseThreads columns and a run of traits each, dealt to the
// blocks in turn; one thread per column, df-1 columns last.
__global__ void __launch_bounds__(kDenseThreads, 2)
dense_finish_kernel(const DenseCol *__restrict__ col, const double *const *__restrict__ cfac_by_group,
                    int T, int per_item, int64_t windows, int64_t n_items, int64_t cols, int64_t ld,
                    double *__restrict__ H, double *__restrict__ P, double pthresh,
                    krux_hit *__restrict__ hits, HitAux *__restrict__ aux, int64_t capacity,
                    unsigned long long *counter) {
  extern __shared__ __align__(16) double tables[];
  __shared__ int ones[kDenseThreads / 32];
  __shared__ uint16_t order[kDenseThreads];
  double *etab = tables, *ftab = tables + 2 * kExpTab;
  for (int i = threadIdx.x; i < 2 * kExpTab; i += blockDim.x) etab[i] = c_exp[i];
  for (int i = threadIdx.x; i < kErfInts * (kErfDeg + 1); i += blockDim.x) ftab[i] = c_erfcx[i];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long pbits = __double_as_longlong(pthresh);  // (positive doubles order as integers)
  for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int64_t j0 = item % windows * kDenseThreads;
    const bool one = j0 + threadIdx.x < cols && col[j0 + threadIdx.x].df == 1;
    const uint32_t bal1 = __ballot_sync(0xffffffffu, one);
    __syncthreads();  // (tables written; the order of the item before read)
    if (lane == 0) ones[warp] = __popc(bal1);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < kDenseThreads / 32; ++w) {
      before += w < warp ? ones[w] : 0;
      total += ones[w];
    }
    before += __popc(bal1 & ((1u << lane) - 1u));
    order[one ? kDenseThreads - total + before : (int)threadIdx.x - before] = (uint16_t)threadIdx.x;
    __syncthreads();
    const int64_t j = j0 + order[threadIdx.x];
    const bool live = j < cols;
    DenseCol c{};
    if (live) c = col[j];
    const double *cfac = cfac_by_group[c.group];
    const int t0 = (int)(item / windows) * per_item, t1 = min(t0 + per_item, T);
    for (int t = t0; t < t1; ++t) {
      const int64_t o = (int64_t)t * ld + j;
      int2 d = make_int2(0, 0);
      if (live) d = *reinterpret_cast<const int2 *>(H + o);
      const double cf = cfac[t];
      double h = 0.0, p = 1.0;
      if (c.df > 0 && __double_as_longlong(cf) > 0) {
        const unsigned long long d0 = (unsigned long long)((long long)d.x * d.x);
        const unsigned long long d1 = (unsigned long long)((long long)d.y * d.y);
        const int e = d.x + d.y;
        const unsigned long long d2 = (unsigned long long)((long long)e * e);
        const unsigned long long num = d0 * c.a + d1 * c.b + d2 * c.c;  // < 2^50
        const double nd = __longlong_as_double((long long)(num | 0x4330000000000000ull)) - 4503599627370496.0;
        h = cf * fma(nd, c.rcp, nd * c.rcp_lo);  // (the quotient to its last place)
        const int hh = __double2hiint(h);
        const bool some = hh >= 0x00200000;  // else 0
        const double x = some ? __hiloint2double(hh - 0x00100000, __double2loint(h)) : 0.0;  // h / 2
        if (c.df == 1) p = some ? erfc_sqrt(x, etab, ftab) : 1.0;
        else p = hh < 0x4095e000 ? exp_neg<kExpBits>(x, etab) : exp(-x);  // (h < 1400)
        if ((unsigned long long)(__double_as_longlong(p) - pbits + 4096) < 8192ull)
          p = p_at_threshold(d.x, d.y, c.n0, c.n1, c.n2, c.df, cf);
      }
      if (live) {
        H[o] = h;
        P[o] = p;
      }
      const bool hit = live && __double_as_longlong(p) < pbits;
      const uint32_t bal = __ballot_sync(0xffffffffu, hit);
      if (bal == 0u) continue;
      unsigned long long base = 0;
      if (lane == 0) base = atomicAdd(counter, (unsigned long long)__popc(bal));
      base = __shfl_sync(0xffffffffu, base, 0) + (unsigned int)__popc(bal & ((1u << lane) - 1u));
      if (hit && base < (unsigned long long)capacity) {
        krux_hit r;
        r.trait = (uint32_t)t;
        r.snp = (uint32_t)c.snp;
        r.d0 = d.x;
        r.d1 = d.y;
        st_hit(hits + base, r);
        HitAux a;
        a.n0 = c.n0;
        a.n1 = c.n1;
        a.n2 = c.n2;
        a.group = (uint16_t)c.group;
        st_aux(aux + base, a);
      }
    }
  }
}

// erfcx on the interval [mid - h, mid + h] as a polynomial in z - mid: interpolation at
// Chebyshev nodes (of one degree more than is kept, in extended precision), turned into
// powers.
void erfcx_poly(long double mid, long double h, double *out) {
  constexpr int n = kErfDeg + 4;
  const long double pi = 3.14159265358979323846264338327950288L;
  static const struct Cosines {
    long double c[n][n];  // of i (j + 1/2) pi / n
    explicit Cosines(long double pi) {
      for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) c[i][j] = std::cos(pi * i * (j + 0.5L) / n);
    }
  } cosines(pi);
  long double f[n], cheb[n];
  for (int j = 0; j < n; ++j) {
    const long double z = mid + h * cosines.c[1][j];
    f[j] = std::exp(z * z) * std::erfc(z);
  }
  for (int i = 0; i < n; ++i) {
    long double c = 0.0L;
    for (int j = 0; j < n; ++j) c += f[j] * cosines.c[i][j];
    cheb[i] = c * (i ? 2.0L : 1.0L) / n;
  }
  // powers of the Chebyshev polynomials up to the kept degree
  long double T0[n] = {1.0L}, T1[n] = {0.0L, 1.0L}, p[n] = {};
  for (int i = 0; i <= kErfDeg; ++i) {
    for (int k = 0; k < n; ++k) p[k] += cheb[i] * T0[k];
    long double T2[n];
    for (int k = 0; k < n; ++k) T2[k] = (k ? 2.0L * T1[k - 1] : 0.0L) - T0[k];
    for (int k = 0; k < n; ++k) {
      T0[k] = T1[k];
      T1[k] = T2[k];
    }
  }
  long double s = 1.0L;
  for (int k = 0; k <= kErfDeg; ++k, s /= h) out[k] = (double)(p[k] * s);
}

const DenseTables &dense_tables() {
  static const DenseTables t = [] {
    DenseTables x;
    fill_exp_table<kExpBits>(x.e);
    for (int i = 0; i < kErfInts; ++i) erfcx_poly((2 * i + 1) * 0.00625L, 0.006275L, x.f + i * (kErfDeg + 1));
    return x;
  }();
  return t;
}

}  // namespace

cudaError_t dense_prepare(cudaStream_t s) {
  static std::atomic<unsigned long long> uploaded{0};
  return once_per_device(uploaded, s, [](cudaStream_t s) {
    const DenseTables &t = dense_tables();
    cudaError_t e = cudaMemcpyToSymbolAsync(c_exp, t.e, sizeof t.e, 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaMemcpyToSymbolAsync(c_erfcx, t.f, sizeof t.f, 0, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(dense_finish_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(DenseTables));
    return e;
  });
}

cudaError_t launch_dense_finish(const GroupDesc *groups, int n_groups, int64_t max_chunks,
                                const double *const *cfac_by_group, int T, int64_t cols,
                                int64_t snp0, int64_t ld, double *H, double *p, DenseCol *col,
                                double pthresh, krux_hit *hits, HitAux *aux, int64_t capacity,
                                unsigned long long *counter, int sm_count, cudaStream_t s) {
  if (n_groups <= 0 || cols <= 0 || T <= 0 || max_chunks <= 0) return cudaSuccess;
  // (a SNP left out of the scan, in a graph replay, keeps an empty column)
  cudaError_t e = cudaMemsetAsync(col, 0, (size_t)cols * sizeof(DenseCol), s);
  if (e != cudaSuccess) return e;
  for (int g0 = 0; g0 < n_groups; g0 += 65535) {
    const dim3 grid((unsigned)((max_chunks * kChunkSnps + 255) / 256),
                    (unsigned)(n_groups - g0 < 65535 ? n_groups - g0 : 65535));
    dense_cols_kernel<<<grid, 256, 0, s>>>(groups, g0, snp0, col);
  }
  // two blocks per SM; runs of traits such that each has eight items, at least 8 traits each
  const int64_t windows = (cols + kDenseThreads - 1) / kDenseThreads;
  int64_t runs = (int64_t)sm_count * 16 / windows + 1;
  if (runs > (T + 7) / 8) runs = (T + 7) / 8;
  const int per = (int)((T + runs - 1) / runs);
  const int64_t items = windows * ((T + per - 1) / per);
  const int grid = (int)(items < 2 * sm_count ? items : 2 * sm_count);
  dense_finish_kernel<<<grid, kDenseThreads, sizeof(DenseTables), s>>>(
      col, cfac_by_group, T, per, windows, items, cols, ld, H, p, pthresh, hits, aux, capacity, counter);
  return cudaGetLastError();
}

}  // namespace krux
