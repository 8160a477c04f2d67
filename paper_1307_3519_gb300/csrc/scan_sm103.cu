// scan_sm103.cu -- fused Kruskal-Wallis scan for sm_103a (tcgen05 + TMA + TMEM).
//
// For a tile of 128 traits and a chunk of 64 SNPs the tensor cores contract the
// centred rank matrix A (traits x samples, FP16 integers) with the packed genotype rows
// of the chunk (Eq. 4: S_i = R I_i^T, here in centred form D_i = 2 S_i - N_i (K+1)),
// accumulating exactly in FP32 in TMEM.  The epilogue never writes the rank sums to
// memory (but for a dense output): it compares Eq. 2 in centred form, H = 3/(K(K+1)C)
// sum_i D_i^2/N_i with D_2 = -D_0 - D_1 and the tie factor C (section "Handling tied
// data"), with the chi-square threshold of the SNP's degrees of freedom (section
// "P-value calculation and empirical FDR correction"); pairs within a relative margin
// of the threshold are decided in FP64.
//
// Plain forms (kFormScan*; 640 threads, one CTA per SM, persistent over work items taken
// from a common counter), on weighted genotype rows (ChunkMeta) in the tensor cores' own
// tile layout (tiled_index):
//   warps 0-15 : epilogue; warp 4k + q reads TMEM lanes 32q.. (traits) and 32 SNPs of a
//                chunk of each accumulator pair, and tests P^2 + Q^2 against the bound
//   warp 16    : producer (rank tiles stream through nA stages by bulk copies; a B tile
//                of nc chunks stays resident while all trait tiles pass)
//   warp 17    : TMEM allocator and tcgen05.mma issuer (one thread; with kFormScanPair
//                over a cluster of two CTAs, cta_group::2)
//   warps 18-19: event warps (candidates to exact sums, decisions and hit records)
// General forms (kFormMulti, kFormPerm, kFormNan; 576 threads): 0/1 indicator rows by TMA
// boxes, warps 0-15 test and append their hits themselves, 16 SNPs each.
// Every mbarrier wait is bounded: on timeout the kernel raises an error bit,
// drains its own asynchronous copies and MMAs, frees TMEM and returns.
#include <atomic>
#include <type_traits>

#include "common.cuh"

namespace krux {

namespace {

// tcgen05 instruction descriptor, kind::f16: D = F32, A = B = F16, both K-major,
// N = 128 (bits 17-22 hold N >> 3), M = 128 (bits 24-28 hold M >> 4).
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
// Same with N = 256: one MMA over a pair of chunks whose B rows are interleaved
// per K atom (256 rows of 32 B), writing two adjacent 128-column accumulators.
constexpr uint32_t kIdesc256 = (1u << 4) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
// Over a pair of CTAs (cta_group::2): M = 256 traits, 128 in each CTA, N = 256, the
// rows of one chunk in each CTA.
constexpr uint32_t kIdescPair = (1u << 4) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
// Two K-major shared-memory layouts: 128-byte swizzle with 64-element K atoms
// (K padded to a multiple of 64, zero-filled by TMA), or 32-byte swizzle with
// 16-element atoms (K padded to a multiple of 16 only).  An atom block holds 128
// rows.
__device__ __forceinline__ uint32_t atom_k(int layout) { return layout ? 16u : 64u; }
__device__ __forceinline__ uint32_t atom_bytes(int layout) { return layout ? 4096u : 16384u; }
// byte offset of K step k (16 elements) inside a tile
__device__ __forceinline__ uint32_t kstep_off(int layout, int k) {
  return layout ? (uint32_t)k * 4096u : (uint32_t)(k >> 2) * 16384u + (uint32_t)(k & 3) * 32u;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor of a K-major swizzled tile: start address,
// leading offset (unused for these layouts), 8-row group stride (SBO: 1024 B for
// the 128-byte swizzle, 256 B for the 32-byte swizzle), version 1, layout type
// (2 = 128-byte swizzle, 6 = 32-byte swizzle).
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, int layout) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;
  d |= (uint64_t)((layout ? 256u : 1024u) >> 4) << 32;
  d |= (uint64_t)1u << 46;
  d |= (uint64_t)(layout ? 6u : 2u) << 61;
  return d;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// One arrival by lane 0 of a converged warp, predicated (no branch).
__device__ __forceinline__ void mbar_arrive_lane0(uint32_t bar, int lane) {
  asm volatile(
      "{\n .reg .pred p;\n setp.eq.s32 p, %1, 0;\n"
      " @p mbarrier.arrive.shared::cta.b64 _, [%0];\n}" ::"r"(bar),
      "r"(lane)
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0u;
}
// Whether the phase of parity `parity` is complete, without waiting.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0u;
}
// The same with a suspend-time hint: a thread whose phase is not complete sleeps
// (issuing nothing) until the phase completes or about `ns` nanoseconds pass.
__device__ __forceinline__ bool mbar_try_wait_sleep(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(ns)
      : "memory");
  return ok != 0u;
}
// Suspend hint of the bounded waits (ns): long enough that a waiting thread
// takes no issue slots from the working warps of its scheduler, short enough
// that timeouts and aborts are still noticed promptly.
constexpr uint32_t kWaitSleepNs = 200000u;

struct WaitCtl {
  volatile int *abort_flag;
  unsigned int *status;
  long long limit;
};

// Bounded wait for the phase of parity `parity`; false on timeout or abort.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, const WaitCtl &w,
                                      unsigned int where) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_wait_sleep(bar, parity, kWaitSleepNs)) return true;
    if (*w.abort_flag) return false;
    if (clock64() - t0 > w.limit) {
      *w.abort_flag = 1;
      atomicOr(w.status, kDevTimeout);
      atomicMax(w.status + 1, where);
      return false;
    }
  }
}

// The same bounded wait, reading its limit and status words from the kernel
// parameters and the abort flag through its shared-memory address (keeps no
// per-thread copies of them in registers).
__device__ __forceinline__ bool wait_bar_p(uint32_t bar, uint32_t parity, const ScanParams &p,
                                         uint32_t abort_addr, unsigned int where) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_wait_sleep(bar, parity, kWaitSleepNs)) return true;
    int ab;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(ab) : "r"(abort_addr) : "memory");
    if (ab) return false;
    if (clock64() - t0 > p.timeout_cycles) {
      asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(abort_addr), "r"(1) : "memory");
      atomicOr(p.status, kDevTimeout);
      atomicMax(p.status + 1, where);
      return false;
    }
  }
}

// A warp's wait: one look and one vote when the phase is complete already, else the
// bounded wait; false (in every lane) when some lane's wait gave up.
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, const ScanParams &p,
                                          uint32_t abort_addr, unsigned int where) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  return __all_sync(0xffffffffu, wait_bar_p(bar, parity, p, abort_addr, where));
}

// Wait used while shutting down: ignores the abort flag (copies and MMAs already
// issued must land before the CTA can release its shared memory and TMEM) and
// gives up only after a fixed bound of about two seconds (reported as 32 + where).
// (inline: it is also reached by warps that have given registers away with
// setmaxnreg, which must call no function compiled for more registers)
__device__ __forceinline__ void wait_drain(uint32_t bar, uint32_t parity, unsigned int *status,
                                           unsigned int where) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > 4000000000LL) {
      atomicOr(status, kDevTimeout);
      atomicMax(status + 1, 32u + where);
      return;
    }
  }
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y,
                                            uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
// ---- the same over the two CTAs of a cluster --------------------------------
__device__ __forceinline__ void tc_mma_pair(uint32_t d_tmem, uint64_t da, uint64_t db,
                                            uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(da), "l"(db), "r"(kIdescPair), "r"(accumulate)
      : "memory");
}
// a box of a tensor map into this CTA, its bytes counted on a barrier (shared::cluster
// address) that may be the other CTA's
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap *map, int x, int y,
                                              uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.cta_group::2 [%0], "
      "[%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
// arrives on the barrier at this offset in both CTAs
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], "
      "%1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of CTA `rank`'s copy of a shared-memory address
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t cluster_addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// Counts bytes as arrived that no copy will bring.
__device__ __forceinline__ void mbar_complete_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster_lane0(uint32_t cluster_addr, int lane) {
  asm volatile(
      "{\n .reg .pred p;\n setp.eq.s32 p, %1, 0;\n"
      " @p mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n}" ::"r"(cluster_addr),
      "r"(lane)
      : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0u;
}
// Bounded wait for arrivals of both CTAs.
__device__ __forceinline__ bool wait_bar_cluster(uint32_t bar, uint32_t parity, const WaitCtl &w,
                                                 unsigned int where) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait_cluster(bar, parity)) {
    if (*w.abort_flag) return false;
    if (clock64() - t0 > w.limit) {
      *w.abort_flag = 1;
      atomicOr(w.status, kDevTimeout);
      atomicMax(w.status + 1, where);
      return false;
    }
  }
  return true;
}

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}

#define KRUX_LD16_REGS(r)                                                                       \
  "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),          \
      "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),  \
      "=r"(r[14]), "=r"(r[15])

// 16 consecutive fp32 columns of this warp's 32 TMEM lanes (one lane per thread).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[kEpiSnps]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : KRUX_LD16_REGS(r)
      : "r"(taddr)
      : "memory");
}
// 8 consecutive fp32 columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[kEpiSnpsM]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Same quadratic form without the bound; with permutation batches the df-1 SNPs
// carry negated alpha, gamma so the sign of the result tells the df apart.
__device__ __forceinline__ float kw_s(float u, float v, float al, float be, float ga) {
  const float w = fmaf(be, v, u);
  const float e = ga * v;
  const float t = e * v;
  const float f = al * w;
  return fmaf(f, w, t);
}

// -ln p for df = 1: -ln erfc(x) = x^2 - ln erfcx(x), x = sqrt(H/2) (no underflow).
__device__ __forceinline__ float key1f(float H) {
  const float x2 = 0.5f * H;
  if (!(x2 > 0.f)) return 0.f;
  return x2 - logf(erfcxf(sqrtf(x2)));
}
__device__ __forceinline__ double key64_of(double H, int df) {
  if (df == 2) return 0.5 * H;
  if (df == 1) {
    const double x2 = 0.5 * H;
    if (!(x2 > 0.0)) return 0.0;
    return x2 - log(erfcx(sqrt(x2)));
  }
  return 0.0;
}

// cis mode: only pairs whose SNP and trait lie within the window are reported.
__device__ __forceinline__ bool in_cis_window(const ScanParams &p, int snp, int trait) {
  if (p.cis_window < 0) return true;
  const long long d = (long long)(p.cis_snp_pos[snp] - p.cis_trait_pos[trait]);
  return d <= p.cis_window && -d <= p.cis_window;
}

// FDR histogram bin of a pair with -ln p = key: b = floor((-log10 p - l0) / w),
// clamped to [0, bins).
__device__ __forceinline__ int fdr_bin(double key, double l0, double w, int bins) {
  const double x = (key * 0.43429448190325182765 - l0) / w;
  if (!(x >= 1.0)) return 0;
  if (x >= (double)(bins - 1)) return bins - 1;
  return (int)x;
}

// Upper chi-square tail with df = 1..4 degrees of freedom, Q(df/2, H/2) for
// integer and half-integer shape: df 1: erfc(sqrt x); df 2: e^-x;
// df 3: erfc(sqrt x) + 2 sqrt(x / pi) e^-x; df 4: e^-x (1 + x); x = H/2.
__device__ __forceinline__ double chi2_tail64(double H, int df) {
  if (df <= 0 || !(H > 0.0)) return 1.0;
  const double x = 0.5 * H;
  if (df == 1) return erfc(sqrt(x));
  if (df == 2) return exp(-x);
  if (df == 3) return erfc(sqrt(x)) + 1.12837916709551257390 * sqrt(x) * exp(-x);
  return exp(-x) * (1.0 + x);
}

// The reported p of a hit (df 1, 2; the decisions use kw_p64): exp(-x), x = H/2, as
// 2^-k 2^-f with k = floor(x log2 e) and f the fraction, both from FP64, and 2^-f
// from exp2f; for df = 1, erfc(z) = exp(-z^2) erfcx(z), z = sqrt(x), with erfcx in
// FP32 (smooth, so its argument's rounding barely moves it).  Relative error a few
// 1e-7; no FP64 transcendental.
__device__ __forceinline__ double kw_p_report(double H, int df) {
  const double x = 0.5 * H;
  if (!(x > 0.0)) return 1.0;
  const double t = x * 1.4426950408889634074;  // x log2(e)
  const double k = floor(t);
  if (k > 1000.0) return 0.0;
  const double two_mk = __longlong_as_double((long long)(1023 - (int)k) << 52);  // 2^-k
  double e = (double)exp2f(-(float)(t - k)) * two_mk;
  if (df == 1) e *= (double)erfcxf(sqrtf((float)x));
  return e;
}

struct EpiTrait {
  int trait;        // global trait row of this thread (may be >= T in the last tile)
  bool valid;
  float ntlo, nthi; // -tau (1 -/+ margin)
  double cfac;
  int nan_cnt;      // 0 unless the rank set has NaN in this trait
  const uint16_t *nan_idx;
};

// Group sizes of a pair after removing the trait's NaN samples (section
// "Handling missing values": N_i(n,m) counts the samples present for both).
__device__ __forceinline__ void pair_counts(int nan_cnt, const uint16_t *nan_idx,
                                            const ChunkMeta &m, const uint64_t *codes, int jj,
                                            int &n0, int &n1, int &n2) {
  n0 = m.n[0][jj];
  n1 = m.n[1][jj];
  n2 = m.n[2][jj];
  for (int i = 0; i < nan_cnt; ++i) {
    const int k = nan_idx[i];
    const int code = (int)((codes[k * 2 + (jj >> 5)] >> (2 * (jj & 31))) & 3ull);
    n0 -= code == 0;
    n1 -= code == 1;
    n2 -= code == 2;
  }
}

__device__ __forceinline__ int df_of(int n0, int n1, int n2) {
  const int g = (n0 > 0) + (n1 > 0) + (n2 > 0);
  return g > 0 ? g - 1 : 0;
}

// ---- packed fp32x2 helpers (two SNPs per instruction) ----------------------
__device__ __forceinline__ uint64_t pk2(uint32_t a, uint32_t b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ void upk2(uint64_t r, uint32_t &a, uint32_t &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(r));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float fmax3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float fmin3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Hot test of kEpiSnps SNPs: true when some pair may lie at or above the lower edge of
// the band (q >= 0).  Two SNPs per packed instruction:
//   w = u + beta v,  q = alpha w^2 + gamma v^2 - tau (1 - margin)
// (with permutation batches the form is signed by df and |form| is tested).
template <bool kSigned>
__device__ __forceinline__ bool hit_fast(const uint32_t (&d0)[kEpiSnps], const uint32_t (&d1)[kEpiSnps],
                                         const ChunkMeta &m, int h, float ntlo) {
  const uint64_t *al = reinterpret_cast<const uint64_t *>(m.alpha + kEpiSnps * h);
  const uint64_t *be = reinterpret_cast<const uint64_t *>(m.beta + kEpiSnps * h);
  const uint64_t *ga = reinterpret_cast<const uint64_t *>(m.gamma + kEpiSnps * h);
  const uint64_t nt2 = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
  uint32_t acc = 0xffffffffu;
#pragma unroll
  for (int j = 0; j < kEpiSnps / 2; j += 2) {
    const ulonglong2 A = *reinterpret_cast<const ulonglong2 *>(al + j);
    const ulonglong2 B = *reinterpret_cast<const ulonglong2 *>(be + j);
    const ulonglong2 G = *reinterpret_cast<const ulonglong2 *>(ga + j);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int jj = 2 * (j + t);
      const uint64_t u2 = pk2(d0[jj], d0[jj + 1]);
      const uint64_t v2 = pk2(d1[jj], d1[jj + 1]);
      const uint64_t a2 = t ? A.y : A.x, b2 = t ? B.y : B.x, g2 = t ? G.y : G.x;
      const uint64_t w2 = ffma2(b2, v2, u2);
      const uint64_t e2 = fmul2(g2, v2);
      uint64_t q2;
      if (!kSigned) {
        q2 = ffma2(e2, v2, nt2);
        q2 = ffma2(fmul2(a2, w2), w2, q2);
      } else {
        q2 = ffma2(fmul2(a2, w2), w2, fmul2(e2, v2));
        q2 = fadd2(q2 & 0x7fffffff7fffffffull, nt2);
      }
      uint32_t qa, qb;
      upk2(q2, qa, qb);
      acc &= qa & qb;
    }
  }
  return (int)acc >= 0;
}

// Small non-negative integer (< 2^23) to float, exactly, without a conversion
// instruction: the integer sits in the mantissa of 2^23.
__device__ __forceinline__ float small_int_f(int x) {
  return __int_as_float(0x4b000000 | x) - 8388608.f;
}

// Hot test of a chunk half for a trait with NaN samples (section "Handling missing
// values": N_i(n,m) counts the samples present for both).  Each pair's group sizes
// come from the genotype codes of the trait's c NaN samples: k_i = the NaN samples
// with genotype i, summed over the samples in 4-bit fields (c <= 15; more take the
// rare path at once), n_i' = n_i - k_i.  The test sum_i D_i^2 / n_i' >= q_df is
// taken without a division, as u^2 n1 n2 + v^2 n0 n2 + w^2 n0 n1 >= q_df n0 n1 n2
// (an emptied group has D_i = 0 and counts as n_i' = 1; q_df of the pair's own df,
// q1, q2 = h_df (1 - margin) / cfac).  True if some pair may be a hit; the rare
// path decides it exactly.
__device__ __forceinline__ bool hit_fast_nan(const uint32_t (&d0)[kEpiSnps],
                                             const uint32_t (&d1)[kEpiSnps], const ChunkMeta &m,
                                             int h, const uint64_t *codes, int c,
                                             const uint16_t *nan_idx, float q1, float q2) {
  if (c > 15) return true;
  // k_i of SNPs 8 b .. 8 b + 7 in the 4-bit fields of kb[i][b]
  uint32_t kb[3][2] = {{0u, 0u}, {0u, 0u}, {0u, 0u}};
  for (int i = 0; i < c; ++i) {
    const int k = nan_idx[i];
    const uint32_t x = (uint32_t)(codes[k * 2 + (h >> 1)] >> (32 * (h & 1)));
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      // the 8 two-bit codes of this half-word, each moved to a 4-bit field
      uint32_t z = (x >> (16 * b)) & 0xffffu;
      z = (z | (z << 8)) & 0x00ff00ffu;
      z = (z | (z << 4)) & 0x0f0f0f0fu;
      z = (z | (z << 2)) & 0x33333333u;
      const uint32_t lo = z & 0x11111111u, hi = (z >> 1) & 0x11111111u;
      kb[0][b] += ~(lo | hi) & 0x11111111u;
      kb[1][b] += lo & ~hi;
      kb[2][b] += hi & ~lo;
    }
  }
  const int jb = kEpiSnps * h;
  const uint4 *p0 = reinterpret_cast<const uint4 *>(&m.n[0][jb]);
  const uint4 *p1 = reinterpret_cast<const uint4 *>(&m.n[1][jb]);
  const uint4 *p2 = reinterpret_cast<const uint4 *>(&m.n[2][jb]);
  const float inf = __int_as_float(0x7f800000);
  bool need = false;
#pragma unroll
  for (int hb = 0; hb < 2; ++hb) {  // SNPs 8 hb .. 8 hb + 7
    const uint4 a0 = p0[hb], a1 = p1[hb], a2 = p2[hb];
    const uint32_t w0[4] = {a0.x, a0.y, a0.z, a0.w}, w1[4] = {a1.x, a1.y, a1.z, a1.w},
                   w2[4] = {a2.x, a2.y, a2.z, a2.w};
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int j = 8 * hb + t;
      const int sh = (t & 1) * 16;
      const int n0 = (int)((w0[t >> 1] >> sh) & 0xffffu) - (int)((kb[0][hb] >> (4 * t)) & 15u);
      const int n1 = (int)((w1[t >> 1] >> sh) & 0xffffu) - (int)((kb[1][hb] >> (4 * t)) & 15u);
      const int n2 = (int)((w2[t >> 1] >> sh) & 0xffffu) - (int)((kb[2][hb] >> (4 * t)) & 15u);
      const int groups = (n0 > 0) + (n1 > 0) + (n2 > 0);
      const float thr = groups == 3 ? q2 : (groups == 2 ? q1 : inf);
      const float f0 = small_int_f(max(n0, 1)), f1 = small_int_f(max(n1, 1)),
                  f2 = small_int_f(max(n2, 1));
      const float u = __uint_as_float(d0[j]), v = __uint_as_float(d1[j]);
      const float w = -(u + v);
      const float f12 = f1 * f2;
      const float num = fmaf(w * w, f0 * f1, fmaf(v * v, f0 * f2, u * u * f12));
      need |= fmaf(-thr, f0 * f12, num) >= 0.f;
    }
  }
  return need;
}

// Rare path of a hit-mode chunk half: dense FP64 output, traits with NaN,
// classification of candidates (FP64 inside the band) and the warp-aggregated
// append of hits.  Called by the whole warp; `dv` holds this lane's kEpiSnps D_0
// then kEpiSnps D_1 values (a local copy, so the hot path keeps them in registers).
__device__ __noinline__ void hit_slow(const uint32_t *dv, bool mine, const ChunkMeta &m,
                                      const uint64_t *codes, int h, int trait, bool valid,
                                      float ntlo, float nthi, double cfac, int nan_cnt,
                                      const uint16_t *nan_idx, const GroupDesc &g,
                                      const ScanParams &p, int lane) {
  const int jb = kEpiSnps * h;
  uint32_t hitmask = 0;
  if (mine && valid) {
    const float *al = m.alpha + jb, *be = m.beta + jb, *ga = m.gamma + jb;
    for (int j = 0; j < kEpiSnps; ++j) {
      const int snp = m.snp[jb + j];
      if (snp < 0 || !in_cis_window(p, snp, trait)) continue;
      const float u = __uint_as_float(dv[j]), v = __uint_as_float(dv[kEpiSnps + j]);
      if (p.dense || nan_cnt > 0) {
        int n0, n1, n2;
        pair_counts(nan_cnt, nan_idx, m, codes, jb + j, n0, n1, n2);
        const int df = df_of(n0, n1, n2);
        if (p.dense) {
          const double H = (df > 0 && cfac > 0.0) ? kw_H64((int)u, (int)v, n0, n1, n2, cfac) : 0.0;
          const double pv = (df > 0 && cfac > 0.0) ? kw_p64(H, df) : 1.0;
          const int64_t o = (int64_t)trait * g.dense_ld + (snp - g.dense_snp0);
          g.dense_H[o] = H;
          g.dense_p[o] = pv;
          if (pv < p.pthresh) hitmask |= 1u << j;
        } else if (df > 0) {
          const float w = -(u + v);
          float Q = 0.f;
          if (n0 > 0) Q += u * u / (float)n0;
          if (n1 > 0) Q += v * v / (float)n1;
          if (n2 > 0) Q += w * w / (float)n2;
          const float hq = (float)cfac * Q;
          const float hd = df == 1 ? p.h1 : p.h2;
          if (hq > hd * (1.f - p.margin)) {
            bool hit = hq > hd * (1.f + p.margin);
            if (!hit) hit = kw_p64(kw_H64((int)u, (int)v, n0, n1, n2, cfac), df) < p.pthresh;
            if (hit) hitmask |= 1u << j;
          }
        }
      } else {
        float sv = kw_s(u, v, al[j], be[j], ga[j]);
        if (p.signed_coef) sv = fabsf(sv);
        if (sv + ntlo >= 0.f) {
          bool hit = sv + nthi > 0.f;
          if (!hit) {
            const double H = kw_H64((int)u, (int)v, m.n[0][jb + j], m.n[1][jb + j], m.n[2][jb + j], cfac);
            hit = kw_p64(H, m.df[jb + j]) < p.pthresh;
          }
          if (hit) hitmask |= 1u << j;
        }
      }
    }
  }
  if (!__any_sync(0xffffffffu, hitmask != 0u)) return;
  // warp-aggregated append: one atomic per warp
  const int cnt = __popc(hitmask);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(g.counter, (unsigned long long)total);
  base = __shfl_sync(0xffffffffu, base, 0);
  unsigned long long idx = base + (unsigned long long)(incl - cnt);
  const unsigned long long cap = (unsigned long long)g.capacity;
  while (hitmask) {
    const int j = __ffs(hitmask) - 1;
    hitmask &= hitmask - 1u;
    if (idx < cap) {
      int n0, n1, n2;
      pair_counts(nan_cnt, nan_idx, m, codes, jb + j, n0, n1, n2);
      krux_hit r;
      r.trait = (uint32_t)trait;
      r.snp = (uint32_t)m.snp[jb + j];
      r.d0 = (int32_t)__uint_as_float(dv[j]);
      r.d1 = (int32_t)__uint_as_float(dv[kEpiSnps + j]);
      st_hit(g.hits + idx, r);
      HitAux a;
      a.n0 = (uint16_t)n0;
      a.n1 = (uint16_t)n1;
      a.n2 = (uint16_t)n2;
      a.group = (uint16_t)g.group_id;
      st_aux(g.aux + idx, a);
    }
    ++idx;
  }
}

// FP64 decision for a pair inside the band (rare): p < P_c from the exact sums.
__device__ __noinline__ bool decide64(float u, float v, int n0, int n1, int n2, int df, double cfac,
                                      double pthresh) {
  return kw_p64(kw_H64((int)u, (int)v, n0, n1, n2, cfac), df) < pthresh;
}
// The same decision inline, for the event warps of the plain scan form: they run
// with fewer registers than the kernel was compiled for (setmaxnreg) and must not
// call a function compiled for the full count.
__device__ __forceinline__ bool decide64_inl(float u, float v, int n0, int n1, int n2, int df,
                                             double cfac, double pthresh) {
  return kw_p64(kw_H64((int)u, (int)v, n0, n1, n2, cfac), df) < pthresh;
}


// Rare path of a hit-mode chunk half without dense output or NaN traits, called
// by the whole warp (inlined: a call costs more in register saves than the
// extra code costs the hot loop).  Each lane classifies its candidates (two SNPs per packed
// instruction: at or above the upper band edge -> hit, inside the band -> FP64),
// then the warp appends the hits in lane order with every lane writing records
// (the source lane of record r is the first lane with inclusive count > r, found
// by a binary search over shuffles; its SNP is the (r - excl)-th set bit of that
// lane's mask and the sums come by shuffle), so the records of an event whose
// hits sit in one lane still leave in whole vector stores.  Records first fill this warp's own
// staging segment (`wn` records already there; no atomic); whatever does not fit
// goes straight to the caller's list through the global counter.  Returns the
// number of hits found (the warp's segment counter advances by it).  A compaction
// pass appends the segments after the launch.
__device__ __forceinline__ unsigned int hit_event(const uint32_t *dv, bool mine, const ChunkMeta &m,
                                               int h, int trait, float ntlo, float nthi,
                                               double cfac, const GroupDesc &g,
                                               const ScanParams &p, unsigned int wn, int lane) {
  const int jb = kEpiSnps * h;
  uint32_t hm = 0;
  if (mine) {
    const uint64_t *al = reinterpret_cast<const uint64_t *>(m.alpha + jb);
    const uint64_t *be = reinterpret_cast<const uint64_t *>(m.beta + jb);
    const uint64_t *ga = reinterpret_cast<const uint64_t *>(m.gamma + jb);
    const uint64_t lo2c = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
    const uint64_t hi2c = pk2(__float_as_uint(nthi), __float_as_uint(nthi));
    uint32_t below = 0, not_sure = 0;  // sign bits of s - tau(1 -/+ margin)
#pragma unroll
    for (int j = 0; j < kEpiSnps; j += 2) {
      const uint64_t u2 = pk2(dv[j], dv[j + 1]);
      const uint64_t v2 = pk2(dv[kEpiSnps + j], dv[kEpiSnps + j + 1]);
      const uint64_t w2 = ffma2(be[j / 2], v2, u2);
      const uint64_t e2 = fmul2(ga[j / 2], v2);
      uint64_t s2 = ffma2(fmul2(al[j / 2], w2), w2, fmul2(e2, v2));
      if (p.signed_coef) s2 &= 0x7fffffff7fffffffull;
      uint32_t la, lb, ha, hb;
      upk2(fadd2(s2, lo2c), la, lb);
      upk2(fadd2(s2, hi2c), ha, hb);
      below |= ((la >> 31) | ((lb >> 31) << 1)) << j;
      not_sure |= ((ha >> 31) | ((hb >> 31) << 1)) << j;
    }
    uint32_t cand = ~below & ((1u << kEpiSnps) - 1u);
    if (p.cis_window < 0) {
      // padding and excluded SNPs carry zero coefficients and are never candidates:
      // the clear hits need no loop, only the band goes on to FP64
      hm = p.provisional != 0 ? cand : (cand & ~not_sure);
      cand = p.provisional != 0 ? 0u : (cand & not_sure);
    }
    while (cand) {
      const int j = __ffs(cand) - 1;
      cand &= cand - 1u;
      if (m.snp[jb + j] < 0 || !in_cis_window(p, m.snp[jb + j], trait)) continue;
      bool hit = p.provisional != 0 || ((not_sure >> j) & 1u) == 0u;
      if (!hit)
        hit = decide64(__uint_as_float(dv[j]), __uint_as_float(dv[kEpiSnps + j]), m.n[0][jb + j],
                       m.n[1][jb + j], m.n[2][jb + j], m.df[jb + j], cfac, p.pthresh);
      if (hit) hm |= 1u << j;
    }
  }
  const unsigned int total = __reduce_add_sync(0xffffffffu, (unsigned int)__popc(hm));
  if (total == 0u) return 0u;
  const unsigned int cap = (unsigned int)p.seg_cap;
  const unsigned int sbase = wn;
  const unsigned int over_from = sbase > cap ? sbase : cap;  // first index beyond the segment
  const unsigned int n_over = sbase + total > over_from ? sbase + total - over_from : 0u;
  unsigned long long gbase = 0;
  if (lane == 0 && n_over > 0) gbase = atomicAdd(g.counter, (unsigned long long)n_over);
  gbase = __shfl_sync(0xffffffffu, gbase, 0);
  const size_t seg0 = ((size_t)blockIdx.x * kEpiWarps + (threadIdx.x >> 5)) * cap;
  const uint16_t gid = (uint16_t)g.group_id;
  // lane l's hits take record indices [incl_l - cnt_l, incl_l) after sbase
  const unsigned int cnt = (unsigned int)__popc(hm);
  unsigned int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  for (unsigned int r0 = 0; r0 < total; r0 += 32u) {
    const unsigned int r = r0 + (unsigned int)lane;
    int lo = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {  // first lane with incl > r
      const unsigned int v = __shfl_sync(0xffffffffu, incl, lo + step - 1);
      if (v <= r) lo += step;
    }
    const int src = lo < 31 ? lo : 31;
    const unsigned int src_incl = __shfl_sync(0xffffffffu, incl, src);
    const unsigned int src_cnt = __shfl_sync(0xffffffffu, cnt, src);
    const uint32_t src_hm = __shfl_sync(0xffffffffu, hm, src);
    const uint32_t src_trait = __shfl_sync(0xffffffffu, (uint32_t)trait, src);
    const int j = (int)__fns(src_hm, 0u, (int)(r - (src_incl - src_cnt)) + 1);
    uint32_t du = 0u, dw = 0u;
#pragma unroll
    for (int jj = 0; jj < kEpiSnps; ++jj) {
      const uint32_t a = __shfl_sync(0xffffffffu, dv[jj], src);
      const uint32_t b = __shfl_sync(0xffffffffu, dv[kEpiSnps + jj], src);
      if (jj == j) {
        du = a;
        dw = b;
      }
    }
    if (r < total) {
      const unsigned int idx = sbase + r;
      krux_hit rec;
      rec.trait = src_trait;
      rec.snp = (uint32_t)m.snp[jb + j];
      rec.d0 = (int32_t)__uint_as_float(du);
      rec.d1 = (int32_t)__uint_as_float(dw);
      HitAux x;
      x.n0 = m.n[0][jb + j];
      x.n1 = m.n[1][jb + j];
      x.n2 = m.n[2][jb + j];
      x.group = gid;
      if (idx < cap) {
        st_hit(p.seg_hits + seg0 + idx, rec);
        st_aux(p.seg_aux + seg0 + idx, x);
      } else {
        const unsigned long long gi = gbase + (idx - over_from);
        if (gi < (unsigned long long)g.capacity) {
          st_hit(g.hits + gi, rec);
          st_aux(g.aux + gi, x);
        }
      }
    }
  }
  return total;
}

// The same event with the records appended SNP column by SNP column (lanes with
// a hit of the same SNP take consecutive records).  Smaller than the lane-order
// append above; the permutation form uses it, where register room matters more.
__device__ __forceinline__ unsigned int hit_event_cols(const uint32_t *dv, bool mine, const ChunkMeta &m,
                                               int h, int trait, float ntlo, float nthi,
                                               double cfac, const GroupDesc &g,
                                               const ScanParams &p, unsigned int wn, int lane) {
  const int jb = kEpiSnps * h;
  uint32_t hm = 0;
  if (mine) {
    const uint64_t *al = reinterpret_cast<const uint64_t *>(m.alpha + jb);
    const uint64_t *be = reinterpret_cast<const uint64_t *>(m.beta + jb);
    const uint64_t *ga = reinterpret_cast<const uint64_t *>(m.gamma + jb);
    const uint64_t lo2c = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
    const uint64_t hi2c = pk2(__float_as_uint(nthi), __float_as_uint(nthi));
    uint32_t below = 0, not_sure = 0;  // sign bits of s - tau(1 -/+ margin)
#pragma unroll
    for (int j = 0; j < kEpiSnps; j += 2) {
      const uint64_t u2 = pk2(dv[j], dv[j + 1]);
      const uint64_t v2 = pk2(dv[kEpiSnps + j], dv[kEpiSnps + j + 1]);
      const uint64_t w2 = ffma2(be[j / 2], v2, u2);
      const uint64_t e2 = fmul2(ga[j / 2], v2);
      uint64_t s2 = ffma2(fmul2(al[j / 2], w2), w2, fmul2(e2, v2));
      if (p.signed_coef) s2 &= 0x7fffffff7fffffffull;
      uint32_t la, lb, ha, hb;
      upk2(fadd2(s2, lo2c), la, lb);
      upk2(fadd2(s2, hi2c), ha, hb);
      below |= ((la >> 31) | ((lb >> 31) << 1)) << j;
      not_sure |= ((ha >> 31) | ((hb >> 31) << 1)) << j;
    }
    uint32_t cand = ~below & ((1u << kEpiSnps) - 1u);
    while (cand) {
      const int j = __ffs(cand) - 1;
      cand &= cand - 1u;
      if (m.snp[jb + j] < 0 || !in_cis_window(p, m.snp[jb + j], trait)) continue;
      bool hit = p.provisional != 0 || ((not_sure >> j) & 1u) == 0u;
      if (!hit)
        hit = decide64(__uint_as_float(dv[j]), __uint_as_float(dv[kEpiSnps + j]), m.n[0][jb + j],
                       m.n[1][jb + j], m.n[2][jb + j], m.df[jb + j], cfac, p.pthresh);
      if (hit) hm |= 1u << j;
    }
  }
  const unsigned int total = __reduce_add_sync(0xffffffffu, (unsigned int)__popc(hm));
  if (total == 0u) return 0u;
  const unsigned int cap = (unsigned int)p.seg_cap;
  const unsigned int sbase = wn;
  const unsigned int over_from = sbase > cap ? sbase : cap;  // first index beyond the segment
  const unsigned int n_over = sbase + total > over_from ? sbase + total - over_from : 0u;
  unsigned long long gbase = 0;
  if (lane == 0 && n_over > 0) gbase = atomicAdd(g.counter, (unsigned long long)n_over);
  gbase = __shfl_sync(0xffffffffu, gbase, 0);
  const size_t seg0 = ((size_t)blockIdx.x * kEpiWarps + (threadIdx.x >> 5)) * cap;
  const uint32_t below_me = (1u << lane) - 1u;
  const uint16_t gid = (uint16_t)g.group_id;
  unsigned int run = sbase;  // index of the next record (same in every lane)
  uint32_t cols = __reduce_or_sync(0xffffffffu, hm);
  while (cols) {
    const int j = __ffs(cols) - 1;
    cols &= cols - 1u;
    const bool mine_j = (hm >> j) & 1u;
    const uint32_t bal = __ballot_sync(0xffffffffu, mine_j);
    if (mine_j) {
      const unsigned int idx = run + (unsigned int)__popc(bal & below_me);
      krux_hit r;
      r.trait = (uint32_t)trait;
      r.snp = (uint32_t)m.snp[jb + j];
      r.d0 = (int32_t)__uint_as_float(dv[j]);
      r.d1 = (int32_t)__uint_as_float(dv[kEpiSnps + j]);
      HitAux x;
      x.n0 = m.n[0][jb + j];
      x.n1 = m.n[1][jb + j];
      x.n2 = m.n[2][jb + j];
      x.group = gid;
      if (idx < cap) {
        st_hit(p.seg_hits + seg0 + idx, r);
        st_aux(p.seg_aux + seg0 + idx, x);
      } else {
        const unsigned long long gi = gbase + (idx - over_from);
        if (gi < (unsigned long long)g.capacity) {
          st_hit(g.hits + gi, r);
          st_aux(g.aux + gi, x);
        }
      }
    }
    run += (unsigned int)__popc(bal);
  }
  return total;
}

// ---- the plain scan form: one warp per chunk of an accumulator pair ----------
// 16 consecutive fp32 columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld16p(uint32_t taddr, uint32_t *r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// kFastSnps / 2 = 16 SNPs' D_0 and D_1 (columns c and 64 + c of the chunk) of this lane.
__device__ __forceinline__ void tmem_ld_half(uint32_t taddr, uint32_t (&u)[kFastSnps / 2],
                                             uint32_t (&v)[kFastSnps / 2]) {
  tmem_ld16p(taddr, u);
  tmem_ld16p(taddr + 64u, v);
}

// The four rows of 8 SNPs (markers with up to five groups; columns 32 i + ..).
__device__ __forceinline__ void tmem_ld8p(uint32_t taddr, uint32_t *r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
                 "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_rows(uint32_t taddr, uint32_t (&u)[2 * kEpiSnpsM],
                                             uint32_t (&v)[2 * kEpiSnpsM]) {
  tmem_ld8p(taddr, u);
  tmem_ld8p(taddr + 32u, u + kEpiSnpsM);
  tmem_ld8p(taddr + 64u, v);
  tmem_ld8p(taddr + 96u, v + kEpiSnpsM);
}

// Hot test of the plain form's traits with NaN samples on NS SNPs of a chunk (from SNP
// `off`): true when some pair may lie at or above the lower edge of the band (q >= 0),
// two SNPs per packed instruction, w = P + beta Q, q = alpha w^2 + gamma Q^2 -
// tau (1 - margin).  Blocks of 16 SNPs; two sign accumulators.
// The coefficients come from the three arrays of a CoefSet.
template <int NS>
__device__ __forceinline__ bool hit_fast_wc(const uint32_t (&d0)[NS], const uint32_t (&d1)[NS],
                                            const float *alpha, const float *beta,
                                            const float *gamma, int off, float ntlo) {
  const uint64_t nt2 = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
  uint32_t acc0 = 0xffffffffu, acc1 = 0xffffffffu;  // AND of the sign bits (two chains)
#pragma unroll
  for (int b = 0; b < NS / 16; ++b) {
    const uint64_t *al = reinterpret_cast<const uint64_t *>(alpha + off + 16 * b);
    const uint64_t *be = reinterpret_cast<const uint64_t *>(beta + off + 16 * b);
    const uint64_t *ga = reinterpret_cast<const uint64_t *>(gamma + off + 16 * b);
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      const ulonglong2 A = *reinterpret_cast<const ulonglong2 *>(al + j);
      const ulonglong2 B = *reinterpret_cast<const ulonglong2 *>(be + j);
      const ulonglong2 G = *reinterpret_cast<const ulonglong2 *>(ga + j);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int jj = 16 * b + 2 * (j + t);
        const uint64_t u2 = pk2(d0[jj], d0[jj + 1]);
        const uint64_t v2 = pk2(d1[jj], d1[jj + 1]);
        const uint64_t a2 = t ? A.y : A.x, b2 = t ? B.y : B.x, g2 = t ? G.y : G.x;
        const uint64_t w2 = ffma2(b2, v2, u2);
        const uint64_t e2 = fmul2(g2, v2);
        uint64_t q2 = ffma2(e2, v2, nt2);
        q2 = ffma2(fmul2(a2, w2), w2, q2);
        uint32_t qa, qb;
        upk2(q2, qa, qb);
        if (t) acc1 &= qa & qb;
        else acc0 &= qa & qb;
      }
    }
    // compiler barrier: the next block's coefficient loads are not hoisted above
    // this one (the accumulator registers stay live throughout)
    if (b + 1 < NS / 16) asm volatile("" ::: "memory");
  }
  return (int)(acc0 & acc1) >= 0;
}
// Hot test of the plain forms on the accumulators P and Q of NS SNPs (weighted rows,
// ChunkMeta): true when some P^2 + Q^2 reaches -ntlo.  Two SNPs per packed
// instruction, two FP32 operations and half a sign accumulation per pair; no
// coefficient is read.  With indicator rows and the coefficients of ChunkMeta the
// same test took five operations and three shared-memory words per SNP: 3.9 ms for
// 20,000 x 500,000 x 102 without planted effects against 2.6 ms with this one.
template <int NS>
__device__ __forceinline__ bool hit_pq(const uint32_t (&P)[NS], const uint32_t (&Q)[NS], float ntlo) {
  const uint64_t nt2 = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
  uint32_t acc0 = 0xffffffffu, acc1 = 0xffffffffu;  // AND of the sign bits (two chains)
#pragma unroll
  for (int j = 0; j < NS; j += 4) {
    const uint64_t q0 = pk2(Q[j], Q[j + 1]), q1 = pk2(Q[j + 2], Q[j + 3]);
    const uint64_t p0 = pk2(P[j], P[j + 1]), p1 = pk2(P[j + 2], P[j + 3]);
    const uint64_t s0 = ffma2(p0, p0, ffma2(q0, q0, nt2));
    const uint64_t s1 = ffma2(p1, p1, ffma2(q1, q1, nt2));
    uint32_t x, y;
    upk2(s0, x, y);
    acc0 &= x & y;
    upk2(s1, x, y);
    acc1 &= x & y;
  }
  return (int)(acc0 & acc1) >= 0;
}

// The same in a permutation batch, where the two classes of SNPs have bounds of their
// own (b1 for df 1, b2 for df 2): the bound of each SNP is selected by its sign
// (ChunkMeta's sgn, +1 for df 2) as -(b1 + b2) / 2 + sgn (b1 - b2) / 2.  A SNP that is never
// tested has sgn 0, so that its zeros stay below the bound also where one class has no
// SNP, and its sum with the other's bound is lost in the rounding (with +1, data of two-group SNPs
// and 10 % monomorphic ones, 16 x 3,000 x 20,000 with FDR counts, sent every trait of every block
// to the event warps: 102 ms).
template <int NS>
__device__ __forceinline__ bool hit_pq2(const uint32_t (&P)[NS], const uint32_t (&Q)[NS],
                                        const float *sgn, float b1, float b2) {
  const float mid = -0.5f * (b1 + b2), dif = 0.5f * (b1 - b2);
  const uint64_t m2 = pk2(__float_as_uint(mid), __float_as_uint(mid));
  const uint64_t f2 = pk2(__float_as_uint(dif), __float_as_uint(dif));
  uint32_t acc0 = 0xffffffffu, acc1 = 0xffffffffu;
#pragma unroll
  for (int j = 0; j < NS; j += 4) {
    const ulonglong2 g = *reinterpret_cast<const ulonglong2 *>(sgn + j);
    const uint64_t q0 = pk2(Q[j], Q[j + 1]), q1 = pk2(Q[j + 2], Q[j + 3]);
    const uint64_t p0 = pk2(P[j], P[j + 1]), p1 = pk2(P[j + 2], P[j + 3]);
    const uint64_t s0 = ffma2(p0, p0, ffma2(q0, q0, ffma2(g.x, f2, m2)));
    const uint64_t s1 = ffma2(p1, p1, ffma2(q1, q1, ffma2(g.y, f2, m2)));
    uint32_t x, y;
    upk2(s0, x, y);
    acc0 &= x & y;
    upk2(s1, x, y);
    acc1 &= x & y;
  }
  return (int)(acc0 & acc1) >= 0;
}

// Seed pass of a permutation batch: the largest P^2 + Q^2 of a block of one class.
template <int NS>
__device__ __forceinline__ float top_pq(const uint32_t (&P)[NS], const uint32_t (&Q)[NS]) {
  float m = 0.f;
#pragma unroll
  for (int j = 0; j < NS; j += 2) {
    const uint64_t q0 = pk2(Q[j], Q[j + 1]), p0 = pk2(P[j], P[j + 1]);
    uint32_t sa, sb;
    upk2(ffma2(p0, p0, fmul2(q0, q0)), sa, sb);
    m = fmax3(m, __uint_as_float(sa), __uint_as_float(sb));
  }
  return m;
}
// And of a mixed block: of the df-2 SNPs into smax and, negated, of the df-1 SNPs into
// smin.
template <int NS>
__device__ __forceinline__ void range_pq(const uint32_t (&P)[NS], const uint32_t (&Q)[NS],
                                         const float *sgn, float &smax, float &smin) {
#pragma unroll
  for (int j = 0; j < NS; j += 2) {
    const uint64_t g = *reinterpret_cast<const uint64_t *>(sgn + j);
    const uint64_t q0 = pk2(Q[j], Q[j + 1]), p0 = pk2(P[j], P[j + 1]);
    const uint64_t s2 = fmul2(g, ffma2(p0, p0, fmul2(q0, q0)));
    uint32_t sa, sb;
    upk2(s2, sa, sb);
    smax = fmax3(smax, __uint_as_float(sa), __uint_as_float(sb));
    smin = fmin3(smin, __uint_as_float(sa), __uint_as_float(sb));
  }
}

// D_0 and D_1 of a pair from its accumulators: P = A0 D_a + A1 D_b, Q = G D_b are exact
// (ChunkMeta), so both quotients round to the integers they are.  w0 = 0 (a SNP that
// is never tested): zeros.  kWhole off: standardised values instead of ranks, whose
// sums are not whole numbers (a regression's SNP has no Q row: D_1 = 0, D_0 = P / A0
// stands for both).
template <bool kWhole = true>
__device__ __forceinline__ void pq_sums(float P, float Q, uint32_t w0, uint32_t w1, float &u, float &v) {
  const float a0 = __half2float(__ushort_as_half((unsigned short)(w0 & 0xffffu)));
  const float a1 = __half2float(__ushort_as_half((unsigned short)(w0 >> 16)));
  const float g = __half2float(__ushort_as_half((unsigned short)(w1 & 0xffffu)));
  if (!(a0 > 0.f)) {
    u = 0.f;
    v = 0.f;
    return;
  }
  float db = kWhole || g > 0.f ? __fdividef(Q, g) : 0.f;
  if (kWhole) db = rintf(db);
  float da = __fdividef(fmaf(-a1, db, P), a0);
  if (kWhole) da = rintf(da);
  const float dl = -(da + db);
  const uint32_t a = (w1 >> 16) & 3u, b = (w1 >> 18) & 3u;
  u = a == 0u ? da : (b == 0u ? db : dl);
  v = a == 1u ? da : (b == 1u ? db : dl);
}

// ---- hit events of the plain scan form, handled by the event warps ---------
// Several epilogue warps claim tickets at once, so one of them may claim an
// entry's use k while uses k-1, k-2 are still pending: a phase-parity wait
// cannot tell those apart.  A filler therefore waits on the entry's release count
// (uses the event warp has finished) reaching k; the uses of an entry are then
// filled in order, and its single consumer can wait on the full barrier by phase
// parity.
template <int kEntries>
struct EvRing {
  EvEntry *ent;
  uint32_t bar0;                // ev_full[e] at bar0 + 8 e
  unsigned int *released;       // [kEntries] uses of each entry the event warps have finished
  unsigned long long *word;     // tickets claimed (low 40 bits), epilogue warps done (above)
  __device__ __forceinline__ uint32_t full(int e) const { return bar0 + 8u * (uint32_t)e; }
};
constexpr unsigned long long kEvTicketMask = (1ull << 40) - 1ull;

// Bounded wait of a lane until the entry of ticket t is free for its use t /
// kEntries; false on timeout or abort.
template <int kEntries>
__device__ __forceinline__ bool ev_gate(const EvRing<kEntries> &ev, unsigned long long t,
                                        const ScanParams &p, uint32_t abort_addr) {
  const unsigned int k = (unsigned int)(t / kEntries);
  const volatile unsigned int *rel = ev.released + (t % kEntries);
  if (*rel >= k) return true;
  const long long t0 = clock64();
  while (*rel < k) {
    __nanosleep(128);
    int ab;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(ab) : "r"(abort_addr) : "memory");
    if (ab) return false;
    if (clock64() - t0 > p.timeout_cycles) {
      asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(abort_addr), "r"(1) : "memory");
      atomicOr(p.status, kDevTimeout);
      atomicMax(p.status + 1, 16u);
      return false;
    }
  }
  return true;
}

// An epilogue warp hands the traits of a half-block whose hot test found a candidate to
// the event warps: one entry per such trait lane (tickets claimed together), each with
// that lane's accumulators and constants (`own`, by the lane) and the SNPs' metadata
// (`meta`, by a half-warp per entry).  Each lane waits for its own entry to be free, and
// all of the warp's entries are filled between one pair of fences (a lap of the ring at
// most: no entry waits for another of the same lap).  One entry after the other, each
// with its own wait, fences and arrival: 20,000 x 100,000 x 102 with 76,000 isolated
// hits 643 us, now 628; 16 x 20,000 x 200,000 permutations 24.9 -> 23.9 ms in the
// main launch.  False if a wait gave up.
template <int kEntries, class Own, class Meta>
__device__ __forceinline__ bool ev_fill(const EvRing<kEntries> &ev, bool need, const ScanParams &p,
                                        uint32_t abort_addr, int lane, Own own, Meta meta) {
  const uint32_t lanes = __ballot_sync(0xffffffffu, need);
  const int n = __popc(lanes), rank = __popc(lanes & ((1u << lane) - 1u));
  unsigned long long t = 0;
  if (lane == 0) t = atomicAdd(ev.word, (unsigned long long)n) & kEvTicketMask;
  t = __shfl_sync(0xffffffffu, t, 0);
  for (int lap = 0; lap < n; lap += kEntries) {
    const bool mine = need && rank >= lap && rank < lap + kEntries;
    const int e = (int)((t + (unsigned long long)rank) % kEntries);
    if (!__all_sync(0xffffffffu, !mine || ev_gate(ev, t + (unsigned long long)rank, p, abort_addr)))
      return false;
    __threadfence_block();  // the event warps' reads of the old contents come first
    __syncwarp();
    if (mine) own(ev.ent[e]);
    for (int i = lap + (lane >> 4); i < min(n, lap + kEntries); i += 2)
      meta(ev.ent[(int)((t + (unsigned long long)i) % kEntries)]);
    __threadfence_block();
    __syncwarp();
    if (mine) mbar_arrive(ev.full(e));
  }
  return true;
}
template <int kEntries>
__device__ __forceinline__ bool ev_submit(const EvRing<kEntries> &ev, const uint32_t (&u)[kEvSnps],
                                          const uint32_t (&v)[kEvSnps], bool need,
                                          const ChunkMeta &m, int off, float tau,
                                          int trait, int group, int ag, float b1, float b2,
                                          uint32_t id1, uint32_t id2, int nan, const ScanParams &p,
                                          uint32_t abort_addr, int lane) {
  const int j = lane & (kEvSnps - 1), jo = off + j;
  const float al = m.alpha[jo], be = m.beta[jo], ga = m.gamma[jo];
  const int32_t sn = m.snp[jo];
  const uint32_t n01 = (uint32_t)m.n[0][jo] | ((uint32_t)m.n[1][jo] << 16);
  const uint32_t n2df = (uint32_t)m.n[2][jo] | ((uint32_t)m.df[jo] << 16);
  const uint32_t w0 = m.pq0[jo], w1 = m.pq1[jo];
  return ev_fill(
      ev, need, p, abort_addr, lane,
      [&](EvEntry &E) {
#pragma unroll
        for (int i = 0; i < kEvSnps; i += 4) {
          *reinterpret_cast<uint4 *>(E.u + i) = make_uint4(u[i], u[i + 1], u[i + 2], u[i + 3]);
          *reinterpret_cast<uint4 *>(E.v + i) = make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        }
        E.tau = tau;
        E.trait = trait;
        E.group = group;
        E.ag = ag;
        E.b1 = b1;
        E.b2 = b2;
        E.id1 = id1;
        E.id2 = id2;
        E.nan = nan;
      },
      [&](EvEntry &E) {
        E.alpha[j] = al;
        E.beta[j] = be;
        E.gamma[j] = ga;
        E.snp[j] = sn;
        E.n01[j] = n01;
        E.n2df[j] = n2df;
        E.pq0[j] = w0;
        E.pq1[j] = w1;
      });
}

// Group fields an event warp needs, cached across entries.
// Identity of a pair for exact-copy detection in permutation batches: a hash of
// its centred sums (copies of a SNP inside an LD block have the same sums and
// group sizes, hence the same statistic; pairs with equal sums and equal FP32
// form values but different group sizes would need an FP32 coincidence on top).
__device__ __forceinline__ uint32_t pair_id(int u, int v) {
  return (uint32_t)u * 0x9E3779B1u ^ (uint32_t)v * 0x85EBCA77u;
}

struct EvGroup {
  int index = -1;
  krux_hit *hits;
  HitAux *aux;
  HitAux2 *aux2;
  unsigned long long *counter;
  int64_t capacity;
  uint16_t gid;
  double *minp_key;
  unsigned long long *minp_bound;
  int64_t rows;
  const uint16_t *nan_idx;  // NaN sample lists, N entries per trait
  const int8_t *geno;       // genotype rows (by output SNP index)
  int64_t ldg;
  int N;
};

__device__ __forceinline__ void ev_group(EvGroup &G, const ScanParams &p, int group) {
  if (group == G.index) return;
  const GroupDesc &g = p.groups[group];
  G.index = group;
  G.hits = g.hits;
  G.aux = g.aux;
  G.aux2 = g.aux2;
  G.counter = g.counter;
  G.capacity = g.capacity;
  G.gid = (uint16_t)g.group_id;
  G.minp_key = g.minp_key;
  G.minp_bound = g.minp_bound;
  G.rows = g.rows_per_agroup;
  G.nan_idx = g.nan_idx;
  G.geno = g.geno;
  G.ldg = g.ldg;
  G.N = g.N;
}

// An event warp works on two entries at a time, one per half-warp: lane 16 h + j takes
// the pair (trait, SNP j) of half h's entry.  What it needs of the entry is copied to
// registers first, so that the entry is free again before the classification, its
// divisions and its global stores.  Event throughput bounds inputs with many hits per
// block: 2,000 x 10,000 x 102 with 1.7 % hits took 506 us a call with one entry per
// warp, held until its stores were issued, and 402 us this way.
struct EvLane {
  float P, Q, al, be, ga, tau, b1, b2;
  uint32_t w0, w1, n01, n2df, id1, id2;
  int snp, trait, group, ag, nan;
  __device__ __forceinline__ void load(const EvEntry &E, int j) {
    P = E.u[j];
    Q = E.v[j];
    w0 = E.pq0[j];
    w1 = E.pq1[j];
    al = E.alpha[j];
    be = E.beta[j];
    ga = E.gamma[j];
    snp = E.snp[j];
    n01 = E.n01[j];
    n2df = E.n2df[j];
    tau = E.tau;
    trait = E.trait;
    group = E.group;
    ag = E.ag;
    b1 = E.b1;
    b2 = E.b2;
    id1 = E.id1;
    id2 = E.id2;
    nan = E.nan;
  }
};

// A permuted pair's entry (section "P-value calculation and empirical FDR
// correction": the minimum p of each permuted trait over all SNPs), one per half-warp:
// the lanes take the pairs past the bounds the entry was filled with, list them for
// their FP64 -ln p, and raise the trait's class bounds (largest df-1 |s| and df-2 s of
// the pairs listed, less the margin: a later pair of the class below them cannot beat
// those pairs).  With the FDR histogram on, every pair at or above the band is listed.
__device__ __forceinline__ void ev_minp(EvLane &E, EvGroup &G, const ScanParams &p, int lane,
                                        bool on, float s, float u, float v, unsigned int &mcn,
                                        int ev_warp) {
  const bool valid = on && E.snp >= 0;
  const uint32_t half = 0xffffu << (lane & 16);
  // b1, b2: the classes' largest decided values when the entry was filled, id1, id2
  // the identities of the pairs that have them; exact copies of those pairs are
  // decided already
  const float keep = 1.f - p.margin;
  const uint32_t pid = pair_id((int)u, (int)v);
  if (p.fdr_hist != nullptr && on) {
    ev_group(G, p, E.group);
    const uint4 bb = __ldcg(reinterpret_cast<const uint4 *>(G.minp_bound) +
                            (int64_t)(E.ag - 1) * G.rows + E.trait);
    E.b1 = fmaxf(__uint_as_float(bb.y), 1e-30f);
    E.id1 = bb.x;
    E.b2 = fmaxf(__uint_as_float(bb.w), 1e-30f);
    E.id2 = bb.z;
  }
  bool cand = valid && ((s > E.b2 * keep && !(s == E.b2 && pid == E.id2)) ||
                        (-s > E.b1 * keep && !(-s == E.b1 && pid == E.id1)));
  // within a class the key grows with the value: only the entry's largest value
  // of each class, and values within the margin of it, can hold the class's best
  float c1 = cand && s < 0.f ? -s : 0.f, c2 = cand && s > 0.f ? s : 0.f;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    c1 = fmaxf(c1, __shfl_xor_sync(0xffffffffu, c1, o));
    c2 = fmaxf(c2, __shfl_xor_sync(0xffffffffu, c2, o));
  }
  cand = cand && (s > 0.f ? s >= c2 * keep : -s >= c1 * keep);
  const bool band = valid && p.fdr_hist != nullptr && fabsf(s) >= E.tau * keep;
  const bool need = cand || band;
  const uint32_t bal = __ballot_sync(0xffffffffu, need);
  const unsigned int n = (unsigned int)__popc(bal);
  // identities of the pairs that hold the classes' largest values (the largest
  // identity among ties)
  const bool h1 = cand && s < 0.f && -s == c1, h2 = cand && s > 0.f && s == c2;
  const uint32_t w1 = __ballot_sync(0xffffffffu, h1) & half, w2 = __ballot_sync(0xffffffffu, h2) & half;
  uint32_t i1 = h1 ? pid : 0u, i2 = h2 ? pid : 0u;
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    i1 = max(i1, __shfl_xor_sync(0xffffffffu, i1, o));
    i2 = max(i2, __shfl_xor_sync(0xffffffffu, i2, o));
  }
  if (mcn + n <= (unsigned int)p.mc_cap) {
    // the list has room: the FP64 work runs after the launch, in parallel
    if (need) {
      MinpPair r;
      r.u = (int32_t)u;
      r.v = (int32_t)v;
      r.n01 = E.n01;
      r.n2df = E.n2df;
      r.trait = E.trait;
      r.agb = E.ag | (band ? 1 << 16 : 0) | (cand ? 1 << 17 : 0);
      const size_t base = ((size_t)blockIdx.x * 2 + ev_warp) * (size_t)p.mc_cap;
      p.mc_list[base + mcn + (unsigned int)__popc(bal & ((1u << lane) - 1u))] = r;
    }
    mcn += n;
  } else if (need) {  // full: decide here
    const int df = (int)(E.n2df >> 16);
    const double cfac = p.groups[E.group].cfac[E.trait];
    double key = -1.0;
    if (df > 0 && cfac > 0.0)
      key = key64_of(kw_H64((int)u, (int)v, (int)(E.n01 & 0xffffu), (int)(E.n01 >> 16),
                            (int)(E.n2df & 0xffffu), cfac),
                     df);
    if (band && key > -log(p.pthresh))
      atomicAdd(p.fdr_hist + (int64_t)E.ag * p.fdr_bins + fdr_bin(key, p.fdr_l0, p.fdr_w, p.fdr_bins),
                1ull);
    if (cand && key > 0.0) {
      ev_group(G, p, E.group);
      atomicMax(reinterpret_cast<unsigned long long *>(G.minp_key + (int64_t)(E.ag - 1) * G.rows +
                                                       E.trait),
                (unsigned long long)__double_as_longlong(key));
    }
  }
  if (on && (lane & 15) == 0) {
    ev_group(G, p, E.group);
    const int64_t idx = (int64_t)(E.ag - 1) * G.rows + E.trait;
    if (c1 > E.b1 && w1)
      atomicMax(G.minp_bound + 2 * idx, ((unsigned long long)__float_as_uint(c1) << 32) | i1);
    if (c2 > E.b2 && w2)
      atomicMax(G.minp_bound + 2 * idx + 1, ((unsigned long long)__float_as_uint(c2) << 32) | i2);
  }
}

// Event modes: the plain scan, a permutation batch, the plain scan with NaN.
enum EvMode { kEvPlain = 0, kEvPerm = 1, kEvNan = 2 };

// An event warp's work on up to two entries (`on`: this lane's half has one): each
// lane classifies its pair in FP32 from the exact sums (at or above the upper band
// edge: hit; inside the band: decided in FP64) and the hits are appended in SNP order,
// one record per lane, into this warp's staging region of kEpiWarps / 2 segments of
// the CTA (`wn` records already there); what does not fit goes to the group's list
// through its counter.  For a trait with NaN
// samples (kEvNan) the pair's group sizes are first made exact (section "Handling
// missing values": N_i' counts the samples present for both): the genotypes of
// the trait's NaN samples at the SNP are taken off N_i, and the form is evaluated
// with those sizes and the df they leave.  Returns the number of hits.
template <int kMode>
__device__ __forceinline__ unsigned int ev_process(EvLane &E, bool on, EvGroup &G,
                                                   const ScanParams &p, unsigned int wn, int lane,
                                                   int ev_warp, unsigned int &mcn) {
  float u, v;
  const bool param = kMode == kEvPlain && p.provisional != 0;
  if (param) pq_sums<false>(E.P, E.Q, E.w0, E.w1, u, v);
  else pq_sums(E.P, E.Q, E.w0, E.w1, u, v);
  const float sv = kw_s(u, v, E.al, E.be, E.ga);
  float s = sv;
  bool act = on && E.snp >= 0;
  if constexpr (kMode == kEvPerm) {
    // permuted pairs: min-p and FDR work, no hit record
    if (__any_sync(0xffffffffu, on && E.ag > 0)) ev_minp(E, G, p, lane, on && E.ag > 0, sv, u, v, mcn, ev_warp);
    act = act && E.ag == 0;
    s = fabsf(sv);  // df-1 values are negated in permutation batches
  }
  if constexpr (kMode == kEvNan) {
    const int c = E.nan;
    if (act && c > 0) {
      ev_group(G, p, E.group);
      int n0 = (int)(E.n01 & 0xffffu), n1 = (int)(E.n01 >> 16), n2 = (int)(E.n2df & 0xffffu);
      const uint16_t *ni = G.nan_idx + (int64_t)E.trait * G.N;
      const int8_t *gr = G.geno + (int64_t)E.snp * G.ldg;
      for (int i = 0; i < c; i += 4) {  // four samples' loads in flight at once
        int k[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) k[t] = i + t < c ? (int)ni[i + t] : -1;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          const int code = k[t] >= 0 ? (int)gr[k[t]] : -1;  // -1 (missing): in no group
          n0 -= code == 0;
          n1 -= code == 1;
          n2 -= code == 2;
        }
      }
      const int df = df_of(n0, n1, n2);
      s = 0.f;
      if (df > 0) {
        const float w = -(u + v);
        float q = 0.f;
        if (n0 > 0) q += u * u / (float)n0;
        if (n1 > 0) q += v * v / (float)n1;
        if (n2 > 0) q += w * w / (float)n2;
        s = q / (df == 1 ? p.h1 : p.h2);
      }
      E.n01 = (uint32_t)n0 | ((uint32_t)n1 << 16);
      E.n2df = (uint32_t)n2 | ((uint32_t)df << 16);
    }
  }
  bool cand = act && s + -E.tau * (1.f - p.margin) >= 0.f;
  if (kMode != kEvPerm && cand) cand = in_cis_window(p, E.snp, E.trait);
  // (the parametric comparison keeps its whole band: it is decided after the launch)
  bool hit = cand && (param || s + -E.tau * (1.f + p.margin) >= 0.f);
  if (cand && !hit)  // inside the band: FP64 (rare)
    hit = decide64_inl(u, v, (int)(E.n01 & 0xffffu), (int)(E.n01 >> 16), (int)(E.n2df & 0xffffu),
                       (int)(E.n2df >> 16), p.groups[E.group].cfac[E.trait], p.pthresh);
  const uint32_t bal = __ballot_sync(0xffffffffu, hit);
  const unsigned int n = (unsigned int)__popc(bal);
  if (n == 0u) return 0u;
  constexpr int kSegs = kEpiWarps / 2;  // staging segments per event warp
  const unsigned int cap = (unsigned int)(kSegs * p.seg_cap);
  const unsigned int idx = wn + (unsigned int)__popc(bal & ((1u << lane) - 1u));
  const bool over = hit && idx >= cap;
  const uint32_t obal = __ballot_sync(0xffffffffu, over);
  unsigned long long gi = 0;
  if (hit) ev_group(G, p, E.group);
  if (obal != 0u) {  // one reservation per half (the halves may belong to different lists)
    const uint32_t mine = obal & (0xffffu << (lane & 16));
    const int lead = mine != 0u ? __ffs((int)mine) - 1 : 0;
    if (over && lane == lead) gi = atomicAdd(G.counter, (unsigned long long)__popc(mine));
    gi = __shfl_sync(0xffffffffu, gi, lead) + (unsigned int)__popc(mine & ((1u << lane) - 1u));
  }
  if (hit) {
    krux_hit rec;
    rec.trait = (uint32_t)E.trait;
    rec.snp = (uint32_t)E.snp;
    rec.d0 = (int32_t)u;
    rec.d1 = (int32_t)v;
    HitAux x;
    x.n0 = (uint16_t)(E.n01 & 0xffffu);
    x.n1 = (uint16_t)(E.n01 >> 16);
    x.n2 = (uint16_t)(E.n2df & 0xffffu);
    x.group = G.gid;
    if (!over) {
      const size_t seg0 = ((size_t)blockIdx.x * kEpiWarps + kSegs * ev_warp) * (size_t)p.seg_cap;
      st_hit(p.seg_hits + seg0 + idx, rec);
      st_aux(p.seg_aux + seg0 + idx, x);
    } else if (gi < (unsigned long long)G.capacity) {
      st_hit(G.hits + gi, rec);
      st_aux(G.aux + gi, x);
    }
  }
  return n;
}

// ---- markers with up to five groups ---------------------------------------
// Hot test of a warp's kEpiSnpsM SNPs of a 32-SNP chunk: true when some pair may
// lie at or above the lower band edge, Q/h_df = sum_i c_i D_i^2 + c_4 (sum_i D_i)^2
// >= tau (1 - margin), two SNPs per packed instruction.
__device__ __forceinline__ bool hit_fast_m(const uint32_t (&d)[kMaxCodeM][kEpiSnpsM],
                                           const ChunkMetaM &m, int h, float ntlo) {
  const int jb = kEpiSnpsM * h;
  const uint64_t nt2 = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
  uint32_t acc = 0xffffffffu;
#pragma unroll
  for (int j = 0; j < kEpiSnpsM; j += 2) {
    uint64_t u[kMaxCodeM];
#pragma unroll
    for (int i = 0; i < kMaxCodeM; ++i) u[i] = pk2(d[i][j], d[i][j + 1]);
    const uint64_t s2 = fadd2(fadd2(u[0], u[1]), fadd2(u[2], u[3]));
    uint64_t q = nt2;
#pragma unroll
    for (int i = 0; i < kMaxCodeM; ++i) {
      const uint64_t c2 = *reinterpret_cast<const uint64_t *>(m.coef[i] + jb + j);
      q = ffma2(fmul2(c2, u[i]), u[i], q);
    }
    const uint64_t c4 = *reinterpret_cast<const uint64_t *>(m.coef[kMaxCodeM] + jb + j);
    q = ffma2(fmul2(c4, s2), s2, q);
    uint32_t qa, qb;
    upk2(q, qa, qb);
    acc &= qa & qb;
  }
  return (int)acc >= 0;
}

// FP64 decision for a pair inside the band: p < P_c from the exact sums.
__device__ __noinline__ bool decide64_m(const int *D, const ChunkMetaM &m, int jj, double cfac,
                                        double pthresh) {
  double Q = 0.0, S = 0.0;
  for (int i = 0; i < kMaxCodeM; ++i) {
    S += (double)D[i];
    if (m.n[i][jj] > 0) Q += (double)D[i] * (double)D[i] / (double)m.n[i][jj];
  }
  if (m.n[kMaxCodeM][jj] > 0) Q += S * S / (double)m.n[kMaxCodeM][jj];
  return chi2_tail64(cfac * Q, m.df[jj]) < pthresh;
}

// Rare path of a chunk of markers with up to five groups, called by the whole
// warp: classification of this lane's candidates and the warp's column-wise
// append into its staging segment (or the list), as hit_event does.  dv holds
// D_i of SNP j at dv[kEpiSnpsM * i + j] (i = 0..3).
__device__ __noinline__ unsigned int hit_event_m(const uint32_t *dv, bool mine, const ChunkMetaM &m,
                                                 int h, int trait, float ntlo, float nthi,
                                                 double cfac, const GroupDesc &g,
                                                 const ScanParams &p, unsigned int wn, int lane) {
  const int jb = kEpiSnpsM * h;
  uint32_t hm = 0;
  if (mine) {
    for (int j = 0; j < kEpiSnpsM; ++j) {
      const int jj = jb + j;
      if (m.snp[jj] < 0 || !in_cis_window(p, m.snp[jj], trait)) continue;
      float S = 0.f, q = 0.f;
      int D[kMaxCodeM];
      for (int i = 0; i < kMaxCodeM; ++i) {
        const float v = __uint_as_float(dv[kEpiSnpsM * i + j]);
        D[i] = (int)v;
        S += v;
        q = fmaf(m.coef[i][jj] * v, v, q);
      }
      q = fmaf(m.coef[kMaxCodeM][jj] * S, S, q);
      if (q + ntlo >= 0.f) {
        bool hit = q + nthi > 0.f;
        if (!hit) hit = decide64_m(D, m, jj, cfac, p.pthresh);
        if (hit) hm |= 1u << j;
      }
    }
  }
  const unsigned int total = __reduce_add_sync(0xffffffffu, (unsigned int)__popc(hm));
  if (total == 0u) return 0u;
  const unsigned int cap = (unsigned int)p.seg_cap;
  const unsigned int sbase = wn;
  const unsigned int over_from = sbase > cap ? sbase : cap;
  const unsigned int n_over = sbase + total > over_from ? sbase + total - over_from : 0u;
  unsigned long long gbase = 0;
  if (lane == 0 && n_over > 0) gbase = atomicAdd(g.counter, (unsigned long long)n_over);
  gbase = __shfl_sync(0xffffffffu, gbase, 0);
  const size_t seg0 = ((size_t)blockIdx.x * kEpiWarps + (threadIdx.x >> 5)) * cap;
  const uint32_t below_me = (1u << lane) - 1u;
  unsigned int run = sbase;
  uint32_t cols = __reduce_or_sync(0xffffffffu, hm);
  while (cols) {
    const int j = __ffs(cols) - 1;
    cols &= cols - 1u;
    const bool mine_j = (hm >> j) & 1u;
    const uint32_t bal = __ballot_sync(0xffffffffu, mine_j);
    if (mine_j) {
      const int jj = jb + j;
      const unsigned int idx = run + (unsigned int)__popc(bal & below_me);
      krux_hit r;
      r.trait = (uint32_t)trait;
      r.snp = (uint32_t)m.snp[jj];
      r.d0 = (int32_t)__uint_as_float(dv[j]);
      r.d1 = (int32_t)__uint_as_float(dv[kEpiSnpsM + j]);
      HitAux x;
      x.n0 = m.n[0][jj];
      x.n1 = m.n[1][jj];
      x.n2 = m.n[2][jj];
      x.group = (uint16_t)g.group_id;
      HitAux2 y;
      y.n3 = m.n[3][jj];
      y.n4 = m.n[4][jj];
      y.pad0_ = y.pad1_ = 0;
      y.d2 = (int32_t)__uint_as_float(dv[2 * kEpiSnpsM + j]);
      y.d3 = (int32_t)__uint_as_float(dv[3 * kEpiSnpsM + j]);
      if (idx < cap) {
        st_hit(p.seg_hits + seg0 + idx, r);
        st_aux(p.seg_aux + seg0 + idx, x);
        p.seg_aux2[seg0 + idx] = y;
      } else {
        const unsigned long long gi = gbase + (idx - over_from);
        if (gi < (unsigned long long)g.capacity) {
          st_hit(g.hits + gi, r);
          st_aux(g.aux + gi, x);
          g.aux2[gi] = y;
        }
      }
    }
    run += (unsigned int)__popc(bal);
  }
  return total;
}

// ---- the same markers in the plain form: weighted rows (PqCoefM), event warps ----
// True when some SNP's sum_i P_i^2 reaches -ntlo; x0 holds P_0, P_1 of 8 SNPs, x1 P_2,
// P_3.  Four FP32 operations per pair instead of eleven and five coefficients; with the
// event warps, paired chunks and one half-block live, 20,000 x 100,000 x 102: 2.07 ms in
// the general form, 1.08 in this one (8 N flop per pair: 78 % of the measured bf16 rate).
__device__ __forceinline__ bool hit_pq_m(const uint32_t (&x0)[2 * kEpiSnpsM],
                                         const uint32_t (&x1)[2 * kEpiSnpsM], float ntlo) {
  const uint64_t nt2 = pk2(__float_as_uint(ntlo), __float_as_uint(ntlo));
  uint32_t acc = 0xffffffffu;
#pragma unroll
  for (int j = 0; j < kEpiSnpsM; j += 2) {
    uint64_t q = nt2;
    const uint64_t a = pk2(x0[j], x0[j + 1]), b = pk2(x0[kEpiSnpsM + j], x0[kEpiSnpsM + j + 1]);
    const uint64_t c = pk2(x1[j], x1[j + 1]), d = pk2(x1[kEpiSnpsM + j], x1[kEpiSnpsM + j + 1]);
    q = ffma2(a, a, ffma2(b, b, ffma2(c, c, ffma2(d, d, q))));
    uint32_t x, y;
    upk2(q, x, y);
    acc &= x & y;
  }
  return (int)acc >= 0;
}

// One entry per trait lane that found a candidate among 8 SNPs (see ev_fill).
template <int kEntries>
__device__ __forceinline__ bool ev_submit_m(const EvRing<kEntries> &ev,
                                            const uint32_t (&x0)[2 * kEpiSnpsM],
                                            const uint32_t (&x1)[2 * kEpiSnpsM], bool need,
                                            const ChunkMetaM &m, int off, float tau,
                                            int trait, int group, const ScanParams &p,
                                            uint32_t abort_addr, int lane) {
  const int j = lane & (kEpiSnpsM - 1), jo = off + j;
  return ev_fill(
      ev, need, p, abort_addr, lane,
      [&](EvEntry &slot) {
        EvEntryM &E = reinterpret_cast<EvEntryM &>(slot);
#pragma unroll
        for (int i = 0; i < kEpiSnpsM; i += 4) {
          *reinterpret_cast<uint4 *>(E.P[0] + i) = make_uint4(x0[i], x0[i + 1], x0[i + 2], x0[i + 3]);
          *reinterpret_cast<uint4 *>(E.P[1] + i) = make_uint4(x0[8 + i], x0[9 + i], x0[10 + i], x0[11 + i]);
          *reinterpret_cast<uint4 *>(E.P[2] + i) = make_uint4(x1[i], x1[i + 1], x1[i + 2], x1[i + 3]);
          *reinterpret_cast<uint4 *>(E.P[3] + i) = make_uint4(x1[8 + i], x1[9 + i], x1[10 + i], x1[11 + i]);
        }
        E.tau = tau;
        E.trait = trait;
        E.group = group;
      },
      [&](EvEntry &slot) {
        EvEntryM &E = reinterpret_cast<EvEntryM &>(slot);
        if (lane & kEpiSnpsM) {  // the half-warp's upper lanes: what the records hold
#pragma unroll
          for (int i = 0; i <= kMaxCodeM; ++i) E.coef[i][j] = m.coef[i][jo];
          E.snp[j] = m.snp[jo];
        } else {
#pragma unroll
          for (int i = 0; i < kMaxCodeM; ++i) E.pq[i][j] = m.pq[i][jo];
          E.order[j] = m.order[jo];
          E.n01[j] = (uint32_t)m.n[0][jo] | ((uint32_t)m.n[1][jo] << 16);
          E.n23[j] = (uint32_t)m.n[2][jo] | ((uint32_t)m.n[3][jo] << 16);
          E.n4df[j] = (uint32_t)m.n[4][jo] | ((uint32_t)m.df[jo] << 16);
        }
      });
}

// An event warp's work on up to two such entries, one per half-warp (lanes 0..7 of a
// half take the entry's SNPs): the exact sums back from the accumulators, last row
// first, the test in FP32 (FP64 inside the band), and the records as in ev_process.
struct EvLaneM {
  float P[kMaxCodeM], coef[kMaxCodeM + 1], tau;
  uint32_t pq[kMaxCodeM], order, n01, n23, n4df;
  int snp, trait, group;
  __device__ __forceinline__ void load(const EvEntryM &E, int j) {
#pragma unroll
    for (int i = 0; i < kMaxCodeM; ++i) {
      P[i] = E.P[i][j];
      pq[i] = E.pq[i][j];
    }
#pragma unroll
    for (int i = 0; i <= kMaxCodeM; ++i) coef[i] = E.coef[i][j];
    order = E.order[j];
    snp = E.snp[j];
    n01 = E.n01[j];
    n23 = E.n23[j];
    n4df = E.n4df[j];
    tau = E.tau;
    trait = E.trait;
    group = E.group;
  }
};
__device__ __forceinline__ unsigned int ev_process_m(const EvLaneM &E, bool on, EvGroup &G,
                                                     const ScanParams &p, unsigned int wn, int lane,
                                                     int ev_warp) {
  const bool act = on && E.snp >= 0;
  float D[kMaxCodeM + 1];
#pragma unroll
  for (int i = 0; i <= kMaxCodeM; ++i) D[i] = 0.f;
  float later = 0.f;
#pragma unroll
  for (int i = kMaxCodeM - 1; i >= 0; --i) {
    const float a = __half2float(__ushort_as_half((unsigned short)(E.pq[i] & 0xffffu)));
    const float c = __half2float(__ushort_as_half((unsigned short)(E.pq[i] >> 16)));
    const float d = a > 0.f ? rintf(__fdividef(fmaf(-c, later, E.P[i]), a)) : 0.f;
    const uint32_t g = (E.order >> (3 * i)) & 7u;
#pragma unroll
    for (int k = 0; k <= kMaxCodeM; ++k)
      if (g == (uint32_t)k) D[k] = d;
    later += d;
  }
  const uint32_t gl = (E.order >> 12) & 7u;
#pragma unroll
  for (int k = 0; k <= kMaxCodeM; ++k)
    if (gl == (uint32_t)k) D[k] = -later;
  float s = 0.f;
#pragma unroll
  for (int k = 0; k <= kMaxCodeM; ++k) s = fmaf(E.coef[k] * D[k], D[k], s);
  bool cand = act && s + -E.tau * (1.f - p.margin) >= 0.f;
  if (cand) cand = in_cis_window(p, E.snp, E.trait);
  bool hit = cand && s + -E.tau * (1.f + p.margin) > 0.f;
  if (cand && !hit) {  // inside the band: FP64 (rare)
    const int n[kMaxCodeM + 1] = {(int)(E.n01 & 0xffffu), (int)(E.n01 >> 16), (int)(E.n23 & 0xffffu),
                                  (int)(E.n23 >> 16), (int)(E.n4df & 0xffffu)};
    double Q = 0.0;
    for (int k = 0; k <= kMaxCodeM; ++k)
      if (n[k] > 0) Q += (double)D[k] * (double)D[k] / (double)n[k];
    hit = chi2_tail64(p.groups[E.group].cfac[E.trait] * Q, (int)(E.n4df >> 16)) < p.pthresh;
  }
  const uint32_t bal = __ballot_sync(0xffffffffu, hit);
  const unsigned int n = (unsigned int)__popc(bal);
  if (n == 0u) return 0u;
  constexpr int kSegs = kEpiWarps / 2;
  const unsigned int cap = (unsigned int)(kSegs * p.seg_cap);
  const unsigned int idx = wn + (unsigned int)__popc(bal & ((1u << lane) - 1u));
  const bool over = hit && idx >= cap;
  const uint32_t obal = __ballot_sync(0xffffffffu, over);
  unsigned long long gi = 0;
  if (hit) ev_group(G, p, E.group);
  if (obal != 0u) {  // one reservation per half (the halves may belong to different lists)
    const uint32_t mine = obal & (0xffffu << (lane & 16));
    const int lead = mine != 0u ? __ffs((int)mine) - 1 : 0;
    if (over && lane == lead) gi = atomicAdd(G.counter, (unsigned long long)__popc(mine));
    gi = __shfl_sync(0xffffffffu, gi, lead) + (unsigned int)__popc(mine & ((1u << lane) - 1u));
  }
  if (hit) {
    krux_hit r;
    r.trait = (uint32_t)E.trait;
    r.snp = (uint32_t)E.snp;
    r.d0 = (int32_t)D[0];
    r.d1 = (int32_t)D[1];
    HitAux x;
    x.n0 = (uint16_t)(E.n01 & 0xffffu);
    x.n1 = (uint16_t)(E.n01 >> 16);
    x.n2 = (uint16_t)(E.n23 & 0xffffu);
    x.group = G.gid;
    HitAux2 y;
    y.n3 = (uint16_t)(E.n23 >> 16);
    y.n4 = (uint16_t)(E.n4df & 0xffffu);
    y.pad0_ = y.pad1_ = 0;
    y.d2 = (int32_t)D[2];
    y.d3 = (int32_t)D[3];
    if (!over) {
      const size_t at = ((size_t)blockIdx.x * kEpiWarps + kSegs * ev_warp) * (size_t)p.seg_cap + idx;
      st_hit(p.seg_hits + at, r);
      st_aux(p.seg_aux + at, x);
      p.seg_aux2[at] = y;
    } else if (gi < (unsigned long long)G.capacity) {
      st_hit(G.hits + gi, r);
      st_aux(G.aux + gi, x);
      G.aux2[gi] = y;
    }
  }
  return n;
}

// Hot filter bounds of one (permutation, trait): the running best -ln p turned
// into bounds on the form, |s| of df-1 SNPs and s of df-2 SNPs.
struct MinpState {
  float s1_lo, s2_lo;
};

// Bounds of the hot filter from the running best key: with key_lo = key (1 -
// margin), a df-2 SNP may beat it iff c2 s > key_lo, a df-1 SNP iff
// -ln erfc(sqrt(c1 |s| / 2)) > key_lo, i.e. c1 |s| > 2 erfcinv(exp(-key_lo))^2 (no
// transcendental left per chunk).  Past p ~ 1e-35 a lower bound of the inverse is
// used (the filter stays conservative).
__device__ __noinline__ MinpState minp_bounds(float key, float c1, float c2, float margin) {
  const float inf = __int_as_float(0x7f800000);
  const float klo = key * (1.f - margin);
  MinpState ms;
  ms.s2_lo = c2 > 0.f ? klo / c2 : inf;
  float h1 = 0.f;
  if (klo > 80.f) {
    h1 = 2.f * (klo - 0.5f * logf(3.14159265f * klo) - 1.f);
  } else if (klo > 0.f) {
    const float x = erfcinvf(expf(-klo));
    h1 = 2.f * x * x * (1.f - 1e-5f);
  }
  ms.s1_lo = c1 > 0.f ? h1 / c1 : inf;
  return ms;
}

// Largest df-2 form value (smax >= 0) and most negative df-1 form value
// (smin <= 0) of a permuted chunk half.
__device__ __forceinline__ void minp_range(const uint32_t (&d0)[kEpiSnps],
                                           const uint32_t (&d1)[kEpiSnps], const ChunkMeta &m,
                                           int h, float &smax_out, float &smin_out) {
  const uint64_t *al = reinterpret_cast<const uint64_t *>(m.alpha + kEpiSnps * h);
  const uint64_t *be = reinterpret_cast<const uint64_t *>(m.beta + kEpiSnps * h);
  const uint64_t *ga = reinterpret_cast<const uint64_t *>(m.gamma + kEpiSnps * h);
  float smax = 0.f, smin = 0.f;
#pragma unroll
  for (int j = 0; j < kEpiSnps / 2; j += 2) {
    const ulonglong2 A = *reinterpret_cast<const ulonglong2 *>(al + j);
    const ulonglong2 B = *reinterpret_cast<const ulonglong2 *>(be + j);
    const ulonglong2 G = *reinterpret_cast<const ulonglong2 *>(ga + j);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int jj = 2 * (j + t);
      const uint64_t u2 = pk2(d0[jj], d0[jj + 1]);
      const uint64_t v2 = pk2(d1[jj], d1[jj + 1]);
      const uint64_t a2 = t ? A.y : A.x, b2 = t ? B.y : B.x, g2 = t ? G.y : G.x;
      const uint64_t w2 = ffma2(b2, v2, u2);
      const uint64_t e2 = fmul2(g2, v2);
      const uint64_t s2 = ffma2(fmul2(a2, w2), w2, fmul2(e2, v2));
      uint32_t sa, sb;
      upk2(s2, sa, sb);
      smax = fmax3(smax, __uint_as_float(sa), __uint_as_float(sb));
      smin = fmin3(smin, __uint_as_float(sa), __uint_as_float(sb));
    }
  }
  smax_out = smax;
  smin_out = smin;
}

// Seed bound of a step: FP32 -ln p of the largest values seen (ms holds them in
// seed mode), less twice the recheck margin so that it stays below the FP64 key of
// the pair that attains it.
__device__ __noinline__ double minp_seed_key(MinpState ms, float c1, float c2, float margin) {
  const float k = fmaxf(ms.s2_lo * c2, key1f(ms.s1_lo * c1));
  return (double)(k * (1.f - 2.f * margin));
}

// Class leader of one (permutation, trait) in a step: the pair with the largest
// form value among its df-1 SNPs (value |s|) or among its df-2 SNPs (value s).
// Within a class -ln p grows with the value (-ln p = c2 s for df 2, a function of
// c1 |s| that increases for df 1), so tracking the value needs no transcendental;
// the FP64 key is computed once, at the end of the step, or earlier on a near tie.
struct MinpCand {
  float s;        // FP32 value (0: no leader yet)
  float u, v;     // centred sums
  int n01;        // n0 | n1 << 16
  int n2df;       // n2 | df << 16
  double k64;     // FP64 -ln p once computed, else -1
};

// Leader state of one (permutation, trait) in a step.  Lives in local memory:
// touched only by the rare paths and at step boundaries.
struct MinpLead {
  MinpCand cls[2];  // [0]: df-1 SNPs, [1]: df-2 SNPs
  double exact;     // best FP64 key of the pairs decided exactly (traits with NaN), else -1
  double start;     // the global value at step start
  float c1, c2;     // H = c1 |s| for df-1 SNPs; -ln p = c2 s for df-2 SNPs
};

// FP64 -ln p of a pair from its exact sums (0 for degenerate pairs).
__device__ __noinline__ double lead_key64(float u, float v, int n0, int n1, int n2, int df,
                                          double cfac) {
  if (df <= 0 || !(cfac > 0.0)) return 0.0;
  return key64_of(kw_H64((int)u, (int)v, n0, n1, n2, cfac), df);
}

__device__ __forceinline__ double cand_key64(MinpCand &C, double cfac) {
  if (C.k64 < 0.0)
    C.k64 = lead_key64(C.u, C.v, C.n01 & 0xffff, C.n01 >> 16, C.n2df & 0xffff, C.n2df >> 16, cfac);
  return C.k64;
}

// Rare path of a permuted chunk half (trait without NaN): every SNP past the hot
// filter's bounds is offered to its class leader.  A clearly larger value (by more
// than the recheck margin) takes the lead without FP64; a near tie is decided on
// the FP64 keys.  The bound of the class then rises to the leader's value less the
// margin, so that only pairs that may beat the leader pass again.  With the FDR
// histogram on, every pair at or above the band gets its FP64 key and, if p < P_c,
// a count in row `row` of the histogram.
__device__ __noinline__ MinpState minp_event(const uint32_t *dv, const ChunkMeta &m, int h,
                                             double cfac, MinpLead *L, MinpState ms, float tau_lo,
                                             const ScanParams &p, int row) {
  const int jb = kEpiSnps * h;
  const float *al = m.alpha + jb, *be = m.beta + jb, *ga = m.gamma + jb;
  const float tie = p.margin;
  for (int j = 0; j < kEpiSnps; ++j) {
    if (m.snp[jb + j] < 0) continue;
    const float u = __uint_as_float(dv[j]), v = __uint_as_float(dv[kEpiSnps + j]);
    const float sv = kw_s(u, v, al[j], be[j], ga[j]);
    const bool lead = sv > ms.s2_lo || -sv > ms.s1_lo;
    const bool band = p.fdr_hist != nullptr && fabsf(sv) >= tau_lo;
    if (!lead && !band) continue;
    const int n0 = m.n[0][jb + j], n1 = m.n[1][jb + j], n2 = m.n[2][jb + j], df = m.df[jb + j];
    double key = -1.0;
    if (band) {
      key = lead_key64(u, v, n0, n1, n2, df, cfac);
      if (key > -log(p.pthresh))
        atomicAdd(p.fdr_hist + (int64_t)row * p.fdr_bins +
                      fdr_bin(key, p.fdr_l0, p.fdr_w, p.fdr_bins),
                  1ull);
    }
    if (!lead) continue;
    const int k = sv > 0.f ? 1 : 0;
    const float a = fabsf(sv);
    MinpCand &C = L->cls[k];
    bool take = a > C.s * (1.f + tie);
    // near tie with the leader: FP64, unless the pair repeats the leader's sums and
    // group sizes (copies of one SNP are common inside LD blocks) and so its key
    const bool same = u == C.u && v == C.v && (n0 | (n1 << 16)) == C.n01 &&
                      (n2 | (df << 16)) == C.n2df;
    if (!take && !same && a >= C.s * (1.f - tie)) {
      if (key < 0.0) key = lead_key64(u, v, n0, n1, n2, df, cfac);
      take = key > cand_key64(C, cfac);
    }
    if (take) {
      C.s = fmaxf(a, C.s);
      C.u = u;
      C.v = v;
      C.n01 = n0 | (n1 << 16);
      C.n2df = n2 | (df << 16);
      C.k64 = key;
    }
    if (k) ms.s2_lo = fmaxf(ms.s2_lo, C.s * (1.f - tie));
    else ms.s1_lo = fmaxf(ms.s1_lo, C.s * (1.f - tie));
  }
  return ms;
}

// Rare path of a permuted chunk half for a trait with NaN: the group sizes of each
// pair come from the genotype codes of its present samples, every pair is decided
// on its FP64 key (max into L->exact) and, with the FDR histogram on, counted.
__device__ __noinline__ void minp_event_nan(const uint32_t *dv, const ChunkMeta &m,
                                            const uint64_t *codes, int h, double cfac,
                                            int nan_cnt, const uint16_t *nan_idx, MinpLead *L,
                                            const ScanParams &p, int row) {
  const int jb = kEpiSnps * h;
  for (int j = 0; j < kEpiSnps; ++j) {
    if (m.snp[jb + j] < 0) continue;
    const float u = __uint_as_float(dv[j]), v = __uint_as_float(dv[kEpiSnps + j]);
    int n0, n1, n2;
    pair_counts(nan_cnt, nan_idx, m, codes, jb + j, n0, n1, n2);
    const double key = lead_key64(u, v, n0, n1, n2, df_of(n0, n1, n2), cfac);
    if (p.fdr_hist != nullptr && key > -log(p.pthresh))
      atomicAdd(p.fdr_hist + (int64_t)row * p.fdr_bins + fdr_bin(key, p.fdr_l0, p.fdr_w, p.fdr_bins),
                1ull);
    L->exact = fmax(L->exact, key);
  }
}

// End of a step: the best FP64 key of the step's leaders, if it beats the global
// value read at step start.
__device__ __noinline__ double minp_step_best(MinpLead *L, double cfac) {
  double best = L->exact;
  for (int k = 0; k < 2; ++k)
    if (L->cls[k].s > 0.f) best = fmax(best, cand_key64(L->cls[k], cfac));
  return best;
}

// Kernel forms.  General ones: markers with up to five genotype groups (kFormMulti: 32-SNP
// chunks, ChunkMetaM), permutation batches (kFormPerm: groups with a min-p key), and
// everything else (kFormNan: exact group sizes of traits with NaN in the hot test); the
// others are plain (fast_form).  The producer's and the MMA warp's code is shared, but for the
// pairs of CTAs' own issuer.  Separate forms keep the state of one out of the registers of
// the others.
enum ScanForm {
  kFormScan = 0,
  kFormMulti = 1,
  kFormPerm = 2,
  kFormNan = 3,
  kFormScanPerm = 4,
  kFormScanNan = 5,
  kFormScanSeed = 6,
  kFormScanPair = 7,
  kFormScanMulti = 8,
  kFormScanDense = 9
};
// the plain scan form, its two passes over permutation batches (the largest values
// first, then the pairs against them), its variant for expression with NaN, the one
// over pairs of CTAs, the one for markers with up to five groups, and the dense one,
// which writes every pair's rank sums (indicator rows) for the FP64 pass after it
constexpr bool fast_form(int f) {
  return f == kFormScan || f == kFormScanPerm || f == kFormScanNan || f == kFormScanSeed ||
         f == kFormScanPair || f == kFormScanMulti || f == kFormScanDense;
}
// The plain form over clusters of two CTAs, for sample counts whose chunk pair leaves
// one CTA's shared memory too little room for rank tiles in flight: the pair's tensor
// cores contract 256 traits with a chunk pair, each CTA holding 128 traits' rank tiles
// and one chunk, so a rank tile is still read once per 128 SNPs.  An MMA is issued by
// the first CTA (cta_group::2) and fills both CTAs' accumulators, 128 traits x 128 SNPs
// in each, which the epilogue reads as in the plain form.  The second CTA's chunk is
// announced by its otherwise idle MMA warp; its rank tiles count on the first CTA's
// barriers themselves.  15,000 x 200,000: N = 256
// 2.00 ms with a pair in one CTA -> 1.75, N = 300 3.06 -> 2.01; N = 400 and 500, which do
// not fit one CTA, 9.02 -> 2.66 and 10.35 -> 3.42 ms (93 % of the measured bf16 rate)
// against the general form.
constexpr bool pair_form(int f) { return f == kFormScanPair; }

// Warp roles of a kernel form: the epilogue warps first, then the producer and
// the MMA issuer (in the plain forms two event warps after them).
template <int kForm>
struct ScanRoles {
  static constexpr int kEpi = fast_form(kForm) ? kFastEpiWarps : kEpiWarps;
  static constexpr int kProducer = kEpi;
  static constexpr int kMma = kEpi + 1;
  static constexpr int kThreads = fast_form(kForm) ? kFastThreads : kScanThreads;
};

template <int kForm>
__global__ void __launch_bounds__(ScanRoles<kForm>::kThreads, 1)
    krux_scan_kernel(const __grid_constant__ ScanParams p) {
  using R = ScanRoles<kForm>;
  extern __shared__ uint8_t smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t *sbase = smem_raw + (base - raw);
  const uint32_t a_tile_bytes = (uint32_t)p.a_tile_bytes;
  const uint32_t sA = base;
  const uint32_t sB = base + (uint32_t)p.nA * a_tile_bytes;
  constexpr uint32_t kMeta = fast_form(kForm) ? sizeof(ChunkMeta) : kMetaGeneral;
  uint8_t *smeta = sbase + (size_t)p.nA * a_tile_bytes + (size_t)p.b_region;
  const auto meta_of = [&](int c) -> const ChunkMeta & {
    return *reinterpret_cast<const ChunkMeta *>(smeta + (uint32_t)c * kMeta);
  };
  uint8_t *scodes = smeta + (uint32_t)p.nc * kMeta;
  const uint32_t codes_stride = (uint32_t)p.kpad * 16u;
  uint8_t *stc = scodes + (size_t)p.nc * codes_stride;  // trait-constant ring
  // permutation form: per trait row, the min-p filter bounds of the current step
  // shared by the four warps that cover the row ((step tag << 32) | float bits;
  // df-1 bounds, then df-2 bounds)
  unsigned long long *sbound =
      reinterpret_cast<unsigned long long *>(stc + (size_t)kTcDepth * kTcBytes);
  // (the plain forms have neither the ring nor these bounds)
  uint64_t *bars = fast_form(kForm) ? reinterpret_cast<uint64_t *>(stc)
                                    : reinterpret_cast<uint64_t *>(sbound + 2 * kTileM);
  const uint32_t bar0 = smem_u32(bars);
  const int nA = p.nA, nc = p.nc;
  const int n_items = p.n_items_dev ? *p.n_items_dev : p.n_items;
  // barrier addresses
  auto a_full = [&](int s) { return bar0 + 8u * (uint32_t)s; };
  auto a_empty = [&](int s) { return bar0 + 8u * (uint32_t)(nA + s); };
  auto b_full = [&](int c) { return bar0 + 8u * (uint32_t)(2 * nA + c); };
  auto b_empty = [&](int c) { return bar0 + 8u * (uint32_t)(2 * nA + nc + c); };
  auto t_full = [&](int s) { return bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + s); };
  auto t_empty = [&](int s) { return bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + kTmemSlots + s); };
  const uint32_t drain = bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + 2 * kTmemSlots);
  auto tc_full = [&](int e) { return bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + 2 * kTmemSlots + 1 + e); };
  auto tc_empty = [&](int e) {
    return bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + 2 * kTmemSlots + 1 + kTcDepth + e);
  };
  auto it_full = [&](int e) {
    return bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + 2 * kTmemSlots + 1 + 2 * kTcDepth + e);
  };
  auto it_empty = [&](int e) {
    return bar0 + 8u * (uint32_t)(2 * nA + 2 * nc + 2 * kTmemSlots + 1 + 2 * kTcDepth + kItemDepth + e);
  };
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(bars + 2 * nA + 2 * nc + 2 * kTmemSlots + 1 +
                                                       2 * kTcDepth + 2 * kItemDepth);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_holder + 1);
  // The work item ring: the producer takes the CTA's next item (from the launch's
  // counter when there is one, so that CTAs whose items hold many hits, or short
  // ones, take fewer or more of them) and the other roles follow through it.
  volatile int *item_ring = reinterpret_cast<volatile int *>(tmem_holder + 4);
  // Plain forms: rank tiles the producer has asked for, the event warps' sign that the
  // CTA moves on while no entry comes (a launch may run for any time without one).
  volatile uint32_t *progress = tmem_holder + 2;
  struct ItemPos {
    uint32_t e = 0, phase = 0;
  };
  auto item_next = [&](ItemPos &q) {
    if (++q.e == (uint32_t)kItemDepth) {
      q.e = 0;
      q.phase ^= 1u;
    }
  };
  // plain scan form: the ring of hit-event buffers after everything else
  constexpr int kEv = pair_form(kForm) ? kEvEntriesPair : kEvEntries;
  EvRing<kEv> ev;
  {
    uint8_t *evr = reinterpret_cast<uint8_t *>(
        (reinterpret_cast<uintptr_t>(tmem_holder) + 32u + 127u) & ~(uintptr_t)127u);
    ev.ent = reinterpret_cast<EvEntry *>(evr);
    ev.bar0 = smem_u32(evr + kEv * sizeof(EvEntry));
    ev.released = reinterpret_cast<unsigned int *>(evr + kEv * sizeof(EvEntry) + kEv * 8);
    ev.word = reinterpret_cast<unsigned long long *>(evr + kEv * sizeof(EvEntry) +
                                                     kEv * 8 + kEv * 4);
  }

  constexpr bool kPair = pair_form(kForm);
  const uint32_t rank = kPair ? cluster_rank() : 0u;  // 0: issues the MMAs
  // Pairs of CTAs: what a CTA has asked for when its roles have ended, own and (after the
  // first cluster barrier of the shutdown) the other's, in the place of the trait
  // constants' barriers.
  struct PairNote {
    uint32_t loads;        // rank tiles (K blocks of them) asked for, in the order both CTAs share
    uint32_t stage_atoms;  // atoms of the last one in each stage, 4 bits each
    uint32_t chunks;       // genotype chunks asked for
    uint32_t announced;    // of the second CTA's chunks, those announced to the first
    uint32_t aborted;
  };
  static_assert(2 * sizeof(PairNote) <= 2 * kTcDepth * sizeof(uint64_t), "notes of a pair");
  volatile PairNote *note =
      reinterpret_cast<volatile PairNote *>(bars + 2 * nA + 2 * nc + 2 * kTmemSlots + 1);
  if (threadIdx.x == 0) {
    for (int s = 0; s < nA; ++s) {
      mbar_init(a_full(s), 1);
      mbar_init(a_empty(s), 1);
    }
    for (int c = 0; c < nc; ++c) {
      // (a pair's first CTA also counts the second's word that its chunk is there)
      mbar_init(b_full(c), kPair && rank == 0u ? 2 : 1);
      mbar_init(b_empty(c), 1 + R::kEpi);
    }
    for (int s = 0; s < kTmemSlots; ++s) {
      mbar_init(t_full(s), 1);
      mbar_init(t_empty(s), kPair ? 2 * R::kEpi : R::kEpi);
    }
    mbar_init(drain, 1);
    for (int e = 0; e < kTcDepth && !fast_form(kForm); ++e) {
      mbar_init(tc_full(e), 1);
      mbar_init(tc_empty(e), R::kEpi);
    }
    for (int e = 0; e < kItemDepth; ++e) {
      mbar_init(it_full(e), 1);
      mbar_init(it_empty(e), 1 + R::kEpi);
    }
    *abort_flag = 0;
    *progress = 0u;
    if constexpr (fast_form(kForm)) {
      for (int e = 0; e < kEv; ++e) {
        mbar_init(ev.full(e), 1);
        ev.released[e] = 0u;
      }
      *ev.word = 0ull;
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if constexpr (kPair) cluster_sync();  // both CTAs run and their barriers exist
  if (warp == R::kMma) {
    if constexpr (kPair) {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                       smem_u32(tmem_holder))
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(
                       smem_u32(tmem_holder))
                   : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
  }
  if constexpr (!fast_form(kForm))
    for (int i = threadIdx.x; i < 2 * kTileM; i += blockDim.x) sbound[i] = 0ull;
  tc_fence_before();
  __syncthreads();
  if constexpr (kPair) cluster_sync();  // both allocations stand before the first MMA
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  const WaitCtl wc{abort_flag, p.status, p.timeout_cycles};
  // plain scan form: the registers of the producer warpgroup (warps 16-19) go to
  // the epilogue warps; each role's code sits under its own setmaxnreg

  if (warp == R::kProducer) {
    if constexpr (fast_form(kForm))
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFastRegsLow) : "memory");
    if (lane == 0) {
      uint32_t a_stage = 0, a_phase = 0, b_bits = 0;
      uint32_t a_used = 0, a_last = 0, b_used = 0, b_last = 0;
      uint32_t tc_e = 0, tc_phase = 0, tc_used = 0, tc_last = 0;
      uint32_t tiles = 0;  // rank tiles asked for
      uint32_t stage_atoms = 0, chunks = 0;  // (PairNote)
      ItemPos ip;
      // (the two CTAs of a pair take the same items, in fixed turns)
      for (int it = kPair ? (int)(blockIdx.x >> 1) : (int)blockIdx.x;;
           it = kPair    ? it + (int)(gridDim.x >> 1)
                : p.next ? (int)(gridDim.x + atomicAdd(p.next, 1u))
                         : it + (int)gridDim.x) {
        if (!wait_bar(it_empty(ip.e), ip.phase ^ 1u, wc, 18)) goto producer_done;
        item_ring[ip.e] = it;
        mbar_arrive(it_full(ip.e));  // (release: the item is visible to who waits for it)
        item_next(ip);
        if (it >= n_items) break;
        const WorkItem w = p.items[it];
        const GroupDesc *g = p.groups + w.group;
        if constexpr (!fast_form(kForm) || kPair) {
          prefetch_map(&g->tmA);
          prefetch_map(&g->tmB);
        }
        const int ncg = g->nc;
        const int nc_item = min(ncg, g->nchunks - w.btile * ncg);
        const uint32_t b_stride = (uint32_t)g->b_stride;
        const uint32_t abytes = atom_bytes(p.layout);
        const int ak = (int)atom_k(p.layout);
        const uint32_t b_tx = (uint32_t)g->n_atoms * abytes;
        const uint32_t codes_bytes = g->codes ? (uint32_t)g->codes_k * 16u : 0u;
        if constexpr (kPair) {
          // this CTA's chunk of the pair, and both chunks' metadata
          const uint32_t ph = b_bits & 1u;
          if (!wait_bar(b_empty(0), ph ^ 1u, wc, 1)) goto producer_done;
          const int chunk = w.btile * 2;
          const bool own = (int)rank < nc_item;
          mbar_expect_tx(b_full(0), (own ? b_tx : 0u) + (uint32_t)nc_item * kMeta);
          if (own)
            bulk_load(sB, g->Bt + (int64_t)(chunk + (int)rank) * kChunkRows * g->Np, b_tx, b_full(0));
          bulk_load(smem_u32(smeta), g->meta + chunk, (uint32_t)nc_item * kMeta, b_full(0));
          ++chunks;
          b_bits ^= 1u;
        }
        for (int c = 0; c < nc_item && !kPair; ++c) {
          const uint32_t ph = (b_bits >> c) & 1u;
          if (!wait_bar(b_empty(c), ph ^ 1u, wc, 1)) goto producer_done;
          const int chunk = w.btile * ncg + c;
          mbar_expect_tx(b_full(c), b_tx + kMeta + codes_bytes);
          // paired groups interleave chunks 2j, 2j+1 per K atom: [atom][chunk of pair][128 rows]
          const uint32_t bbase = g->pair ? sB + (uint32_t)(c >> 1) * 2u * b_stride + (uint32_t)(c & 1) * abytes
                                         : sB + (uint32_t)c * b_stride;
          const uint32_t astep = g->pair ? 2u * abytes : abytes;
          if constexpr (fast_form(kForm)) {
            const __half *src = g->Bt + (int64_t)chunk * kChunkRows * g->Np;
            for (int a = 0; a < g->n_atoms; ++a)
              bulk_load(bbase + (uint32_t)a * astep, src + a * 2048, abytes, b_full(c));
          } else {
            for (int a = 0; a < g->n_atoms; ++a)
              tma_load_2d(bbase + (uint32_t)a * astep, &g->tmB, a * ak, g->b_row0 + chunk * kChunkRows,
                          b_full(c));
          }
          bulk_load(smem_u32(smeta) + (uint32_t)c * kMeta, g->meta + chunk, kMeta, b_full(c));
          if (codes_bytes)
            bulk_load(smem_u32(scodes + (size_t)c * codes_stride), g->codes + (size_t)chunk * g->codes_k * 2,
                      codes_bytes, b_full(c));
          b_used |= 1u << c;
          b_last = (b_last & ~(1u << c)) | (ph << c);
          b_bits ^= 1u << c;
        }
        const int atoms_per_block = p.ka / ak;
        if constexpr (fast_form(kForm)) {
          // the rank tiles lie in step order; the descriptor's fields stay in registers
          // (every barrier operation and copy would have them read again)
          const int n_atoms = g->n_atoms;
          const __half *tile = g->At + (int64_t)w.step_begin * (kTileM * g->Np);
          if constexpr (kPair) {
            // a pair's step is two tiles, one per CTA (an odd last one: the same twice);
            // both CTAs' copies count on the first CTA's barrier, where the MMAs wait
            const int last_tile = g->n_ttiles - 1, tile_rows = 32 * n_atoms;
            for (int step = w.step_begin; step < w.step_end; ++step) {
              const int y = min(2 * step + (int)rank, last_tile) * tile_rows;
              for (int a0 = 0; a0 < n_atoms; a0 += atoms_per_block) {
                if (!wait_bar(a_empty(a_stage), a_phase ^ 1u, wc, 2)) goto producer_done;
                const int na = min(atoms_per_block, n_atoms - a0);
                if (rank == 0u) mbar_expect_tx(a_full(a_stage), (uint32_t)na * 8192u);
                tma_load_pair(sA + (uint32_t)a_stage * a_tile_bytes,
                              na == atoms_per_block ? &g->tmA : &g->tmB, 0, y + 32 * a0,
                              peer_addr(a_full(a_stage), 0u));
                stage_atoms = (stage_atoms & ~(15u << (4 * a_stage))) | ((uint32_t)na << (4 * a_stage));
                *progress = ++tiles;
                if (++a_stage == (uint32_t)nA) {
                  a_stage = 0;
                  a_phase ^= 1u;
                }
              }
            }
            continue;
          }
          for (int step = w.step_begin; step < w.step_end; ++step) {
            for (int a0 = 0; a0 < n_atoms; a0 += atoms_per_block) {
              if (!wait_bar(a_empty(a_stage), a_phase ^ 1u, wc, 2)) goto producer_done;
              const int na = min(atoms_per_block, n_atoms - a0);
              mbar_expect_tx(a_full(a_stage), (uint32_t)na * 4096u);
              bulk_load(sA + (uint32_t)a_stage * a_tile_bytes, tile + a0 * 2048, (uint32_t)na * 4096u,
                        a_full(a_stage));
              *progress = ++tiles;
              a_used |= 1u << a_stage;
              a_last = (a_last & ~(1u << a_stage)) | (a_phase << a_stage);
              if (++a_stage == (uint32_t)nA) {
                a_stage = 0;
                a_phase ^= 1u;
              }
            }
            tile += n_atoms * 2048;
          }
          continue;
        }
        for (int step = w.step_begin; step < w.step_end; ++step) {
          const int ag = step / g->n_ttiles, tt = step - ag * g->n_ttiles;
          const int row0 = g->a_row0 + ag * g->rows_per_agroup + tt * kTileM;
          // the rank tile of this step, in K blocks of p.ka samples
          for (int kb = 0; kb < g->nkb; ++kb) {
            if (!wait_bar(a_empty(a_stage), a_phase ^ 1u, wc, 2)) goto producer_done;
            const int a0 = kb * atoms_per_block;
            const int na = min(atoms_per_block, g->n_atoms - a0);
            mbar_expect_tx(a_full(a_stage), (uint32_t)na * abytes);
            for (int a = 0; a < na; ++a)
              tma_load_2d(sA + (uint32_t)a_stage * a_tile_bytes + (uint32_t)a * abytes, &g->tmA,
                          (a0 + a) * ak, row0, a_full(a_stage));
            a_used |= 1u << a_stage;
            a_last = (a_last & ~(1u << a_stage)) | (a_phase << a_stage);
            if (++a_stage == (uint32_t)nA) {
              a_stage = 0;
              a_phase ^= 1u;
            }
          }
          // this step's per-trait constants into the ring (padded to whole tiles)
          if constexpr (!fast_form(kForm)) {
            if (!wait_bar(tc_empty(tc_e), tc_phase ^ 1u, wc, 8)) goto producer_done;
            const bool with_key = g->minp_key != nullptr && ag > 0;
            const uint32_t tx = 512u + 1024u + (g->nan_cnt ? 256u : 0u) + (with_key ? 1024u : 0u);
            const uint32_t dst = smem_u32(stc + (size_t)tc_e * kTcBytes);
            const int64_t r0 = (int64_t)tt * kTileM;
            mbar_expect_tx(tc_full(tc_e), tx);
            bulk_load(dst, g->tau + r0, 512u, tc_full(tc_e));
            bulk_load(dst + 512u, g->cfac + r0, 1024u, tc_full(tc_e));
            if (with_key) {
              const int64_t kr = (int64_t)(ag - 1) * g->rows_per_agroup + r0;
              bulk_load(dst + 1536u, g->minp_key + kr, 1024u, tc_full(tc_e));
            }
            if (g->nan_cnt) bulk_load(dst + 2560u, g->nan_cnt + r0, 256u, tc_full(tc_e));
            tc_used |= 1u << tc_e;
            tc_last = (tc_last & ~(1u << tc_e)) | (tc_phase << tc_e);
            if (++tc_e == (uint32_t)kTcDepth) {
              tc_e = 0;
              tc_phase ^= 1u;
            }
          }
        }
        // The general forms' steps differ in length by up to a factor of ten (traits with many
        // NaN samples): the next item is taken when this one's first chunk is free, which its
        // copies wait for anyway, and not by a CTA that still has most of this one to do
        if (p.next && !wait_bar(b_empty(0), (b_bits & 1u) ^ 1u, wc, 1)) goto producer_done;
      }
    producer_done:
      // let every copy this thread issued land before the CTA can exit (a pair of CTAs
      // counts them together and drains them after both producers have ended, see below)
      if constexpr (kPair) {
        note[0].loads = tiles;
        note[0].stage_atoms = stage_atoms;
        note[0].chunks = chunks;
      }
      for (int s = 0; s < nA; ++s)
        if ((a_used >> s) & 1u) wait_drain(a_full(s), (a_last >> s) & 1u, p.status, 10);
      for (int c = 0; c < nc; ++c)
        if ((b_used >> c) & 1u) wait_drain(b_full(c), (b_last >> c) & 1u, p.status, 11);
      for (int e = 0; e < kTcDepth; ++e)
        if ((tc_used >> e) & 1u) wait_drain(tc_full(e), (tc_last >> e) & 1u, p.status, 13);
    }
    __syncwarp();
  } else if (warp == R::kMma && kPair) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFastRegsLow) : "memory");
    if (lane == 0) {
      uint32_t a_stage = 0, a_phase = 0, b_bits = 0, ps = 0, ps_phase = 0;
      uint32_t announced = 0;
      ItemPos ip;
      while (true) {
        if (!wait_bar(it_full(ip.e), ip.phase, wc, 19)) goto pair_done;
        const int it = item_ring[ip.e];
        mbar_arrive(it_empty(ip.e));
        item_next(ip);
        if (it >= n_items) break;
        const WorkItem w = p.items[it];
        const GroupDesc *g = p.groups + w.group;
        const int ksteps = g->Np / 16;
        const int kpb = p.ka / 16;
        if (rank != 0u) {
          // announce this CTA's chunk to the issuing one
          if (!wait_bar(b_full(0), b_bits, wc, 4)) goto pair_done;
          mbar_arrive_cluster(peer_addr(b_full(0), 0u));
          ++announced;
        } else {
          if (!wait_bar_cluster(b_full(0), b_bits, wc, 4)) goto pair_done;
          for (int step = w.step_begin; step < w.step_end; ++step) {
            if (!wait_bar_cluster(t_empty(ps), ps_phase ^ 1u, wc, 5)) goto pair_done;
            const uint32_t d_tmem = tmem_base + ps * 256u;
            uint64_t db = umma_desc(sB, 1);
            for (int k = 0; k < ksteps;) {
              if (!wait_bar_cluster(a_full(a_stage), a_phase, wc, 3)) goto pair_done;
              tc_fence_after();
              uint64_t da = umma_desc(sA + a_stage * a_tile_bytes, 1);
              for (const int k1 = min(k + kpb, ksteps); k < k1; ++k) {
                tc_mma_pair(d_tmem, da, db, k > 0 ? 1u : 0u);
                da += 4096u >> 4;
                db += 4096u >> 4;
              }
              tc_commit_pair(a_empty(a_stage));
              if (++a_stage == (uint32_t)nA) {
                a_stage = 0;
                a_phase ^= 1u;
              }
            }
            tc_commit_pair(t_full(ps));
            ps ^= 1u;
            if (ps == 0u) ps_phase ^= 1u;
          }
          tc_commit_pair(b_empty(0));
        }
        b_bits ^= 1u;
      }
    pair_done:
      note[0].announced = announced;
      if (rank == 0u) {
        // all issued MMAs must finish before TMEM is released (and their commits have
        // arrived at the second CTA before it ends: it waits for this one below)
        tc_commit_pair(drain);
        wait_drain(drain, 0, p.status, 12);
      }
    }
    __syncwarp();
  } else if (warp == R::kMma && fast_form(kForm)) {
    // MMA issuer of the plain scan form: one N = 256 MMA chain per chunk pair (N =
    // 128 for an odd last chunk) into accumulator pair `ps` (TMEM columns ps *
    // 256 ..), released by the 16 epilogue warps as soon as they have loaded it
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFastRegsLow) : "memory");
    if (lane == 0) {
      uint32_t a_stage = 0, a_phase = 0, b_bits = 0, ps = 0, ps_phase = 0;
      ItemPos ip;
      while (true) {
        if (!wait_bar(it_full(ip.e), ip.phase, wc, 19)) goto fast_mma_done;
        const int it = item_ring[ip.e];
        mbar_arrive(it_empty(ip.e));
        item_next(ip);
        if (it >= n_items) break;
        const WorkItem w = p.items[it];
        const GroupDesc *g = p.groups + w.group;
        const int ncg = g->nc;
        const int nc_item = min(ncg, g->nchunks - w.btile * ncg);
        const uint32_t b_stride = (uint32_t)g->b_stride;
        const int ksteps = g->Np / 16;
        if (g->nkb > 1) {
          // one resident pair, its K in blocks of p.ka samples per rank stage
          const bool two = nc_item > 1;
          const uint32_t idesc = two ? kIdesc256 : kIdesc;
          const int kpb = p.ka / 16;
          if (!wait_bar(b_full(0), b_bits & 1u, wc, 4)) goto fast_mma_done;
          if (two && !wait_bar(b_full(1), (b_bits >> 1) & 1u, wc, 4)) goto fast_mma_done;
          for (int step = w.step_begin; step < w.step_end; ++step) {
            if (!wait_bar(t_empty(ps), ps_phase ^ 1u, wc, 5)) goto fast_mma_done;
            const uint32_t d_tmem = tmem_base + ps * 256u;
            uint64_t db = umma_desc(sB, 1);
            for (int k = 0; k < ksteps;) {
              if (!wait_bar(a_full(a_stage), a_phase, wc, 3)) goto fast_mma_done;
              tc_fence_after();
              uint64_t da = umma_desc(sA + a_stage * a_tile_bytes, 1);
              for (const int k1 = min(k + kpb, ksteps); k < k1; ++k) {
                tc_mma(d_tmem, da, db, idesc, k > 0 ? 1u : 0u);
                da += 4096u >> 4;
                db += 8192u >> 4;
              }
              tc_commit(a_empty(a_stage));
              if (++a_stage == (uint32_t)nA) {
                a_stage = 0;
                a_phase ^= 1u;
              }
            }
            tc_commit(t_full(ps));
            ps ^= 1u;
            if (ps == 0u) ps_phase ^= 1u;
          }
          for (int c = 0; c < nc_item; ++c) {
            tc_commit(b_empty(c));
            b_bits ^= 1u << c;
          }
          continue;
        }
        for (int step = w.step_begin; step < w.step_end; ++step) {
          if (!wait_bar(a_full(a_stage), a_phase, wc, 3)) goto fast_mma_done;
          tc_fence_after();
          const uint32_t a_tile = sA + a_stage * a_tile_bytes;
          for (int c = 0; c < nc_item; c += 2) {
            const bool two = c + 1 < nc_item;
            if (step == w.step_begin) {
              if (!wait_bar(b_full(c), (b_bits >> c) & 1u, wc, 4)) goto fast_mma_done;
              if (two && !wait_bar(b_full(c + 1), (b_bits >> (c + 1)) & 1u, wc, 4)) goto fast_mma_done;
            }
            if (!wait_bar(t_empty(ps), ps_phase ^ 1u, wc, 5)) goto fast_mma_done;
            tc_fence_after();
            // pair layout: [K atom][chunk of the pair][128 rows of 32 B]; a K step
            // moves the start address field only (it never carries)
            const uint32_t b_tile = sB + (uint32_t)(c >> 1) * 2u * b_stride;
            uint64_t da = umma_desc(a_tile, 1), db = umma_desc(b_tile, 1);
            const uint32_t d_tmem = tmem_base + ps * 256u;
            const uint32_t idesc = two ? kIdesc256 : kIdesc;
            tc_mma(d_tmem, da, db, idesc, 0u);
            for (int k = 1; k < ksteps; ++k) {
              da += 4096u >> 4;
              db += 8192u >> 4;
              tc_mma(d_tmem, da, db, idesc, 1u);
            }
            tc_commit(t_full(ps));
            ps ^= 1u;
            if (ps == 0u) ps_phase ^= 1u;
          }
          tc_commit(a_empty(a_stage));
          if (++a_stage == (uint32_t)nA) {
            a_stage = 0;
            a_phase ^= 1u;
          }
        }
        for (int c = 0; c < nc_item; ++c) {
          tc_commit(b_empty(c));
          b_bits ^= 1u << c;
        }
      }
    fast_mma_done:
      // all issued MMAs must finish before TMEM is released
      tc_commit(drain);
      wait_drain(drain, 0, p.status, 12);
    }
    __syncwarp();
  } else if (warp == R::kMma) {
    if (lane == 0) {
      uint32_t a_stage = 0, a_phase = 0, b_bits = 0, slot = 0, slot_phase = 0;
      ItemPos ip;
      while (true) {
        if (!wait_bar(it_full(ip.e), ip.phase, wc, 19)) goto mma_done;
        const int it = item_ring[ip.e];
        mbar_arrive(it_empty(ip.e));
        item_next(ip);
        if (it >= n_items) break;
        const WorkItem w = p.items[it];
        const GroupDesc *g = p.groups + w.group;
        const int ncg = g->nc;
        const int nc_item = min(ncg, g->nchunks - w.btile * ncg);
        const uint32_t b_stride = (uint32_t)g->b_stride;
        const int ksteps = g->Np / 16;
        const int kpb = p.ka / 16;  // K steps per block
        for (int step = w.step_begin; step < w.step_end; ++step) {
          if (g->pair && (slot & 1u)) {
            // paired accumulators start on an even slot: retire this one unused
            if (!wait_bar(t_empty(slot), slot_phase ^ 1u, wc, 14)) goto mma_done;
            tc_fence_after();
            tc_commit(t_full(slot));
            if (++slot == (uint32_t)kTmemSlots) {
              slot = 0;
              slot_phase ^= 1u;
            }
          }
          for (int kb = 0; kb < g->nkb; ++kb) {
            if (!wait_bar(a_full(a_stage), a_phase, wc, 3)) goto mma_done;
            tc_fence_after();
            const int k0 = kb * kpb;
            const int nk = min(kpb, ksteps - k0);
            const uint32_t a_tile = sA + a_stage * a_tile_bytes;
            for (int c = 0; c < nc_item;) {
              const bool two = g->pair && c + 1 < nc_item;
              uint32_t sc = slot + (uint32_t)c, ph = slot_phase;
              if (sc >= (uint32_t)kTmemSlots) {
                sc -= kTmemSlots;
                ph ^= 1u;
              }
              if (kb == 0) {
                for (int j = 0; j < (two ? 2 : 1); ++j) {
                  const uint32_t sj = sc + (uint32_t)j;  // sc is even when two: sj stays in range
                  if (step == w.step_begin) {
                    if (!wait_bar(b_full(c + j), (b_bits >> (c + j)) & 1u, wc, 4)) goto mma_done;
                  }
                  if (!wait_bar(t_empty(sj), ph ^ 1u, wc, 5)) goto mma_done;
                }
                tc_fence_after();
              }
              const uint32_t d_tmem = tmem_base + sc * 128u;
              // descriptors are built once per chunk and K block; a K step only moves
              // the start address field (bits 0-13, address >> 4), which never carries
              if (p.layout) {
                const uint32_t b_tile = g->pair ? sB + (uint32_t)(c >> 1) * 2u * b_stride
                                                : sB + (uint32_t)c * b_stride;
                const uint32_t bstep = g->pair ? 8192u : 4096u;
                const uint32_t idesc = two ? kIdesc256 : kIdesc;
                uint64_t da = umma_desc(a_tile, 1), db = umma_desc(b_tile + (uint32_t)k0 * bstep, 1);
                tc_mma(d_tmem, da, db, idesc, kb > 0 ? 1u : 0u);
                for (int k = 1; k < nk; ++k) {
                  da += 4096u >> 4;
                  db += bstep >> 4;
                  tc_mma(d_tmem, da, db, idesc, 1u);
                }
              } else {
                const uint32_t b_tile = sB + (uint32_t)c * b_stride;
                const uint64_t da = umma_desc(a_tile, 0), db = umma_desc(b_tile, 0);
                for (int k = 0; k < nk; ++k) {
                  const uint64_t oa = (uint64_t)(kstep_off(0, k) >> 4);
                  const uint64_t ob = (uint64_t)(kstep_off(0, k0 + k) >> 4);
                  tc_mma(d_tmem, da + oa, db + ob, kIdesc, (kb > 0 || k > 0) ? 1u : 0u);
                }
              }
              if (kb == g->nkb - 1) {
                tc_commit(t_full(sc));
                if (two) tc_commit(t_full(sc + 1u));
              }
              c += two ? 2 : 1;
            }
            tc_commit(a_empty(a_stage));
            if (++a_stage == (uint32_t)nA) {
              a_stage = 0;
              a_phase ^= 1u;
            }
          }
          slot += (uint32_t)nc_item;
          if (slot >= (uint32_t)kTmemSlots) {
            slot -= kTmemSlots;
            slot_phase ^= 1u;
          }
        }
        for (int c = 0; c < nc_item; ++c) {
          tc_commit(b_empty(c));
          b_bits ^= 1u << c;
        }
      }
    mma_done:
      // all issued MMAs must finish before TMEM is released
      tc_commit(drain);
      wait_drain(drain, 0, p.status, 12);
    }
    __syncwarp();
  } else if constexpr (fast_form(kForm)) {
    // epilogue warps of the plain scan form: warp 4k + q owns lane quarter q of
    // kFastSnps SNPs of one chunk of every accumulator pair; it loads and tests them in
    // two halves, releases the pair after the second load, and hands a half-block with a
    // candidate to the event warps
    if (warp >= R::kEpi) {  // the two event warps of the producer warpgroup
      asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kFastRegsLow) : "memory");
      const int e = warp - (R::kMma + 1);
      unsigned int wn = 0;  // hits this event warp has appended to its staging region
      unsigned int mcn = 0;  // permuted pairs it has passed on to the deferred FP64 pass
      EvGroup G;
      // half h of event warp e takes the tickets 2 e + h, + 4, ...
      const int half = lane >> 4;
      unsigned long long t = (unsigned long long)(2 * e + half);
      bool idle = false;
      long long t0 = 0;
      uint32_t seen = 0;
      // (the seed pass and the dense form submit nothing)
      while (kForm != kFormScanSeed && kForm != kFormScanDense) {
        const int b = (int)(t % kEv);
        // the halves' first lanes look whether their ticket is filled, or no more can come
        int got = 0;
        if ((lane & 15) == 0) {
          if (mbar_test(ev.full(b), (uint32_t)((t / kEv) & 1ull))) {
            got = 1;
          } else {
            const unsigned long long wv = *reinterpret_cast<volatile unsigned long long *>(ev.word);
            if (*abort_flag || ((wv >> 40) >= (unsigned long long)kFastEpiWarps && t >= (wv & kEvTicketMask)))
              got = 2;
          }
        }
        got = __shfl_sync(0xffffffffu, got, lane & 16);
        const bool on = got == 1;
        if (!__any_sync(0xffffffffu, on)) {
          if (__all_sync(0xffffffffu, got == 2)) break;
          // idle for as long as the CTA works on items without a candidate.  Every other
          // wait of the CTA gives up by itself, so the end of the epilogue warps always
          // comes; this limit, counted from the producer's last rank tile, is a last resort
          const long long now = clock64();
          const uint32_t at = *progress;
          if (!idle || at != seen) t0 = now;
          idle = true;
          seen = at;
          if (__any_sync(0xffffffffu, ((now - t0) >> 1) > p.timeout_cycles)) {
            if (lane == 0) {
              *abort_flag = 1;
              atomicOr(p.status, kDevTimeout);
              atomicMax(p.status + 1, 17u);
            }
            break;
          }
          __nanosleep(400);
          continue;
        }
        idle = false;
        __syncwarp();
        auto release = [&]() {  // this use of the entry is finished
          __syncwarp();
          if (on && (lane & 15) == 0) {
            __threadfence_block();
            atomicAdd(ev.released + b, 1u);
          }
        };
        if constexpr (kForm == kFormScanMulti) {
          EvLaneM E;
          E.load(reinterpret_cast<const EvEntryM &>(ev.ent[b]), lane & (kEpiSnpsM - 1));
          release();
          wn += ev_process_m(E, on && (lane & 15) < kEpiSnpsM, G, p, wn, lane, e);
          if (on) t += 4;
          continue;
        }
        EvLane E;
        E.load(ev.ent[b], lane & (kEvSnps - 1));
        release();
        wn += ev_process<kForm == kFormScanPerm ? kEvPerm : (kForm == kFormScanNan ? kEvNan : kEvPlain)>(
            E, on, G, p, wn, lane, e, mcn);
        if (on) t += 4;
      }
      if constexpr (kForm == kFormScanPerm)
        if (lane == 0 && p.mc_cnt != nullptr) p.mc_cnt[blockIdx.x * 2 + e] = min(mcn, (unsigned int)p.mc_cap);
      if (lane == 0 && p.seg_cap > 0) {  // this event warp's staging segments
        constexpr int kSegs = kEpiWarps / 2;
        const unsigned int cap = (unsigned int)p.seg_cap;
        for (int sgi = 0; sgi < kSegs; ++sgi) {
          const unsigned int lo = cap * (unsigned int)sgi;
          p.seg_cnt[blockIdx.x * kEpiWarps + kSegs * e + sgi] = wn > lo ? min(wn - lo, cap) : 0u;
        }
      }
    } else {
      asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFastRegsHigh) : "memory");
      constexpr int kPerChunk = kChunkSnps / kFastSnps;  // warps per chunk and lane quarter
      const int q = warp & 3, k = warp >> 2;
      const int h = k / kPerChunk;                     // chunk of the pair
      constexpr bool kMultiF = kForm == kFormScanMulti;
      const int off = (kMultiF ? kFastSnps / 2 : kFastSnps) * (k % kPerChunk);  // first SNP within the chunk
      const int row = 32 * q + lane;
      const uint32_t abort_addr = smem_u32(const_cast<const int *>(abort_flag));
      const uint32_t lane_cols =
          tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(128 * h + off);
      uint32_t ps = 0, ps_phase = 0, b_bits = 0;
      constexpr int kH = kFastSnps / 2;
      // permutation batches: per class (df 1, df 2) a pair may pass when its value
      // exceeds the largest decided one of the lane's trait, staged for the step, less
      // the margin (at most the band's lower edge while FDR counts are on).  The
      // unpermuted group tests both classes against tau.
      constexpr bool kTwo = kForm == kFormScanPerm;
      constexpr bool kNan = kForm == kFormScanNan;
      constexpr bool kSeed = kForm == kFormScanSeed;
      constexpr float kBoundMin = 1e-30f, kBoundMax = 1e30f;
      constexpr int kMany = 8;
      // expression with NaN: the bound of this lane's trait is coefficient set
      // nset - 1 of the chunk's block (0: the chunk metadata's exact coefficients;
      // -1: more NaN samples than any set covers, every pair goes to the exact
      // test).  The warp first tests all its lanes with the loosest set any of them
      // needs (wset: one address for the whole warp), and only when some lane
      // passes, and the lanes' sets differ (mixed), each lane again with its own set
      // (lanes reading different addresses cost several shared-memory passes per
      // load).  One register: nset + 1 in bits 0-3, wset in bits 4-7, mixed bit 8,
      // the trait's NaN count from bit 9.
      int nsw = 1;
      // the hot test's bounds of the step: -tau (1 - margin), or the classes' bounds
      float ntlo = 0.f, bnd1 = 0.f, bnd2 = 0.f;
      float tau_s = 0.f;  // the lane's tau
      // seed pass: this lane's largest df-2 value and df-1 |value| in the step and
      // the 16-SNP blocks (positions in the group's SNP order) that hold them
      float smax = 0.f, smin = 0.f;
      int pos2 = 0, pos1 = 0;
      // What only a candidate needs (tau, the factor of H, decided values and their
      // identities) is read from global memory when there is one: the hot loop holds
      // the bounds and the accumulators alone (with tau, the decided values and their
      // identities in registers, and the seed pass in the same kernel, the permutation
      // form spilled 268 bytes in the loop: 75.7 ms per call of 16 x 20,000 x 200,000
      // against 52.8).
      auto test = [&](const uint32_t(&x0)[kH], const uint32_t(&x1)[kH], const ChunkMeta &mc, int o,
                      const uint8_t *blk, uint32_t cls) -> bool {
        if constexpr (kTwo) {
          if (cls == 0u || cls == 0xffffffffu) return hit_pq<kH>(x0, x1, cls ? -bnd2 : -bnd1);
          return hit_pq2<kH>(x0, x1, mc.sgn + o, bnd1, bnd2);
        } else if constexpr (kNan) {
          const int wset = (nsw >> 4) & 15, nset = (nsw & 15) - 1;
          if (wset == 0) return hit_pq<kH>(x0, x1, ntlo);
          const float *cw = coef_set(blk, wset - 1)->alpha;
          bool need = hit_fast_wc<kH>(x0, x1, cw, cw + kChunkSnps, cw + 2 * kChunkSnps, o, ntlo);
          if (((nsw >> 8) & 1) && __any_sync(0xffffffffu, need)) {
            const float *cf = coef_set(blk, max(nset, 1) - 1)->alpha;
            const bool own = nset > 0 ? hit_fast_wc<kH>(x0, x1, cf, cf + kChunkSnps, cf + 2 * kChunkSnps,
                                                        o, ntlo)
                                      : hit_pq<kH>(x0, x1, ntlo);
            need = own && need;
          }
          return need;
        } else {
          return hit_pq<kH>(x0, x1, ntlo);
        }
      };
      // a permuted trait's two class words, (value bits << 32) | identity (seed pass:
      // position) of the largest value so far, and the values alone; other CTAs raise
      // them during the launch
      auto class_words = [&](const GroupDesc &g, int ag, int trait) -> uint4 {
        const unsigned long long *b = kSeed ? g.minp_seed : g.minp_bound;
        return __ldcg(reinterpret_cast<const uint4 *>(b) + (int64_t)(ag - 1) * g.rows_per_agroup + trait);
      };
      auto class_values = [&](const GroupDesc &g, int ag, int trait, float &v1, float &v2) {
        if (ag == 0) return;
        const uint4 bb = class_words(g, ag, trait);
        v1 = __uint_as_float(bb.y);
        v2 = __uint_as_float(bb.w);
      };
      // a permuted block past the hot test: whether the lane has a pair that still
      // needs the event warps (past its class's bound but not an exact copy of the
      // class's decided pair -- copies are common inside LD blocks -- or in the FDR band)
      auto minp_filter = [&](const uint32_t(&x0)[kH], const uint32_t(&x1)[kH], const ChunkMeta &mc,
                             int o, float tau, float mx1, float mx2, uint32_t id1,
                             uint32_t id2) -> bool {
        const float tlo = p.fdr_hist != nullptr ? tau * (1.f - p.margin) : kBoundMax;
        bool any = false;
        for (int j = 0; j < kH; ++j) {
          // P^2 + Q^2 is never below |s|: most pairs stop here
          const float pj = __uint_as_float(x0[j]), qj = __uint_as_float(x1[j]);
          const float top = fmaf(pj, pj, qj * qj) * 1.00001f;
          const bool two = mc.sgn[o + j] > 0.f;
          const float bnd = two ? bnd2 : bnd1;
          if (!(top > bnd || top >= tlo)) continue;
          float u, v;
          pq_sums(pj, qj, mc.pq0[o + j], mc.pq1[o + j], u, v);
          const float sv = fabsf(kw_s(u, v, mc.alpha[o + j], mc.beta[o + j], mc.gamma[o + j]));
          const bool past = sv > bnd && !(sv == (two ? mx2 : mx1) &&
                                          pair_id((int)u, (int)v) == (two ? id2 : id1));
          any = any || past || sv >= tlo;
        }
        return any;
      };
      // a half-block with a candidate: to the event warps; false if a wait gave up
      auto hand_over = [&](const uint32_t(&x0)[kH], const uint32_t(&x1)[kH], bool need,
                           const ChunkMeta &mc, int o, const GroupDesc &g, int ag, int tt,
                           int group) -> bool {
        const int trait = tt * kTileM + row;
        const float tau = tau_s;
        bool real = need;
        float mx1 = 0.f, mx2 = 0.f;
        uint32_t id1 = 0u, id2 = 0u;
        if constexpr (kTwo) {
          // (with the FDR histogram on, nearly every candidate is a pair of its band: all go
          // to the event warps, which read the class words themselves.  Read and filtered
          // here, a round trip to L2 with the accumulator slot held, 16 x 20,000 x 200,000
          // took 44.1 ms, now 40.5.  Not so where more than kMany traits of the warp have one: those
          // are values that repeat, as in the only block of a small batch, and most are copies of
          // the decided pair: 3 x 128 x 16 x 300 286 -> 255 us)
          if (ag > 0 && (p.fdr_hist == nullptr || __popc(__ballot_sync(0xffffffffu, need)) > kMany)) {
            const uint4 bb = class_words(g, ag, trait);
            mx1 = fmaxf(__uint_as_float(bb.y), kBoundMin);
            id1 = bb.x;
            mx2 = fmaxf(__uint_as_float(bb.w), kBoundMin);
            id2 = bb.z;
            if (need) real = minp_filter(x0, x1, mc, o, tau, mx1, mx2, id1, id2);
            if (!__any_sync(0xffffffffu, real)) return true;
          }
        }
        return ev_submit(ev, x0, x1, real, mc, o, tau, trait, group, ag, mx1, mx2, id1, id2,
                         kNan ? nsw >> 9 : 0, p, abort_addr, lane);
      };
      // one accumulator pair: wait for it, load and test this warp's two halves one
      // after the other (release after the second load) and hand any candidate
      // half-block to the event warps; false if a wait gave up.  Only one half's
      // accumulators are live: with the second half's load overlapping the first
      // half's test the loop held 64 of them and spilled (N = 128, 15,000 x 200,000:
      // 0.898 against 0.875 ms; the permutation form's main launch of 16 x 20,000 x
      // 200,000: 30.9 against 25.1 ms); the four warps of a scheduler cover each
      // other's loads.  The two halves are spelt out (20,000 x 200,000: N = 24 845 -> 753 us,
      // 48 864 -> 829, 102 1067 -> 1052, 256 2295 -> 2201; 176 to 224, bound by the tensor
      // cores, 0.6 to 1 % longer; 16 permutations 45.3 -> 44.2 ms), but for the NaN form,
      // whose two tests make the code long (missing values 1.15 -> 1.18 ms).
      auto pair_slot = [&](uint32_t ps, uint32_t phase, const ChunkMeta &mc, int c, int chunk0,
                           const GroupDesc &g, int ag, int tt, int group) -> bool {
        if (!wait_warp(t_full(ps), phase, p, abort_addr, 7)) return false;
        tc_fence_after();
        uint32_t x0[kH], x1[kH];
        const uint32_t taddr = lane_cols + ps * 256u;
#pragma unroll(kNan ? 1 : 2)
        for (int half = 0; half < 2; ++half) {
          if constexpr (kMultiF) {  // 8 SNPs, P_i of SNP j in column 32 i + j of the chunk
            tmem_ld_rows(taddr + (uint32_t)(kEpiSnpsM * half), x0, x1);
          } else {
            tmem_ld_half(taddr + (uint32_t)(kH * half), x0, x1);
          }
          const int o = off + kH * half;
          // permutation batches: the classes of the block's tested SNPs (all ones: df 2, zero:
          // df 1, else both; in the order of launch_class_order nearly every block is of one class)
          uint32_t cls = 0u;
          if constexpr (kTwo || kSeed) {
            const float sg = mc.sgn[o + (lane & (kH - 1))];
            const bool one = __any_sync(0xffffffffu, sg < 0.f), two = __any_sync(0xffffffffu, sg > 0.f);
            cls = !one ? 0xffffffffu : (two ? 1u : 0u);
          }
          tmem_wait_ld();
          if (half) {
            tc_fence_before();
            __syncwarp();
            if constexpr (kPair) mbar_arrive_cluster_lane0(peer_addr(t_empty(ps), 0u), lane);
            else mbar_arrive_lane0(t_empty(ps), lane);
          }
          if constexpr (kSeed) {
            const int pos = (chunk0 + c) * kChunkSnps + o;
            float hi = 0.f, lo = 0.f;
            if (cls == 0u || cls == 0xffffffffu) {
              const float top = top_pq<kH>(x0, x1);
              if (cls) hi = top;
              else lo = -top;
            } else {
              range_pq<kH>(x0, x1, mc.sgn + o, hi, lo);
            }
            if (hi > smax) { smax = hi; pos2 = pos; }
            if (lo < smin) { smin = lo; pos1 = pos; }
          } else {
            const uint8_t *blk = kNan ? scodes + (size_t)c * codes_stride : nullptr;
            if constexpr (kForm == kFormScanDense) {
              const int trait = tt * kTileM + row;
              const int snp0 = mc.snp[o];
              const bool in_row = __all_sync(0xffffffffu, snp0 >= 0 && mc.snp[o + (lane & (kH - 1))] ==
                                                                           snp0 + (lane & (kH - 1)));
              if (trait < g.T) {
                int2 *out = reinterpret_cast<int2 *>(g.dense_H + (int64_t)trait * g.dense_ld) - g.dense_snp0;
                const auto pair_of = [&](int j) {
                  return make_int2(__float2int_rn(__uint_as_float(x0[j])), __float2int_rn(__uint_as_float(x1[j])));
                };
                // 16 columns in a row: two per store, from the first or the second one on as
                // the row's alignment has it.  Bound by its stores: 1,000 x 20,003 x 102
                // with one column each 231 us, now 109
                if (in_row) {
                  int2 *at = out + snp0;
                  const bool odd = ((uintptr_t)at & 15u) != 0;
                  int2 v[kH];
#pragma unroll
                  for (int j = 0; j < kH; ++j) v[j] = pair_of(j);
                  if (odd) {
                    at[0] = v[0];
                    at[kH - 1] = v[kH - 1];
                  }
#pragma unroll
                  for (int j = 0; j < kH; j += 2) {
                    const int2 a = odd ? v[j + 1] : v[j], b = odd ? v[(j + 2) % kH] : v[j + 1];
                    if (j + 2 < kH || !odd)
                      *reinterpret_cast<int4 *>(at + j + (odd ? 1 : 0)) = make_int4(a.x, a.y, b.x, b.y);
                  }
                } else {
#pragma unroll
                  for (int j = 0; j < kH; ++j) {
                    const int snp = mc.snp[o + j];
                    if (snp >= 0) out[snp] = pair_of(j);
                  }
                }
              }
              continue;
            }
            if constexpr (kMultiF) {
              const bool need = hit_pq_m(x0, x1, ntlo);
              if (__any_sync(0xffffffffu, need)) {
                const int trait = tt * kTileM + row;
                if (!ev_submit_m(ev, x0, x1, need, reinterpret_cast<const ChunkMetaM &>(mc),
                                 off + kEpiSnpsM * half, tau_s, trait, group, p,
                                 abort_addr, lane))
                  return false;
              }
              continue;
            }
            const bool need = test(x0, x1, mc, o, blk, cls);
            if (__any_sync(0xffffffffu, need) && !hand_over(x0, x1, need, mc, o, g, ag, tt, group))
              return false;
          }
        }
        return true;
      };
      ItemPos ip;
      while (true) {
        if (!wait_warp(it_full(ip.e), ip.phase, p, abort_addr, 20)) goto epi_done_scan;
        const int it = item_ring[ip.e];
        __syncwarp();
        mbar_arrive_lane0(it_empty(ip.e), lane);
        item_next(ip);
        if (it >= n_items) break;
        const WorkItem w = p.items[it];
        const GroupDesc &g = p.groups[w.group];
        const int g_nc = g.nc, g_ntt = g.n_ttiles;
        const int nc_item = min(g_nc, g.nchunks - w.btile * g_nc);
        const int chunk0 = w.btile * g_nc;  // the work item's first chunk in the group
        const float *g_tau = g.tau + row;
        const uint16_t *g_nan = kNan ? g.nan_cnt : nullptr;
        // the step's rank-matrix group (> 0: a permutation) and its trait tile (of a
        // pair's two tiles, this CTA's)
        int ag = kPair ? 0 : w.step_begin / g_ntt;
        int tt = kPair ? 2 * w.step_begin + (int)rank : w.step_begin - ag * g_ntt;
        // this warp's chunks of the B tile (h and 2 + h) must have landed
        if constexpr (kPair) {
          if (!wait_warp(b_full(0), b_bits & 1u, p, abort_addr, 6)) goto epi_done_scan;
        } else {
          bool ok = true;
          for (int c = h; c < nc_item; c += 2) ok = ok && wait_bar_p(b_full(c), (b_bits >> c) & 1u, p, abort_addr, 6);
          if (!__all_sync(0xffffffffu, ok)) goto epi_done_scan;
        }
        // the constants of the lane's trait, one step ahead
        const float kNever = __int_as_float(0x7f800000);
        float tau_n = kPair && tt >= g_ntt ? kNever : g_tau[tt * kTileM];
        uint32_t nan_n = 0u;
        float v1_n = 0.f, v2_n = 0.f;
        if constexpr (kNan)
          if (g_nan) nan_n = g_nan[tt * kTileM + row];
        if constexpr (kTwo || kSeed) class_values(g, ag, tt * kTileM + row, v1_n, v2_n);
        for (int step = w.step_begin; step < w.step_end; ++step) {
          const float tau = tau_n, v1 = v1_n, v2 = v2_n;
          const int ag0 = ag, tt0 = tt;
          if constexpr (kPair) {
            tt += 2;  // (past the last tile, an odd one's second half: never a candidate)
            tau_n = tt < g_ntt ? g_tau[tt * kTileM] : kNever;
          } else {
            if (++tt == g_ntt) {
              tt = 0;
              ++ag;
            }
            tau_n = g_tau[tt * kTileM];  // (past the last step: a row that exists, unused)
          }
          ntlo = -tau * (1.f - p.margin);
          tau_s = tau;
          if constexpr (kNan) {
            const int nan_c = (int)nan_n;
            if (g_nan) nan_n = g_nan[tt * kTileM + row];
            const int nset = nan_c == 0 ? 0 : (nan_c <= kNanCMax ? nan_set_of(nan_c) + 1 : -1);
            const int wset = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(nset, 0));
            const bool mixed = __any_sync(0xffffffffu, nset >= 0 && nset != wset);
            nsw = (nset + 1) | (wset << 4) | (mixed ? 256 : 0) | (nan_c << 9);
            // (a trait beyond the last set: +inf lets every pair through)
            if (nset < 0 && tau < kBoundMax) ntlo = __int_as_float(0x7f800000);
          }
          if constexpr (kTwo || kSeed)
            if (step + 1 < w.step_end) class_values(g, ag, tt * kTileM + row, v1_n, v2_n);
          if constexpr (kTwo) {
            // unpermuted group: both classes against tau (less the margin); a
            // permuted one: the classes' largest decided values
            const float keep = 1.f - p.margin;
            if (ag0 > 0) {
              const float cap = p.fdr_hist != nullptr ? fminf(tau * keep, kBoundMax) : kBoundMax;
              bnd1 = fminf(fmaxf(v1, kBoundMin) * keep, cap);
              bnd2 = fminf(fmaxf(v2, kBoundMin) * keep, cap);
            } else {
              bnd1 = fminf(tau * keep, kBoundMax);
              bnd2 = bnd1;
            }
          }
          smax = 0.f;
          smin = 0.f;
          pos2 = 0;
          pos1 = 0;
          for (int c = h; c - h < nc_item; c += 2) {
            if (c < nc_item) {
              if (!pair_slot(ps, ps_phase, meta_of(c), c, chunk0, g, ag0, tt0, w.group))
                goto epi_done_scan;
            } else {  // an odd last chunk leaves warps 8-15 idle: release only
              if (!wait_warp(t_full(ps), ps_phase, p, abort_addr, 7)) goto epi_done_scan;
              tc_fence_after();
              tc_fence_before();
              __syncwarp();
              if constexpr (kPair) mbar_arrive_cluster_lane0(peer_addr(t_empty(ps), 0u), lane);
              else mbar_arrive_lane0(t_empty(ps), lane);
            }
            ps ^= 1u;
            if (ps == 0u) ps_phase ^= 1u;
          }
          if constexpr (kSeed) {
            // the step's largest values and their blocks (the largest over all steps
            // is decided exactly after the launch), written only past the record read
            // before the step
            const int trait = tt0 * kTileM + row;
            if (ag0 > 0 && trait < g.T) {
              unsigned long long *rp =
                  g.minp_seed + 2 * ((int64_t)(ag0 - 1) * g.rows_per_agroup + trait);
              if (-smin > v1)
                atomicMax(rp, ((unsigned long long)__float_as_uint(-smin) << 32) | (uint32_t)(pos1 + 1));
              if (smax > v2)
                atomicMax(rp + 1, ((unsigned long long)__float_as_uint(smax) << 32) | (uint32_t)(pos2 + 1));
            }
          }
        }
        // the chunks' metadata is no longer needed
        __syncwarp();
        if (lane == 0)
          for (int c = 0; c < (kPair ? 1 : nc_item); ++c) mbar_arrive(b_empty(c));
        for (int c = 0; c < (kPair ? 1 : nc_item); ++c) b_bits ^= 1u << c;
      }
    epi_done_scan:
      tc_fence_before();
      __syncwarp();
      if (lane == 0) atomicAdd(ev.word, 1ull << 40);  // no more events from this warp
    }
  } else {
    // epilogue warps
    const int q = warp & 3, h = warp >> 2;  // lane quarter, SNP group of the chunk
    uint32_t slot = 0, slot_phase = 0, b_bits = 0, tc_e = 0, tc_phase = 0;
    unsigned int wn = 0;  // hits this warp has appended to its staging segment
    uint32_t step_tag = 0;  // steps begun by this warp (the same count in every epilogue warp)
    ItemPos ip;
    while (true) {
      if (!__all_sync(0xffffffffu, wait_bar(it_full(ip.e), ip.phase, wc, 20))) goto epi_done;
      const int it = item_ring[ip.e];
      __syncwarp();
      if (lane == 0) mbar_arrive(it_empty(ip.e));
      item_next(ip);
      if (it >= n_items) break;
      const WorkItem w = p.items[it];
      const GroupDesc &g = p.groups[w.group];
      const int nc_item = min(g.nc, g.nchunks - w.btile * g.nc);
      const int g_ntt = g.n_ttiles, g_T = g.T, g_N = g.N;
      const bool g_has_nan = g.nan_cnt != nullptr;
      for (int step = w.step_begin; step < w.step_end; ++step) {
        const int ag = step / g_ntt, tt = step - ag * g_ntt;
        if (g.pair && (slot & 1u)) {
          // the MMA warp retired this slot unused (paired accumulators start even)
          if (!__all_sync(0xffffffffu, wait_bar(t_full(slot), slot_phase, wc, 15))) goto epi_done;
          __syncwarp();
          if (lane == 0) mbar_arrive(t_empty(slot));
          if (++slot == (uint32_t)kTmemSlots) {
            slot = 0;
            slot_phase ^= 1u;
          }
        }
        if constexpr (kForm == kFormPerm) ++step_tag;
        // this step's trait constants, staged by the producer
        if (!__all_sync(0xffffffffu, wait_bar(tc_full(tc_e), tc_phase, wc, 9))) goto epi_done;
        const uint8_t *tcp = stc + (size_t)tc_e * kTcBytes;
        const int row = 32 * q + lane;
        EpiTrait et;
        et.trait = tt * kTileM + row;
        et.valid = et.trait < g_T;
        const float tau = reinterpret_cast<const float *>(tcp)[row];
        et.ntlo = -tau * (1.f - p.margin);
        et.nthi = -tau * (1.f + p.margin);
        et.cfac = reinterpret_cast<const double *>(tcp + 512)[row];
        et.nan_cnt = g_has_nan ? (int)reinterpret_cast<const uint16_t *>(tcp + 2560u)[row] : 0;
        et.nan_idx = g_has_nan && et.valid
                         ? g.nan_idx + ag * g.nan_ag_stride + (int64_t)et.trait * g_N
                         : nullptr;
        const bool minp_mode = kForm == kFormPerm && g.minp_key != nullptr && ag > 0;
        const bool seed_pass = kForm == kFormPerm && p.seed_bound != 0;
        // traits with NaN (form kFormNan): the hot test's bounds on sum_i D_i^2 / n_i'
        float nan_q1 = 0.f, nan_q2 = 0.f;
        if (kForm == kFormNan) {
          const float cf = (float)et.cfac;
          nan_q1 = cf > 0.f ? p.h1 * (1.f - p.margin) / cf : __int_as_float(0x7f800000);
          nan_q2 = cf > 0.f ? p.h2 * (1.f - p.margin) / cf : __int_as_float(0x7f800000);
        }
        // with the FDR histogram on, permuted pairs at or above the band are counted
        const float fdr_tau_lo = p.fdr_hist != nullptr ? -et.ntlo : __int_as_float(0x7f800000);
        // min-p state: FP64 work only in permuted groups (FP64 issue is slow here)
        MinpState ms;
        MinpLead lead;
        double *key_ptr = nullptr;
        if (minp_mode) {
          lead.start = 0.0;
          lead.c1 = 0.f;
          lead.c2 = 0.f;
          if (et.valid) {
            lead.c1 = (float)et.cfac * p.h1;  // FP32: these only scale the filter
            lead.c2 = (float)et.cfac * p.h2 * 0.5f;
            key_ptr = g.minp_key + (int64_t)(ag - 1) * g.rows_per_agroup + et.trait;
            lead.start = reinterpret_cast<const double *>(tcp + 1536)[row];
          }
          for (int k = 0; k < 2; ++k) {
            lead.cls[k].s = 0.f;
            lead.cls[k].u = __int_as_float(0x7fc00000);  // NaN: equal to no pair
            lead.cls[k].k64 = -1.0;
          }
          lead.exact = -1.0;
          ms = minp_bounds((float)lead.start, lead.c1, lead.c2, p.margin);
          if (seed_pass) {  // ms tracks the largest values instead
            ms.s1_lo = 0.f;
            ms.s2_lo = 0.f;
          }
        }
        for (int c = 0; c < nc_item; ++c) {
          bool ok = true;
          if (step == w.step_begin) ok = wait_bar(b_full(c), (b_bits >> c) & 1u, wc, 6);
          ok = ok && wait_bar(t_full(slot), slot_phase, wc, 7);
          if (!__all_sync(0xffffffffu, ok)) goto epi_done;
          tc_fence_after();
          if constexpr (kForm == kFormMulti) {
            // markers with up to five groups: this warp's 8 SNPs of a 32-SNP chunk,
            // D_i of SNP j in column 32 i + j (i = 0..3)
            uint32_t dd[kMaxCodeM][kEpiSnpsM];
            const uint32_t tb =
                tmem_base + ((uint32_t)(32 * q) << 16) + slot * 128u + (uint32_t)(kEpiSnpsM * h);
#pragma unroll
            for (int i = 0; i < kMaxCodeM; ++i) tmem_ld8(tb + (uint32_t)(kChunkSnpsM * i), dd[i]);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(t_empty(slot));
            if (++slot == (uint32_t)kTmemSlots) {
              slot = 0;
              slot_phase ^= 1u;
            }
            const ChunkMetaM &mm = reinterpret_cast<const ChunkMetaM &>(meta_of(c));
            const bool need = hit_fast_m(dd, mm, h, et.ntlo);
            if (__any_sync(0xffffffffu, need)) {
              uint32_t dv[kMaxCodeM * kEpiSnpsM];
#pragma unroll
              for (int i = 0; i < kMaxCodeM; ++i)
#pragma unroll
                for (int j = 0; j < kEpiSnpsM; ++j) dv[kEpiSnpsM * i + j] = dd[i][j];
              wn += hit_event_m(dv, need && et.valid, mm, h, et.trait, et.ntlo, et.nthi, et.cfac,
                                g, p, wn, lane);
            }
          } else {
            uint32_t d0[kEpiSnps], d1[kEpiSnps];
            const uint32_t taddr =
                tmem_base + ((uint32_t)(32 * q) << 16) + slot * 128u + (uint32_t)(kEpiSnps * h);
            tmem_ld16(taddr, d0);
            tmem_ld16(taddr + 64u, d1);
            tmem_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(t_empty(slot));
            if (++slot == (uint32_t)kTmemSlots) {
              slot = 0;
              slot_phase ^= 1u;
            }
            const uint64_t *codes =
                g.codes ? reinterpret_cast<const uint64_t *>(scodes + (size_t)c * codes_stride) : nullptr;
            const ChunkMeta &mc = meta_of(c);
            bool need;
            if (minp_mode && seed_pass) {
              // seed pass: only the range of the values (traits with NaN sit out)
              float smax, smin;
              minp_range(d0, d1, mc, h, smax, smin);
              ms.s2_lo = fmaxf(ms.s2_lo, smax);
              ms.s1_lo = fmaxf(ms.s1_lo, -smin);
              need = false;
            } else if (minp_mode) {
              if (!et.valid) {
                need = false;
              } else if (et.nan_cnt > 0) {
                need = true;
              } else {
                float smax, smin;
                minp_range(d0, d1, mc, h, smax, smin);
                need = smax > ms.s2_lo || -smin > ms.s1_lo || fmaxf(smax, -smin) >= fdr_tau_lo;
                if (need) {
                  // the row's bounds from the other warps' leaders of this step first
                  const unsigned long long b1 = sbound[row], b2 = sbound[kTileM + row];
                  if ((uint32_t)(b1 >> 32) == step_tag)
                    ms.s1_lo = fmaxf(ms.s1_lo, __uint_as_float((uint32_t)b1));
                  if ((uint32_t)(b2 >> 32) == step_tag)
                    ms.s2_lo = fmaxf(ms.s2_lo, __uint_as_float((uint32_t)b2));
                  need = smax > ms.s2_lo || -smin > ms.s1_lo || fmaxf(smax, -smin) >= fdr_tau_lo;
                }
              }
            }
            else if (kForm == kFormNan && et.nan_cnt > 0)
              need = p.dense || hit_fast_nan(d0, d1, mc, h, codes, et.nan_cnt, et.nan_idx,
                                             nan_q1, nan_q2);
            else
              need = p.dense || et.nan_cnt > 0 ||
                     (p.signed_coef ? hit_fast<true>(d0, d1, mc, h, et.ntlo)
                                    : hit_fast<false>(d0, d1, mc, h, et.ntlo));
            if (__any_sync(0xffffffffu, need)) {
              // rare paths work on a local copy of the accumulators
              uint32_t dv[2 * kEpiSnps];
  #pragma unroll
              for (int j = 0; j < kEpiSnps; ++j) {
                dv[j] = d0[j];
                dv[kEpiSnps + j] = d1[j];
              }
              if (minp_mode) {
                if (need) {
                  if (et.nan_cnt > 0)
                    minp_event_nan(dv, mc, codes, h, et.cfac, et.nan_cnt, et.nan_idx, &lead, p, ag);
                  else {
                    ms = minp_event(dv, mc, h, et.cfac, &lead, ms, fdr_tau_lo, p, ag);
                    const unsigned long long tag = (unsigned long long)step_tag << 32;
                    atomicMax(&sbound[row], tag | __float_as_uint(ms.s1_lo));
                    atomicMax(&sbound[kTileM + row], tag | __float_as_uint(ms.s2_lo));
                  }
                }
              } else if (__any_sync(0xffffffffu, p.dense || et.nan_cnt > 0)) {
                hit_slow(dv, need, mc, codes, h, et.trait, et.valid, et.ntlo, et.nthi, et.cfac,
                         et.nan_cnt, et.nan_idx, g, p, lane);
              } else {
                if constexpr (kForm == kFormPerm)
                  wn += hit_event_cols(dv, need && et.valid, mc, h, et.trait, et.ntlo, et.nthi,
                                       et.cfac, g, p, wn, lane);
                else
                  wn += hit_event(dv, need && et.valid, mc, h, et.trait, et.ntlo, et.nthi, et.cfac,
                                  g, p, wn, lane);
              }
            }
          }
          if (step == w.step_end - 1) {
            __syncwarp();
            if (lane == 0) mbar_arrive(b_empty(c));
          }
        }
        if (minp_mode && key_ptr != nullptr) {
          const double k64 = !seed_pass         ? minp_step_best(&lead, et.cfac)
                             : et.nan_cnt == 0 ? minp_seed_key(ms, lead.c1, lead.c2, p.margin)
                                               : -1.0;
          if (k64 > lead.start)
            atomicMax(reinterpret_cast<unsigned long long *>(key_ptr),
                      (unsigned long long)__double_as_longlong(k64));
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(tc_empty(tc_e));
        if (++tc_e == (uint32_t)kTcDepth) {
          tc_e = 0;
          tc_phase ^= 1u;
        }
      }
      for (int c = 0; c < nc_item; ++c) b_bits ^= 1u << c;
    }
  epi_done:
    tc_fence_before();
    if (lane == 0 && p.seg_cap > 0)
      p.seg_cnt[blockIdx.x * kEpiWarps + warp] = min(wn, (unsigned int)p.seg_cap);
  }

  __syncthreads();
  if constexpr (kPair) {
    // Both CTAs' roles have ended, and each tells the other what it has asked for.
    if (threadIdx.x == 0) {
      note[0].aborted = (uint32_t)*abort_flag;
      const uint32_t to = peer_addr(smem_u32(const_cast<PairNote *>(note + 1)), rank ^ 1u);
      st_cluster(to + offsetof(PairNote, loads), note[0].loads);
      st_cluster(to + offsetof(PairNote, stage_atoms), note[0].stage_atoms);
      st_cluster(to + offsetof(PairNote, chunks), note[0].chunks);
      st_cluster(to + offsetof(PairNote, announced), note[0].announced);
      st_cluster(to + offsetof(PairNote, aborted), note[0].aborted);
    }
    cluster_sync();
    // Without a wait that gave up, the MMAs waited for every copy.  After one the CTAs may
    // have stopped at different tiles, at most nA apart (tile i is asked for when the MMAs
    // have read tile i - nA, which takes both halves), and the first CTA's barriers lack
    // what the one behind never asked for: those bytes are counted as arrived where the
    // first CTA expects both halves, and the second CTA's half alone is expected where it
    // had not armed the barrier yet.  Then every copy can be waited for.
    if (note[0].aborted | note[1].aborted) {
      if (threadIdx.x == 0) {
        const uint32_t chunks = note[0].chunks;
        if (rank == 0u) {
          const uint32_t n0 = note[0].loads, n1 = note[1].loads, most = max(n0, n1);
          const uint32_t atoms = n0 > n1 ? note[0].stage_atoms : note[1].stage_atoms;
          for (uint32_t i = min(n0, n1); i < most; ++i) {
            const uint32_t st = i % (uint32_t)nA, half = ((atoms >> (4 * st)) & 15u) * 4096u;
            if (n0 > n1) mbar_complete_tx(a_full(st), half);
            else mbar_expect_tx(a_full(st), half);
          }
          for (uint32_t i = most > (uint32_t)nA ? most - (uint32_t)nA : 0u; i < most; ++i)
            wait_drain(a_full(i % (uint32_t)nA), (i / (uint32_t)nA) & 1u, p.status, 10);
          // (a chunk that the second CTA has not announced: its arrival is made here)
          if (chunks > note[1].announced) mbar_arrive(b_full(0));
        }
        if (chunks > 0u) wait_drain(b_full(0), (chunks - 1u) & 1u, p.status, 11);
      }
      cluster_sync();  // the second CTA's copies are counted in the first one's memory
    }
    if (warp == R::kMma) {
      if (rank != 0u && lane == 0) wait_drain(drain, 0, p.status, 12);
      __syncwarp();
      tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
    }
    return;
  }
  if (warp == R::kMma && !kPair) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
}

// Appends every staging segment (one per epilogue warp of every CTA) after the
// directly appended hits: block b copies segment b to offset
// direct + sum_{c<b} seg_cnt[c] (entries past the capacity are dropped); block 0
// also writes the exact total.
__global__ void seg_compact_kernel(const krux_hit *__restrict__ seg_hits,
                                   const HitAux *__restrict__ seg_aux,
                                   const HitAux2 *__restrict__ seg_aux2,
                                   const unsigned int *__restrict__ seg_cnt, int n_seg,
                                   int seg_cap, const unsigned long long *__restrict__ direct,
                                   krux_hit *__restrict__ out, HitAux *__restrict__ out_aux,
                                   HitAux2 *__restrict__ out_aux2, int64_t capacity,
                                   unsigned long long *total) {
  __shared__ unsigned long long part[2][8];
  const int b = blockIdx.x;
  unsigned long long before = 0, all = 0;
  for (int c = threadIdx.x; c < n_seg; c += blockDim.x) {
    const unsigned long long v = seg_cnt[c];
    all += v;
    if (c < b) before += v;
  }
  for (int o = 16; o > 0; o >>= 1) {
    before += __shfl_xor_sync(0xffffffffu, before, o);
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  if ((threadIdx.x & 31) == 0) {
    part[0][threadIdx.x >> 5] = before;
    part[1][threadIdx.x >> 5] = all;
  }
  __syncthreads();
  unsigned long long off = *direct, tot = *direct;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    off += part[0][w];
    tot += part[1][w];
  }
  if (b == 0 && threadIdx.x == 0) *total = tot;
  const unsigned int n = seg_cnt[b];
  const size_t s0 = (size_t)b * seg_cap;
  for (unsigned int i = threadIdx.x; i < n; i += blockDim.x) {
    const unsigned long long o = off + i;
    if (o < (unsigned long long)capacity) {
      st_hit(out + o, ld_hit(seg_hits + s0 + i));
      st_aux(out_aux + o, ld_aux(seg_aux + s0 + i));
      if (out_aux2 != nullptr) out_aux2[o] = seg_aux2[s0 + i];
    }
  }
}

// 1/n in FP64 for n = 0..kMaxN (entry 0 unused): the finalisation multiplies
// instead of dividing (FP64 division is slow on this part).
__device__ double c_rcp[kMaxN + 1];  // (global, read through L1: the indices differ by lane)

// FP64 statistic and p-value of each stored hit, from its exact centred sums.
__device__ __forceinline__ void finalize_one(const krux_hit *__restrict__ hits,
                                             const HitAux *__restrict__ aux,
                                             const HitAux2 *__restrict__ aux2, int64_t i,
                                             const double *const *__restrict__ cfac_by_group,
                                             double *__restrict__ H, double *__restrict__ P,
                                             unsigned long long *fdr_hist, int fdr_bins,
                                             double fdr_l0, double fdr_w, double pthresh) {
  const krux_hit r = ld_hit(hits + i);
  const HitAux a = ld_aux(aux + i);
  const double cf = cfac_by_group[a.group][r.trait];
  int df;
  double Q;
  if (aux2 == nullptr) {
    df = df_of(a.n0, a.n1, a.n2);
    const double D0 = (double)r.d0, D1 = (double)r.d1, D2 = -(double)(r.d0 + r.d1);
    Q = D0 * D0 * __ldg(&c_rcp[a.n0]);
    Q = fma(D1 * D1, __ldg(&c_rcp[a.n1]), Q);
    Q = fma(D2 * D2, __ldg(&c_rcp[a.n2]), Q);
  } else {  // five groups: D_4 = -(D_0 + D_1 + D_2 + D_3)
    const HitAux2 b = aux2[i];
    const int n[5] = {a.n0, a.n1, a.n2, b.n3, b.n4};
    const double D[5] = {(double)r.d0, (double)r.d1, (double)b.d2, (double)b.d3,
                         -((double)r.d0 + (double)r.d1 + (double)b.d2 + (double)b.d3)};
    int groups = 0;
    Q = 0.0;
    for (int k = 0; k < 5; ++k) {
      groups += n[k] > 0;
      Q = fma(D[k] * D[k], __ldg(&c_rcp[n[k]]), Q);
    }
    df = groups > 0 ? groups - 1 : 0;
  }
  const double h = cf * Q;
  H[i] = h;
  double pv;
  if (df < 1 || df > 2) {  // markers with more groups: df 3, 4
    pv = chi2_tail64(h, df);
  } else {
    pv = kw_p_report(h, df);
    if (pv >= pthresh) pv = kw_p64(h, df);  // a hit's p stays below P_c as decided
  }
  P[i] = pv;
  if (fdr_hist != nullptr)  // row 0: the real data's hits by -log10 p bin
    atomicAdd(fdr_hist + fdr_bin(key64_of(h, df), fdr_l0, fdr_w, fdr_bins), 1ull);
}

__global__ void finalize_kernel(const krux_hit *__restrict__ hits, const HitAux *__restrict__ aux,
                                int64_t n, const double *const *__restrict__ cfac_by_group,
                                double *__restrict__ H, double *__restrict__ P,
                                unsigned long long *fdr_hist, int fdr_bins, double fdr_l0,
                                double fdr_w, double pthresh) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    finalize_one(hits, aux, nullptr, i, cfac_by_group, H, P, fdr_hist, fdr_bins, fdr_l0, fdr_w,
                 pthresh);
}

// The same over min(*count, capacity) hits, the count read on the device (no host
// round trip between the scan and the finalisation; capturable in a graph).
__global__ void finalize_dev_kernel(const krux_hit *__restrict__ hits,
                                    const HitAux *__restrict__ aux,
                                    const HitAux2 *__restrict__ aux2,
                                    const unsigned long long *__restrict__ count, int64_t capacity,
                                    const double *const *__restrict__ cfac_by_group,
                                    double *__restrict__ H, double *__restrict__ P,
                                    unsigned long long *fdr_hist, int fdr_bins, double fdr_l0,
                                    double fdr_w, double pthresh) {
  const unsigned long long c = *count;
  const int64_t n = c < (unsigned long long)capacity ? (int64_t)c : capacity;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    finalize_one(hits, aux, aux2, i, cfac_by_group, H, P, fdr_hist, fdr_bins, fdr_l0, fdr_w, pthresh);
}

// The deferred FP64 pass of a plain-form permutation launch: every listed pair's
// -ln p (section "P-value calculation and empirical FDR correction"), the largest
// per (permutation, trait) into the key, and pairs of the FDR band with p < P_c
// into the histogram row of their permutation.
__global__ void minp_cands_kernel(const MinpPair *__restrict__ list, const unsigned int *__restrict__ cnt,
                                  int n_lists, int cap, const double *__restrict__ cfac, int rows_pad,
                                  double lp, double *key, unsigned long long *fdr_hist, int fdr_bins,
                                  double fdr_l0, double fdr_w) {
  for (int l = blockIdx.y; l < n_lists; l += gridDim.y) {
    const unsigned int n = min(cnt[l], (unsigned int)cap);
    for (unsigned int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
      const MinpPair r = list[(size_t)l * cap + i];
      const int df = (int)(r.n2df >> 16), ag = r.agb & 0xffff;
      const double cf = cfac[r.trait];
      if (df <= 0 || !(cf > 0.0)) continue;
      const double k = key64_of(kw_H64(r.u, r.v, (int)(r.n01 & 0xffffu), (int)(r.n01 >> 16),
                                       (int)(r.n2df & 0xffffu), cf),
                                df);
      if (r.agb & (1 << 17))
        atomicMax(reinterpret_cast<unsigned long long *>(key + (int64_t)(ag - 1) * rows_pad + r.trait),
                  (unsigned long long)__double_as_longlong(k));
      if ((r.agb & (1 << 16)) && fdr_hist != nullptr && k > lp)
        atomicAdd(fdr_hist + (int64_t)ag * fdr_bins + fdr_bin(k, fdr_l0, fdr_w, fdr_bins), 1ull);
    }
  }
}

// After a plain-form seed pass of a permutation batch: each (permutation q, trait,
// class) whose seed record names a 16-SNP block.  The block's centred rank sums are
// recomputed as integers (the permuted centred ranks against the genotype indicators, as
// the contraction forms them), its largest value of the class is found again with the
// fast test's FP32 expression, that pair's FP64 -ln p (section "P-value calculation and
// empirical FDR correction") is folded into the key, and its value becomes the class's
// largest decided value.
//
// A warp works on `per` records in turn, its lanes on the samples (whole genotype rows),
// then lane j on the block's SNP j, and keeps each record's winner in a lane of its own:
// the FP64 part, the slowest unit of this chip, runs once for all of them.  With one
// record per warp, FP64 on a single lane and a rank loaded again for each SNP, 16 x
// 20,000 permuted traits took 2.82 ms, with 32 0.90.  kI: the samples of a lane.
// A batch too small to give every SM 16 warps of 32 records takes fewer in a warp, whose
// records are a chain of dependent loads (whole calls: 3 x 2,000 x 10,000, N = 102 527 -> 414
// us, N = 300 1,140 -> 563; 3 x 128 x 500, N = 200 447 -> 289).
template <int kI>
__global__ void __launch_bounds__(256)
    seed_decide_kernel(const unsigned long long *__restrict__ rec, const __half *__restrict__ stack,
                       int rows_pad, int Np, int N, int T, int P, const int8_t *__restrict__ geno,
                       int64_t ldg, int64_t n_snps, const ChunkMeta *__restrict__ meta, const double *__restrict__ cfac, double *key,
                       unsigned long long *bound, int per) {
  const int lane = threadIdx.x & 31;
  const int64_t nrec = (int64_t)P * T * 2;
  const bool packed = N <= 360;  // both sums (at most K^2 / 4) fit 16 bits
  for (int64_t r0 = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * per; r0 < nrec;
       r0 += (int64_t)gridDim.x * (blockDim.x >> 5) * per) {
    float best = 0.f;  // of record r0 + lane
    int bu = 0, bv = 0;
    int64_t bpos = -1;
    const unsigned long long mine =
        lane < per && r0 + lane < nrec ? rec[2 * ((r0 + lane) / 2 / T * rows_pad + (r0 + lane) / 2 % T) + (lane & 1)] : 0ull;
    uint32_t todo = __ballot_sync(0xffffffffu, mine != 0ull);
    while (todo) {
      const int i = __ffs((int)todo) - 1;
      todo &= todo - 1u;
      const int64_t qt = (r0 + i) >> 1;
      const int q = (int)(qt / T), trait = (int)(qt % T);
      const int64_t pos0 = (int64_t)__shfl_sync(0xffffffffu, (uint32_t)mine, i) - 1;
      const int64_t arow = (int64_t)(1 + q) * rows_pad + trait;  // (the plain forms' layout)
      int ak[kI];
#pragma unroll
      for (int t = 0; t < kI; ++t) {
        const int k = lane + 32 * t;
        ak[t] = k < N ? (int)__half2float(stack[tiled_index(arow, k, Np)]) : 0;
      }
      const int nj = (int)min((int64_t)16, n_snps - pos0);
      int snp = -1;  // of position lane
      if (lane < nj) snp = meta[(pos0 + lane) / kChunkSnps].snp[(pos0 + lane) % kChunkSnps];
      int d0 = 0, d1 = 0;  // of SNP lane
#pragma unroll 4
      for (int j = 0; j < nj; ++j) {
        const int8_t *g = geno + max(__shfl_sync(0xffffffffu, snp, j), 0) * ldg;
        int a = 0, b = 0;
#pragma unroll
        for (int t = 0; t < kI; ++t) {
          const int k = lane + 32 * t;
          if (k < N) {
            const int8_t gk = g[k];
            a += gk == 0 ? ak[t] : 0;
            b += gk == 1 ? ak[t] : 0;
          }
        }
        if (packed) {
          a = __reduce_add_sync(0xffffffffu, a + (b << 16));
          b = (a - (int)(int16_t)a) >> 16;
          a = (int)(int16_t)a;
        } else {
          a = __reduce_add_sync(0xffffffffu, a);
          b = __reduce_add_sync(0xffffffffu, b);
        }
        if (lane == j) {
          d0 = a;
          d1 = b;
        }
      }
      float val = 0.f;
      if (lane < nj) {
        const ChunkMeta &m = meta[(pos0 + lane) / kChunkSnps];
        const int w = (int)((pos0 + lane) % kChunkSnps);
        if (snp >= 0) {
          const float sv = kw_s((float)d0, (float)d1, m.alpha[w], m.beta[w], m.gamma[w]);
          val = fmaxf((i & 1) ? sv : -sv, 0.f);
        }
      }
      // (the first SNP of the largest value)
      const uint32_t top = __reduce_max_sync(0xffffffffu, __float_as_uint(val));
      if (top == 0u) continue;
      const int w = __ffs((int)__ballot_sync(0xffffffffu, __float_as_uint(val) == top)) - 1;
      d0 = __shfl_sync(0xffffffffu, d0, w);
      d1 = __shfl_sync(0xffffffffu, d1, w);
      if (lane == i) {
        best = __uint_as_float(top);
        bu = d0;
        bv = d1;
        bpos = pos0 + w;
      }
    }
    if (bpos < 0) continue;
    const int cls = lane & 1;
    const int64_t qt = (r0 + lane) >> 1;
    const int q = (int)(qt / T), trait = (int)(qt % T);
    const int64_t idx = (int64_t)q * rows_pad + trait;
    const ChunkMeta &m = meta[bpos / kChunkSnps];
    const int w = (int)(bpos % kChunkSnps);
    const int df = m.df[w];
    const double cf = cfac[trait];
    if (df > 0 && cf > 0.0) {
      const double k64 = key64_of(kw_H64(bu, bv, m.n[0][w], m.n[1][w], m.n[2][w], cf), df);
      atomicMax(reinterpret_cast<unsigned long long *>(key + idx),
                (unsigned long long)__double_as_longlong(k64));
    }
    atomicMax(bound + 2 * idx + cls, ((unsigned long long)__float_as_uint(best) << 32) | pair_id(bu, bv));
  }
}

// minimum p of each (permutation, trait) from its best -ln p (key rows of ld entries)
__global__ void minp_from_key_kernel(const double *__restrict__ key, double *__restrict__ minp,
                                     int P, int T, int ld) {
  const int64_t n = (int64_t)P * T;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    minp[i] = exp(-key[(i / T) * ld + i % T]);
}

}  // namespace

cudaError_t launch_seg_compact(const krux_hit *seg_hits, const HitAux *seg_aux,
                               const HitAux2 *seg_aux2, const unsigned int *seg_cnt, int n_seg,
                               int seg_cap, const unsigned long long *direct, krux_hit *out,
                               HitAux *out_aux, HitAux2 *out_aux2, int64_t capacity,
                               unsigned long long *total, cudaStream_t s) {
  if (n_seg <= 0) return cudaSuccess;
  seg_compact_kernel<<<n_seg, 256, 0, s>>>(seg_hits, seg_aux, seg_aux2, seg_cnt, n_seg, seg_cap,
                                           direct, out, out_aux, out_aux2, capacity, total);
  return cudaGetLastError();
}

cudaError_t launch_minp_from_key(const double *key, double *minp, int P, int T, int ld,
                                 cudaStream_t s) {
  const int64_t n = (int64_t)P * T;
  if (n <= 0) return cudaSuccess;
  int grid = (int)((n + 255) / 256);
  if (grid > 4096) grid = 4096;
  minp_from_key_kernel<<<grid, 256, 0, s>>>(key, minp, P, T, ld);
  return cudaGetLastError();
}

cudaError_t launch_minp_cands(const MinpPair *list, const unsigned int *cnt, int n_lists, int cap,
                              const double *cfac, int rows_pad, double pthresh, double *key,
                              unsigned long long *fdr_hist, int fdr_bins, double fdr_l0,
                              double fdr_w, cudaStream_t s) {
  if (n_lists <= 0 || cap <= 0) return cudaSuccess;
  const dim3 grid((unsigned)((cap + 255) / 256 < 64 ? (cap + 255) / 256 : 64),
                  (unsigned)(n_lists < 65535 ? n_lists : 65535));
  minp_cands_kernel<<<grid, 256, 0, s>>>(list, cnt, n_lists, cap, cfac, rows_pad, -log(pthresh), key,
                                         fdr_hist, fdr_bins, fdr_l0, fdr_w);
  return cudaGetLastError();
}

cudaError_t launch_seed_decide(const unsigned long long *rec, const __half *stack, int rows_pad,
                               int Np, int N, int T, int P, const int8_t *geno, int64_t ldg,
                               int64_t n_snps, const ChunkMeta *meta,
                               const double *cfac, double *key, unsigned long long *bound,
                               cudaStream_t s) {
  const int64_t records = (int64_t)P * T * 2;
  if (records <= 0) return cudaSuccess;
  int per = 32;  // records of a warp (even: a lane's class is its parity)
  while (per > 2 && records < (int64_t)per * 152 * 48) per >>= 1;
  const int64_t blocks = ((records + per - 1) / per + 7) / 8;
  const int grid = (int)(blocks < 65535 ? blocks : 65535);
  auto *kernel = N <= 128   ? seed_decide_kernel<4>
                 : N <= 192 ? seed_decide_kernel<6>
                 : N <= 256 ? seed_decide_kernel<8>
                 : N <= 320 ? seed_decide_kernel<10>
                 : N <= 384 ? seed_decide_kernel<12>
                            : seed_decide_kernel<16>;
  kernel<<<grid, 256, 0, s>>>(rec, stack, rows_pad, Np, N, T, P, geno, ldg, n_snps, meta, cfac,
                              key, bound, per);
  return cudaGetLastError();
}

size_t scan_smem_bytes(int nc, int nA, int kpad) {
  return scan_smem_bytes2(nc, nA, (size_t)128 * kpad * 2, (size_t)nc * 128 * kpad * 2, kpad);
}

size_t scan_smem_bytes2(int nc, int nA, size_t a_tile_bytes, size_t b_region, int codes_k) {
  return 1024 + (size_t)nA * a_tile_bytes + b_region + (size_t)nc * kMetaGeneral +
         (size_t)nc * codes_k * 16 + (size_t)kTcDepth * kTcBytes + 16 * (size_t)kTileM +
         8 * (size_t)(2 * nA + 2 * nc + 2 * kTmemSlots + 1 + 2 * kTcDepth + 2 * kItemDepth) + 32;
}

bool fast_form_ok();
cudaError_t scan_set_smem_all(size_t smem);

cudaError_t scan_set_smem(size_t smem) {
  (void)fast_form_ok();  // its one-time check happens here, before any graph capture
  // the attribute is per device: skip the calls when it already has this value
  static std::atomic<size_t> last[64];
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 &&
      last[dev].load(std::memory_order_acquire) == smem + 1)
    return cudaSuccess;
  cudaError_t e = scan_set_smem_all(smem);
  if (e == cudaSuccess && dev >= 0 && dev < 64) last[dev].store(smem + 1, std::memory_order_release);
  return e;
}

cudaError_t scan_set_smem_all(size_t smem) {
  cudaError_t e = cudaFuncSetAttribute(krux_scan_kernel<kFormScan>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormScanNan>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormScanPerm>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormScanPair>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormScanMulti>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormScanDense>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormScanSeed>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormMulti>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(krux_scan_kernel<kFormNan>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(krux_scan_kernel<kFormPerm>,
                              cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// The kernel form launch_scan_only picks for these parameters (the ScanForm value).
int scan_form_of(const ScanParams &p) {
  const bool plain = p.fast && fast_form_ok();
  if (p.dense && plain) return kFormScanDense;
  if (p.multi) return plain ? kFormScanMulti : kFormMulti;
  if (p.perm) return !plain ? kFormPerm : (p.seed_bound ? kFormScanSeed : kFormScanPerm);
  if (!plain) return kFormNan;
  return p.fast_nan ? kFormScanNan : (p.pair_cta ? kFormScanPair : kFormScan);
}

// Launch of the pair form: clusters of two CTAs.
static void pair_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, int grid, size_t smem,
                        cudaStream_t s) {
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kFastThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = 2;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
}

// Pairs of CTAs that run at one time (its items are taken in fixed turns, so a grid
// must not exceed them), 0 where the pair form cannot run; looked up once per device.
int pair_clusters() {
  static std::atomic<int> known[64];
  int dev = 0;
  if (!fast_form_ok() || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int v = known[dev].load(std::memory_order_acquire);
  if (v == 0) {
    constexpr size_t kSmem = 232448;
    cudaFuncAttributes a;
    int n = 0;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute attr{};
    pair_config(cfg, attr, 2, kSmem, nullptr);
    const bool ok = cudaFuncGetAttributes(&a, krux_scan_kernel<kFormScanPair>) == cudaSuccess &&
                    a.numRegs == kFastRegsLaunch && a.maxThreadsPerBlock >= kFastThreads &&
                    cudaFuncSetAttribute(krux_scan_kernel<kFormScanPair>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kSmem) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, krux_scan_kernel<kFormScanPair>, &cfg) == cudaSuccess;
    v = 1 + (ok ? n : 0);
    known[dev].store(v, std::memory_order_release);
  }
  return v - 1;
}

cudaError_t launch_scan_only(const ScanParams &p, int grid, size_t smem, cudaStream_t s) {
  switch (scan_form_of(p)) {
    case kFormScan: krux_scan_kernel<kFormScan><<<grid, kFastThreads, smem, s>>>(p); break;
    case kFormScanNan: krux_scan_kernel<kFormScanNan><<<grid, kFastThreads, smem, s>>>(p); break;
    case kFormScanDense: krux_scan_kernel<kFormScanDense><<<grid, kFastThreads, smem, s>>>(p); break;
    case kFormScanMulti: krux_scan_kernel<kFormScanMulti><<<grid, kFastThreads, smem, s>>>(p); break;
    case kFormScanSeed: krux_scan_kernel<kFormScanSeed><<<grid, kFastThreads, smem, s>>>(p); break;
    case kFormScanPerm: krux_scan_kernel<kFormScanPerm><<<grid, kFastThreads, smem, s>>>(p); break;
    case kFormScanPair: {
      cudaLaunchConfig_t cfg{};
      cudaLaunchAttribute attr{};
      pair_config(cfg, attr, grid, smem, s);
      return cudaLaunchKernelEx(&cfg, krux_scan_kernel<kFormScanPair>, p);
    }
    case kFormMulti: krux_scan_kernel<kFormMulti><<<grid, kScanThreads, smem, s>>>(p); break;
    case kFormPerm: krux_scan_kernel<kFormPerm><<<grid, kScanThreads, smem, s>>>(p); break;
    default:  // NaN beyond the coefficient sets, and whatever fits no plain form
      krux_scan_kernel<kFormNan><<<grid, kScanThreads, smem, s>>>(p);
  }
  return cudaGetLastError();
}

// The plain scan form moves registers between its warpgroups with setmaxnreg,
// which is sound only if the kernel was built with exactly the launch register
// count the split assumes (else an increase could wait for registers that were
// never there): checked once, before its first launch.
bool fast_form_ok() {
  static std::atomic<int> ok{-1};
  int v = ok.load(std::memory_order_acquire);
  if (v < 0) {
    // the plain-form kernels were built at the register count their warp roles'
    // setmaxnreg split assumes
    cudaFuncAttributes a, b, c, d, m, n;
    v = cudaFuncGetAttributes(&a, krux_scan_kernel<kFormScan>) == cudaSuccess &&
                cudaFuncGetAttributes(&b, krux_scan_kernel<kFormScanPerm>) == cudaSuccess &&
                cudaFuncGetAttributes(&c, krux_scan_kernel<kFormScanNan>) == cudaSuccess &&
                cudaFuncGetAttributes(&d, krux_scan_kernel<kFormScanSeed>) == cudaSuccess &&
                d.numRegs == kFastRegsLaunch && d.maxThreadsPerBlock >= kFastThreads &&
                cudaFuncGetAttributes(&m, krux_scan_kernel<kFormScanMulti>) == cudaSuccess &&
                m.numRegs == kFastRegsLaunch && m.maxThreadsPerBlock >= kFastThreads &&
                cudaFuncGetAttributes(&n, krux_scan_kernel<kFormScanDense>) == cudaSuccess &&
                n.numRegs == kFastRegsLaunch && n.maxThreadsPerBlock >= kFastThreads &&
                a.numRegs == kFastRegsLaunch && a.maxThreadsPerBlock >= kFastThreads &&
                b.numRegs == kFastRegsLaunch && b.maxThreadsPerBlock >= kFastThreads &&
                c.numRegs == kFastRegsLaunch && c.maxThreadsPerBlock >= kFastThreads
            ? 1
            : 0;
    ok.store(v, std::memory_order_release);
  }
  return v == 1;
}

cudaError_t launch_scan(const ScanParams &p, int grid, size_t smem, cudaStream_t s) {
  cudaError_t e = scan_set_smem(smem);
  if (e != cudaSuccess) return e;
  return launch_scan_only(p, grid, smem, s);
}

cudaError_t finalize_prepare(cudaStream_t s) {
  static std::atomic<unsigned long long> uploaded{0};
  return once_per_device(uploaded, s, [](cudaStream_t s) {
    static const struct Reciprocals {
      double t[kMaxN + 1];
      Reciprocals() {
        t[0] = 0.0;  // empty groups have D_i = 0 and contribute nothing
        for (int k = 1; k <= kMaxN; ++k) t[k] = 1.0 / (double)k;
      }
    } rcp;
    return cudaMemcpyToSymbolAsync(c_rcp, rcp.t, sizeof rcp.t, 0, cudaMemcpyHostToDevice, s);
  });
}

cudaError_t launch_finalize(const krux_hit *hits, const HitAux *aux, int64_t n,
                            const double *const *cfac_by_group, double *H, double *p,
                            cudaStream_t s, unsigned long long *fdr_hist, int fdr_bins,
                            double fdr_l0, double fdr_w, double pthresh) {
  if (n <= 0) return cudaSuccess;
  cudaError_t e = finalize_prepare(s);
  if (e != cudaSuccess) return e;
  int grid = (int)((n + 255) / 256);
  if (grid > 152 * 8) grid = 152 * 8;
  finalize_kernel<<<grid, 256, 0, s>>>(hits, aux, n, cfac_by_group, H, p, fdr_hist, fdr_bins, fdr_l0,
                                       fdr_w, pthresh);
  return cudaGetLastError();
}

cudaError_t launch_finalize_dev(const krux_hit *hits, const HitAux *aux, const HitAux2 *aux2,
                                const unsigned long long *count, int64_t capacity,
                                const double *const *cfac_by_group, double *H, double *p,
                                int sm_count, cudaStream_t s, unsigned long long *fdr_hist,
                                int fdr_bins, double fdr_l0, double fdr_w, double pthresh) {
  if (capacity <= 0) return cudaSuccess;
  int grid = sm_count * 4;
  const int64_t need = (capacity + 255) / 256;
  if (need < grid) grid = (int)need;
  finalize_dev_kernel<<<grid, 256, 0, s>>>(hits, aux, aux2, count, capacity, cfac_by_group, H, p,
                                           fdr_hist, fdr_bins, fdr_l0, fdr_w, pthresh);
  return cudaGetLastError();
}

}  // namespace krux

