// What the two Gram-matrix solves over a thread-block cluster share (kernels_pj.cu: the
// truncation eigen-solve; kernels_range.cu: the zip-up range basis): access to the other
// CTAs' shared memory, a barrier over the CTAs that work on a problem, and sums of products in
// the working precision.
#pragma once

#include <type_traits>

#include "builder.cuh"
#include "df64.cuh"

namespace qlb {

namespace {

// Threads per CTA: FP64 one warp for each of the SM's four partitions, as a warp-wide FP64
// instruction holds a partition's pipe for 64 clocks and what every warp computes for itself
// (norms, thresholds, candidates) is paid per warp; double-float two, to cover its chains.
template <typename R>
struct ClThreads {
  static constexpr int v = std::is_same<R, double>::value ? 128 : 256;
};
constexpr int FC_MAX_N = 256;
constexpr int FC_MAX_C = 16;
// Residuals under 1e-30 of the trace (amplitudes 1e-15 of the state's) are not taken as
// pivots: they are below what the sites hold, and FP32 seeds need their range.
constexpr float FC_TINY = 1e-30f;

template <typename R>
struct FcEps;
template <>
struct FcEps<double> {
  static constexpr double v = 2.220446049250313e-16;
  static constexpr double pivot = 2.220446049250313e-16;
};
template <>
struct FcEps<df64> {
  static constexpr double v = 1.4210854715202004e-14;      // 2^-46: what a chain of double-float operations keeps
  static constexpr double pivot = 3.552713678800501e-15;   // 2^-48: the significand
};

// ------------------------------------------------------------------ cluster access

__device__ __forceinline__ unsigned cta_rank_in_cluster() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// address of the same shared variable in CTA `rank` of the cluster
template <typename T>
__device__ __forceinline__ T* on_cta(T* p, int rank) {
  unsigned long long out;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(out) : "l"((unsigned long long)p), "r"(rank));
  return (T*)out;
}
__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
// `bytes` of our shared memory at src to CTA `rank`'s at the place of dst, counted on that
// CTA's mbarrier at the place of bar
__device__ __forceinline__ void send_block(int rank, const void* dst, const void* src, unsigned bytes,
                                           const unsigned long long* bar) {
  unsigned rd, rb;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rd) : "r"(smem_addr(dst)), "r"(rank));
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_addr(bar)), "r"(rank));
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(rd),
               "r"(smem_addr(src)), "r"(bytes), "r"(rb)
               : "memory");
}
// waits for phase `parity` of our mbarrier, a second at most; false when the wait gave up
__device__ __forceinline__ bool bounded_wait(const unsigned long long* bar, unsigned parity) {
  unsigned long long t0 = 0;
  for (;;) {
    unsigned done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (!t0) t0 = t;
    if (t - t0 > 1000000000ull) return false;
  }
}

// Barrier over the CTAs that work on the problem, in two halves: every CTA's mbarrier
// counts one arrival of each of them.  Unlike the hardware's cluster barrier it leaves out
// the CTAs that have nothing to do, and its waits are bounded.
//
// A wait that gives up is lost for the whole CTA (`lost` is the same in every thread): the
// CTA takes part in no further phase and goes to leave(), where the others meet it, as
// their next wait gives up too.  The vote costs a block barrier a phase (~1 % of a step).
struct ClusterBarrier {
  const unsigned long long* bar;
  int* gave_up;  // of this CTA; set by any CTA that lost a wait
  int ca;
  unsigned phase;
  bool lost;
  // what one thread's bounded wait came to, for all threads; a block barrier
  __device__ __forceinline__ bool agree(bool ok) {
    lost = __syncthreads_or(!ok) != 0;
    return !lost;
  }
  // behind a block barrier
  __device__ __forceinline__ void post() {
    if ((int)threadIdx.x < ca) {
      unsigned rb;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(smem_addr(bar)), "r"((int)threadIdx.x));
      asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(rb) : "memory");
    }
  }
  __device__ __forceinline__ void arrive() {
    __syncthreads();
    post();
  }
  __device__ __forceinline__ bool wait() { return agree(bounded_wait(bar, phase++ & 1)); }
  __device__ __forceinline__ bool sync() {
    if (ca == 1) {
      __syncthreads();
      return true;
    }
    arrive();
    return wait();
  }
  // The way out of every CTA that works on the problem, lost or not: none of them touches
  // another one's shared memory any more.  True when any lost a wait (the same in all).  The
  // hardware's barrier waits for the CTAs that have not exited; each reaches it, as the
  // waits before are bounded and a lost CTA skips the rest.
  __device__ __forceinline__ bool leave() {
    if (ca == 1) {
      __syncthreads();
      return false;
    }
    if (lost && (int)threadIdx.x < ca) *on_cta(gave_up, (int)threadIdx.x) = 1;
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    return *(volatile int*)gave_up != 0;
  }
};

// ------------------------------------------------------------------ arithmetic

__device__ __forceinline__ double pmac(double c, double a, double b) { return fma(a, b, c); }
__device__ __forceinline__ df64 pmac(df64 c, df64 a, df64 b) { return df_mac(c, a, b); }
__device__ __forceinline__ double pzero(double) { return 0.0; }
__device__ __forceinline__ df64 pzero(df64) { return df64(0.f, 0.f); }
__device__ __forceinline__ float to_f(double x) { return (float)x; }
__device__ __forceinline__ float to_f(df64 x) { return x.hi; }
__device__ __forceinline__ double from_f(double, float x) { return (double)x; }
__device__ __forceinline__ df64 from_f(df64, float x) { return df64(x, 0.f); }

__device__ __forceinline__ double sx(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ df64 sx(df64 v, int m) {
  return df64(__shfl_xor_sync(0xffffffffu, v.hi, m), __shfl_xor_sync(0xffffffffu, v.lo, m));
}
__device__ __forceinline__ double sget(double v, int lane) { return __shfl_sync(0xffffffffu, v, lane); }
__device__ __forceinline__ df64 sget(df64 v, int lane) {
  return df64(__shfl_sync(0xffffffffu, v.hi, lane), __shfl_sync(0xffffffffu, v.lo, lane));
}
template <typename R>
__device__ __forceinline__ cx<R> csub_r(cx<R> a, cx<R> b) {
  return mk<R>(a.re - b.re, a.im - b.im);
}

// a <= b for finite a and b >= 0 (doubles: by their bit patterns, off the FP64 pipe)
__device__ __forceinline__ bool le_nn(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b);
}
__device__ __forceinline__ bool le_nn(df64 a, df64 b) { return a <= b; }

// 1 / sqrt(w) for w in FP32's normal range: FP32 seed y (relative error e / 2 ~ 1e-7)
// and one third-order step, y (1 + e/2 + 3 e^2 / 8) with e = 1 - w y^2, so no division
// or square root runs on the FP64 pipe
__device__ __forceinline__ double rsqrt_r(double w) {
  const double y = (double)rsqrtf((float)w);
  const double e = fma(-w * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ df64 rsqrt_r(df64 w) {
  const df64 y = df64(rsqrtf(w.hi), 0.f);
  const df64 e = df_mac(df64(1.f, 0.f), -(w * y), y);
  return df_mac(y, e * y, df64(0.5f, 0.375f * e.hi));
}

// Running sum of products.  Double-float: the high word takes a two-sum per product and
// every error term goes to one FP32 word (Ogita, Rump & Oishi 2005, "Accurate sum and dot
// product", Dot2 with the operands' low words), renormalised once at the end; the chain
// from product to product is then one FP32 addition instead of a renormalised sum.
template <typename R>
struct Acc;
template <>
struct Acc<double> {
  double s = 0.0;
  __device__ __forceinline__ void mac(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ double value() const { return s; }
  __device__ __forceinline__ void add_from(Acc o, int m) { s += __shfl_xor_sync(0xffffffffu, o.s, m); }
};
template <>
struct Acc<df64> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void mac(df64 a, df64 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p), t;
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    df_two_sum(s, p, s, t);
    c = __fadd_rn(c, __fadd_rn(e, t));
  }
  __device__ __forceinline__ df64 value() const {
    df64 r;
    df_two_sum(s, c, r.hi, r.lo);
    return r;
  }
  // plus o of lane ^ m
  __device__ __forceinline__ void add_from(Acc o, int m) {
    float t;
    const float os = __shfl_xor_sync(0xffffffffu, o.s, m), oc = __shfl_xor_sync(0xffffffffu, o.c, m);
    df_two_sum(s, os, s, t);
    c = __fadd_rn(__fadd_rn(c, oc), t);  // the same bits on both lanes
  }
};

// a x + b y + c z, one renormalisation
__device__ __forceinline__ double mul3(double a, double x, double b, double y, double c, double z) {
  return fma(c, z, fma(b, y, a * x));
}
__device__ __forceinline__ df64 mul3(df64 a, df64 x, df64 b, df64 y, df64 c, df64 z) {
  const float p1 = __fmul_rn(a.hi, x.hi), p2 = __fmul_rn(b.hi, y.hi), p3 = __fmul_rn(c.hi, z.hi);
  const float e1 = __fmaf_rn(a.lo, x.hi, __fmaf_rn(a.hi, x.lo, __fmaf_rn(a.hi, x.hi, -p1)));
  const float e2 = __fmaf_rn(b.lo, y.hi, __fmaf_rn(b.hi, y.lo, __fmaf_rn(b.hi, y.hi, -p2)));
  const float e3 = __fmaf_rn(c.lo, z.hi, __fmaf_rn(c.hi, z.lo, __fmaf_rn(c.hi, z.hi, -p3)));
  float s, t, u, v;
  df_two_sum(p1, p2, s, t);
  df_two_sum(s, p3, u, v);
  df64 r;
  df_quick_two_sum(u, __fadd_rn(__fadd_rn(e1, e2), __fadd_rn(e3, __fadd_rn(t, v))), r.hi, r.lo);
  return r;
}

// squared norm of a column as kept beside it (FP32 pair in both forms: rotations need it
// to FP32's relative accuracy, and its difference to another one's to the same)
__device__ __forceinline__ df64 to_df(double x) { return df64(x); }
__device__ __forceinline__ df64 to_df(df64 x) { return x; }

// sums of two values over groups of LP lanes (LP a power of two >= 2), the first exchange
// also splitting them over the lanes: even lanes of a group get re, odd lanes im
template <typename R>
__device__ __forceinline__ R csum(Acc<R> re, Acc<R> im, int LP) {
  const bool h = threadIdx.x & 1;
  Acc<R> q = h ? im : re;
  q.add_from(h ? re : im, 1);
  for (int o = 2; o < LP; o <<= 1) q.add_from(q, o);
  return q.value();
}

// ------------------------------------------------------------------ truncation rule

// Kept count of weights w[0..m) in falling order: relative discarded weight, cap (>= 1), no
// cut through a degenerate cluster.  Called by a whole warp; total and kept receive sums of the
// weights.
__device__ __forceinline__ int truncation_count(const double* w, int m, double tol, int cap, double gap, double& total,
                                                double& kept) {
  const int lane = threadIdx.x & 31;
  // lane l has the weights [l q, (l + 1) q)
  const int q = (m + 31) / 32, i0 = min(m, lane * q), i1 = min(m, i0 + q);
  double part = 0.0;
  for (int i = i0; i < i1; i++) part += w[i];
  double tail = part;  // of this lane's weights and all later ones
  for (int o = 1; o < 32; o <<= 1) {
    const double v = __shfl_down_sync(0xffffffffu, tail, o);
    if (lane + o < 32) tail += v;
  }
  total = __shfl_sync(0xffffffffu, tail, 0);
  double after = __shfl_down_sync(0xffffffffu, tail, 1);
  if (lane == 31) after = 0.0;
  // the smallest count whose discarded weight is within the cutoff
  int mine = i1;
  while (mine > i0 && after + w[mine - 1] <= tol * total) after += w[--mine];
  const unsigned whole = __ballot_sync(0xffffffffu, mine == i0);
  const int first = __clz(~whole);  // lanes whose weights all go, from the last one down
  int k = first == 32 ? 0 : __shfl_sync(0xffffffffu, mine, 31 - first);
  if (k < 1) k = 1;
  if (k > cap) k = cap;
  if (k < m) {
    auto same = [&](int j) { return ::sqrt(w[j]) >= (1.0 - gap) * ::sqrt(w[j - 1]); };
    if (same(k)) {  // a cut through a degenerate cluster: extend it under the cap, else cut before it
      int j = k;
      while (j < m && j < cap && same(j)) j++;
      if (j < m && same(j)) {
        j = k;
        while (j > 1 && same(j)) j--;
      }
      k = j;
    }
  }
  kept = 0.0;
  for (int i = i0; i < min(i1, k); i++) kept += w[i];
  for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
  return k;
}

}  // namespace

}  // namespace qlb
