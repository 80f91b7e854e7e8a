// Householder QR of a tall matrix and the product of its unitary factor with a small one: what the
// operator builder's SVD does before and after rotating the n rows of R (svd_osj).  Always FP64.
//
// Factorisation.  Rows of A are spread over the CTAs of a cluster and stay in shared memory while
// they fit.  With x the part of column j below row j, alpha = A_jj and norm = |(alpha, x)|,
//   v = (alpha + norm alpha / |alpha|, x),  H = 1 - tau v v^dag,  tau = 2 / v^dag v
// (Householder 1958) takes the column to -norm alpha / |alpha| in row j.  tau comes from the v
// that was formed, so H is unitary to rounding whatever the error of norm.  v's head is kept
// aside and its rest is the column as it stands, so a step needs from the other CTAs only the
// sums x^dag A_:l of the columns l >= j and row j: one barrier a step, as
// v^dag A_:l = conj(v_j) A_jl + x^dag A_:l.  The CTAs sum the parts in the same order.
//
// Product.  U = H_0 ... H_(n-1) [C; 0], one CTA to a column of C: no exchange.
//
// What bounds it: a step takes ~9,000 cycles for its barriers, the chain of dependent FP64 operations
// that makes norm, head and factor of the reflector in one warp and, with more CTAs, the reads
// between them; the FP64 work of a recompression's small cores is less.  Measured on GB300 (QR, product, in
// brackets rotating R's rows between them): 12 x 3 13 and 8 us (42), 40 x 10 44 and 24 us (175),
// 64 x 16 73 and 39 us (294), 172 x 43 230 and 125 us (1,676), 1,000 x 64 0.61 and 0.47 ms (2.8).

#include <algorithm>
#include <cfloat>

#include "cluster.cuh"

namespace qlb {

namespace {

constexpr int TQ_NT = 256;
constexpr size_t TQ_SMEM_LIMIT = 200 * 1024;

// 2^t for a normal result
__device__ __forceinline__ double tq_pow2(int t) { return __hiloint2double((1023 + t) << 20, 0); }
// 1 / sqrt(x) of a normal x > 0, taken to [1, 4) by a power of four
__device__ __forceinline__ double tq_rsqrt(double x) {
  const int t = -((((__double2hiint(x) >> 20) & 0x7ff) - 1023) >> 1);
  return rsqrt_r(x * tq_pow2(2 * t)) * tq_pow2(t);
}

// entries of the buffers beside the slice: parts of the sums and row j (two sets in turn), totals
__host__ __device__ inline size_t tq_head(int n) { return 5 * (size_t)n; }

__global__ void __launch_bounds__(TQ_NT, 1) k_tall_qr(zd* A, int m, int n, int dagger, zd* R, zd* v0_out,
                                                      double* tau_out, int* status, int* count, int resident, int stall) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ unsigned long long s_cbar;
  __shared__ int s_gave_up;
  __shared__ double s_scal[5];  // v's head, tau, R_jj
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ca = (int)gridDim.x, rank = (int)cta_rank_in_cluster();
  zd* const part = (zd*)sm;         // [2][n], read by the others
  zd* const row = part + 2 * n;     // [2][n], the owner's is read by the others
  zd* const tot = row + 2 * n;      // [n]

  if (tid == 0) {
    s_gave_up = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&s_cbar)), "r"(ca + (stall == rank + 1))
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // once, with every CTA of the cluster: the barrier above is set up
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  ClusterBarrier cb{&s_cbar, &s_gave_up, ca, 0u, false};

  const int rpc = (m + ca - 1) / ca, r0 = min(m, rank * rpc), nl = min(m, r0 + rpc) - r0;
  zd* const g = A + (long)r0 * n;  // our rows
  zd* a = g;
  long ld = n;
  if (resident) {
    a = tot + n;
    ld = n | 1;
    for (int x = tid; x < nl * n; x += TQ_NT) a[(x / n) * ld + x % n] = g[x];
  }
  __syncthreads();
  for (int j = 0; j < n; j++) {
    const int par = (j & 1) * n, nc = n - j;
    const int rb = min(nl, max(0, j + 1 - r0)), nr = nl - rb;  // our rows below row j
    const int owner = j / rpc;
    // x^dag A_:l, a group of lanes to a column
    int G = 32;
    while (G > 4 && (nc * G > TQ_NT || G >= 2 * nr)) G >>= 1;
    const int gid = tid / G, gl = tid % G, ng = TQ_NT / G;
    for (int c0 = 0; c0 < nc; c0 += ng) {
      if (c0 + (warp * 32) / G >= nc) break;  // no column for this warp
      const int l = j + c0 + gid;
      double re = 0.0, im = 0.0;
      if (l < n)
        for (int r = rb + gl; r < nl; r += G) {
          const zd x = a[r * ld + j], y = a[r * ld + l];
          re = fma(x.im, y.im, fma(x.re, y.re, re));
          im = fma(-x.im, y.re, fma(x.re, y.im, im));
        }
      for (int o = 1; o < G; o <<= 1) {
        re += __shfl_xor_sync(0xffffffffu, re, o);
        im += __shfl_xor_sync(0xffffffffu, im, o);
      }
      if (l < n && gl == 0) part[par + l] = mk<double>(re, im);
    }
    if (rank == owner)
      for (int l = j + tid; l < n; l += TQ_NT) row[par + l] = a[(j - r0) * ld + l];
    if (!cb.sync()) break;
    // all parts, four lanes to a column
    for (int c0 = 0; c0 < nc; c0 += TQ_NT / 4) {
      if (c0 + warp * 8 >= nc) break;
      const int l = j + c0 + tid / 4;
      zd s = mk<double>(0.0, 0.0);
      if (l < n) {
        if (ca == 1) {
          if ((lane & 3) == 0) s = part[par + l];
        } else {
          for (int r = lane & 3; r < ca; r += 4) s = cadd(s, *on_cta(&part[par + l], r));
          if ((lane & 3) == 3 && rank != owner) row[par + l] = *on_cta(&row[par + l], owner);
        }
      }
      for (int o = 1; o < 4; o <<= 1) {
        s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
        s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
      }
      if (l < n && (lane & 3) == 0) tot[l] = s;
    }
    __syncthreads();
    if (warp == 0) {
      const zd alpha = row[par + j];
      const double x2 = tot[j].re, a2 = cabs2(alpha), n2 = a2 + x2;
      zd v = mk<double>(0.0, 0.0), d = alpha;
      double tau = 0.0;
      if (x2 > 0.0 && n2 >= DBL_MIN && ::isfinite(n2)) {
        const double norm = n2 * tq_rsqrt(n2);
        if (a2 >= DBL_MIN) {
          const double f = norm * tq_rsqrt(a2);
          d = mk<double>(-f * alpha.re, -f * alpha.im);
        } else {
          d = mk<double>(-norm, 0.0);
        }
        v = csub(alpha, d);
        const double q = cabs2(v) + x2, i2 = tq_rsqrt(q), i1 = i2 * i2;
        tau = 2.0 * fma(i1, fma(-q, i1, 1.0), i1);
      }
      if (lane == 0) {
        s_scal[0] = v.re;
        s_scal[1] = v.im;
        s_scal[2] = tau;
        s_scal[3] = d.re;
        s_scal[4] = d.im;
      }
    }
    __syncthreads();
    const zd v = mk<double>(s_scal[0], s_scal[1]);
    const double tau = s_scal[2];
    for (int l = tid; l < n; l += TQ_NT) {
      zd d = mk<double>(0.0, 0.0);
      if (l == j) d = mk<double>(s_scal[3], s_scal[4]);
      if (l > j) {
        zd h = tot[l];
        cfma(h, cconj(v), row[par + l]);
        h = cscale(h, tau);
        tot[l] = h;
        d = csub(row[par + l], cmul(v, h));
      }
      if (rank == owner) R[dagger ? (long)l * n + j : (long)j * n + l] = dagger ? cconj(d) : d;
    }
    if (rank == 0 && tid == 0) {
      v0_out[j] = v;
      tau_out[j] = tau;
    }
    __syncthreads();
    for (int x = tid; x < nr * (nc - 1); x += TQ_NT) {
      const int r = x / (nc - 1), l = j + 1 + x - r * (nc - 1);
      zd& y = a[(rb + r) * ld + l];
      const zd w = a[(rb + r) * ld + j];
      cfma(y, mk<double>(-w.re, -w.im), tot[l]);
    }
    __syncthreads();
  }
  const bool gave_up = cb.leave();
  if (rank == 0 && tid == 0) {
    *status = gave_up ? -2 : 0;
    *count = 0;
  }
  if (gave_up) return;
  if (resident)
    for (int x = tid; x < nl * n; x += TQ_NT) g[x] = a[(x / n) * ld + x % n];
}

// in_smem: the column in shared memory (m entries), else in its place in U
__global__ void k_tall_apply(const zd* A, int m, int n, const zd* v0, const double* tau, const zd* C, const int* kp,
                             zd* U, int in_smem) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ double s_sum[2][TQ_NT / 32][2];
  const int k = min(*kp, n), c = blockIdx.x;
  if (c >= k) return;
  const int tid = threadIdx.x, nt = blockDim.x, nw = nt >> 5;
  zd* const u = in_smem ? (zd*)sm : U + c;
  const long su = in_smem ? 1 : k;
  for (int r = tid; r < m; r += nt) u[r * su] = r < n ? C[(long)r * k + c] : mk<double>(0.0, 0.0);
  __syncthreads();
  int par = 0;
  for (int j = n - 1; j >= 0; j--) {
    const double t = tau[j];
    if (t == 0.0) continue;
    const zd vj = v0[j], uj = u[j * su];
    zd w = mk<double>(0.0, 0.0);
    for (int r = j + 1 + tid; r < m; r += nt) cfma(w, cconj(A[(long)r * n + j]), u[r * su]);
    for (int o = 16; o > 0; o >>= 1) {
      w.re += __shfl_xor_sync(0xffffffffu, w.re, o);
      w.im += __shfl_xor_sync(0xffffffffu, w.im, o);
    }
    if ((tid & 31) == 0) {
      s_sum[par][tid >> 5][0] = w.re;
      s_sum[par][tid >> 5][1] = w.im;
    }
    __syncthreads();
    w = mk<double>(s_sum[par][0][0], s_sum[par][0][1]);
    for (int i = 1; i < nw; i++) w = cadd(w, mk<double>(s_sum[par][i][0], s_sum[par][i][1]));
    cfma(w, cconj(vj), uj);
    w = cscale(w, -t);
    for (int r = j + 1 + tid; r < m; r += nt) cfma(u[r * su], A[(long)r * n + j], w);
    if (tid == 0) cfma(u[j * su], vj, w);
    par ^= 1;
    __syncthreads();
  }
  if (in_smem)
    for (int r = tid; r < m; r += nt) U[(long)r * k + c] = u[r];
}

struct TallPlan {
  int ca, resident;
  size_t smem;
  long cycles;  // of a step, by the count of FP64 operations
};

// Cycles of the first step on ca CTAs by what depends on their number: 64 per FP64 instruction of a
// warp, and 3,000 for a barrier and the reads between them.
TallPlan tall_split(int m, int n, int ca) {
  TallPlan p{};
  p.ca = ca;
  const int nl = (m + ca - 1) / ca;
  int g = 32;
  while (g > 4 && (n * g > TQ_NT || g >= 2 * nl)) g >>= 1;
  int lg = 0;
  while ((1 << lg) < g) lg++;
  const long warps = std::min<long>(TQ_NT / 32, ((long)n * g + 31) / 32);
  const long sums = ((long)n * g + TQ_NT - 1) / TQ_NT * ((warps + 3) / 4) * (4L * ((nl + g - 1) / g) + 2 * lg);
  const long rest = 2L * 4 * (((long)nl * n + TQ_NT - 1) / TQ_NT) + ((long)n * 4 + TQ_NT - 1) / TQ_NT * 2L * (ca / 2 + 4);
  const size_t head = tq_head(n) * sizeof(zd), rows = sizeof(zd) * (size_t)nl * (n | 1);
  p.resident = head + rows <= TQ_SMEM_LIMIT;
  p.smem = head + (p.resident ? rows : 0);
  p.cycles = 64 * (sums + rest) + (ca > 1 ? 5000 : 2000);
  return p;
}
TallPlan tall_plan(int m, int n) {
  TallPlan best = tall_split(m, n, 1);
  for (int ca = 2; ca <= FC_MAX_C; ca *= 2) {
    const TallPlan p = tall_split(m, n, ca);
    if (p.resident == best.resident ? p.cycles < best.cycles : p.resident > best.resident) best = p;
  }
  return best;
}

}  // namespace

cudaError_t launch_tall_qr(zd* A, int m, int n, int dagger, zd* R, zd* v0, double* tau, int* status, int* count,
                           int stall, cudaStream_t s) {
  const TallPlan p = tall_plan(m, n);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.ca, 1, 1);
  cfg.blockDim = dim3(TQ_NT, 1, 1);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.ca;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_tall_qr, A, m, n, dagger, R, v0, tau, status, count, p.resident, stall);
}

cudaError_t launch_tall_apply(const zd* A, int m, int n, const zd* v0, const double* tau, const zd* C, const int* k,
                              zd* U, cudaStream_t s) {
  const size_t smem = sizeof(zd) * (size_t)m;
  const int in_smem = smem <= TQ_SMEM_LIMIT;
  const int nt = m <= 128 ? 32 : m <= 1024 ? 128 : TQ_NT;
  k_tall_apply<<<n, nt, in_smem ? smem : 0, s>>>(A, m, n, v0, tau, C, k, U, in_smem);
  return cudaGetLastError();
}

void init_tallqr_attributes() {
  cudaFuncSetAttribute(k_tall_qr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TQ_SMEM_LIMIT);
  cudaFuncSetAttribute(k_tall_qr, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  cudaFuncSetAttribute(k_tall_apply, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TQ_SMEM_LIMIT);
}

}  // namespace qlb
