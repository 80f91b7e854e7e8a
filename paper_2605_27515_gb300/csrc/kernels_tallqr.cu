// QR of a tall matrix, what the operator builder's SVD does before rotating the n rows of R
// (svd_osj): classical Gram-Schmidt on the columns, again while a pass takes more than three
// quarters of a column's squared norm ("twice is enough", Giraud, Langou & Rozloznik 2005).
// Always FP64.
//
// Gram-Schmidt and not reflectors: a basis vector is a combination of A's columns, so rows that are
// zero in the columns it comes from stay exactly zero, as they do under the rotations of the matrix's
// own rows.  Products of such operators keep the exact zeros between far Fock levels, which an
// explicit step that amplifies high levels needs; Householder's fill them with rounding
// (a^2 - alpha^2 at N = 64: 1,222 entries of up to 5e-15 beyond the second diagonal, none here).
//
// Rows of A are spread over the CTAs of a cluster and stay in shared memory while they fit.  A pass
// forms the products of column j with the basis so far and its norm (one barrier over the CTAs),
// sums the CTAs' parts in the same order and subtracts.  A column of which three passes leave
// nothing brings no new direction: its place in Q and its row of R are zero (the first column's
// place is a unit vector, so that a zero matrix has a left factor).
//
// What bounds it: a pass is its barriers, the reads between CTAs and two chains of FP64 sums; the
// FP64 work of a recompression's small cores is less.  Measured on GB300 (in brackets rotating R's
// rows behind it, and the product Q U): 12 x 3 13 us (42 and 6), 40 x 10 42 (176 and 6), 64 x 16 70
// (296 and 7), 172 x 43 224 (1,677 and 10), 1,000 x 64 677 (2,763 and 43).

#include <algorithm>
#include <cfloat>

#include "cluster.cuh"

namespace qlb {

namespace {

constexpr int TQ_NT = 256;
constexpr int TQ_NW = TQ_NT / 32;
constexpr size_t TQ_SMEM_LIMIT = 200 * 1024;

// 2^t for a normal result
__device__ __forceinline__ double tq_pow2(int t) { return __hiloint2double((1023 + t) << 20, 0); }
// 1 / sqrt(x) of a normal x > 0, taken to [1, 4) by a power of four
__device__ __forceinline__ double tq_rsqrt(double x) {
  const int t = -((((__double2hiint(x) >> 20) & 0x7ff) - 1023) >> 1);
  return rsqrt_r(x * tq_pow2(2 * t)) * tq_pow2(t);
}

// entries of the buffers beside the slice: parts of the sums (two sets in turn), totals, R's column
__host__ __device__ inline size_t tq_head(int n) { return 4 * (size_t)n; }

__global__ void __launch_bounds__(TQ_NT, 1) k_tall_qr(zd* A, int m, int n, int dagger, zd* R, int* status, int* count,
                                                      int resident, int stall) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ unsigned long long s_cbar;
  __shared__ int s_gave_up;
  __shared__ double s_left, s_inv;
  __shared__ int s_state;  // of a pass: 0 again, 1 done, 2 nothing there
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ca = (int)gridDim.x, rank = (int)cta_rank_in_cluster();
  zd* part = (zd*)sm;           // [n], two in turn; read by the others
  zd* other = part + n;
  zd* const tot = part + 2 * n; // [n]
  zd* const col = tot + n;      // [n]

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
    a = col + n;
    ld = n | 1;
    for (int x = tid; x < nl * n; x += TQ_NT) a[(x / n) * ld + x % n] = g[x];
  }
  __syncthreads();
  for (int j = 0; j < n && !cb.lost; j++) {
    for (int i = tid; i < n; i += TQ_NT) col[i] = mk<double>(0.0, 0.0);
    int state = 0;
    for (int pass = 0; pass < 3 && state == 0; pass++) {
      // our part of q_i^dag a_j, i < j, and of |a_j|^2: a group of lanes to each
      int G = 32;
      while (G > 4 && ((j + 1) * G > TQ_NT || G >= 2 * nl)) G >>= 1;
      const int gid = tid / G, gl = tid % G, ng = TQ_NT / G;
      for (int i0 = 0; i0 <= j; i0 += ng) {
        if (i0 + (warp * 32) / G > j) break;  // no product for this warp
        const int i = i0 + gid;
        double re = 0.0, im = 0.0;
        if (i <= j)
          for (int r = gl; r < nl; r += G) {
            const zd x = a[r * ld + i], y = a[r * ld + j];
            re = fma(x.im, y.im, fma(x.re, y.re, re));
            im = fma(-x.im, y.re, fma(x.re, y.im, im));
          }
        for (int o = 1; o < G; o <<= 1) {
          re += __shfl_xor_sync(0xffffffffu, re, o);
          im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (i <= j && gl == 0) part[i] = mk<double>(re, im);
      }
      if (!cb.sync()) break;
      // all parts, four lanes to a product
      for (int i0 = 0; i0 <= j; i0 += TQ_NT / 4) {
        if (i0 + warp * 8 > j) break;
        const int i = i0 + tid / 4;
        zd s = mk<double>(0.0, 0.0);
        if (i <= j) {
          if (ca == 1) {
            if ((lane & 3) == 0) s = part[i];
          } else {
            for (int r = lane & 3; r < ca; r += 4) s = cadd(s, *on_cta(&part[i], r));
          }
        }
        for (int o = 1; o < 4; o <<= 1) {
          s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
          s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
        }
        if (i <= j && (lane & 3) == 0) {
          tot[i] = s;
          if (i < j) col[i] = cadd(col[i], s);
        }
      }
      __syncthreads();
      if (warp == 0) {
        double gone = 0.0;
        for (int i = lane; i < j; i += 32) gone += cabs2(tot[i]);
        for (int o = 16; o > 0; o >>= 1) gone += __shfl_xor_sync(0xffffffffu, gone, o);
        const double was = tot[j].re, left = was - gone;
        if (lane == 0) {
          const bool done = left >= 0.25 * was && left >= DBL_MIN;
          const double inv = done ? tq_rsqrt(left) : 0.0;
          s_state = done ? 1 : was > 0.0 ? 0 : 2;
          s_inv = inv;
          s_left = done ? left * inv : 0.0;
        }
      }
      // a_j -= sum_i q_i (q_i^dag a_j), eight lanes to a row
      for (int k0 = 0; k0 < nl; k0 += TQ_NT / 8) {
        if (k0 + warp * 4 >= nl) break;
        const int r = k0 + tid / 8;
        zd s = mk<double>(0.0, 0.0);
        if (r < nl)
          for (int i = tid & 7; i < j; i += 8) cfma(s, a[r * ld + i], tot[i]);
        for (int o = 1; o < 8; o <<= 1) {
          s.re += __shfl_xor_sync(0xffffffffu, s.re, o);
          s.im += __shfl_xor_sync(0xffffffffu, s.im, o);
        }
        if (r < nl && (tid & 7) == 0) a[r * ld + j] = csub(a[r * ld + j], s);
      }
      __syncthreads();
      state = s_state;
      zd* const t = part;
      part = other;
      other = t;
    }
    if (cb.lost) break;
    const double norm = state == 1 ? s_left : 0.0, inv = state == 1 ? s_inv : 0.0;
    for (int r = tid; r < nl; r += TQ_NT) {
      zd v = cscale(a[r * ld + j], inv);
      if (state != 1) v = mk<double>(j == 0 && r0 + r == 0 ? 1.0 : 0.0, 0.0);
      a[r * ld + j] = v;
    }
    if (rank == 0)
      for (int i = tid; i < n; i += TQ_NT) {
        const zd v = i == j ? mk<double>(norm, 0.0) : col[i];  // (zero below the diagonal)
        R[dagger ? (long)j * n + i : (long)i * n + j] = dagger ? cconj(v) : v;
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

struct TallPlan {
  int ca, resident;
  size_t smem;
  long cycles;  // of a pass, by the count of FP64 operations
};

// Cycles of a pass of the last column on ca CTAs by what depends on their number: 64 per FP64
// instruction of a warp, and 3,000 for a barrier and the reads between them.
TallPlan tall_split(int m, int n, int ca) {
  TallPlan p{};
  p.ca = ca;
  const int nl = (m + ca - 1) / ca;
  int g = 32;
  while (g > 4 && (n * g > TQ_NT || g >= 2 * nl)) g >>= 1;
  int lg = 0;
  while ((1 << lg) < g) lg++;
  const long warps = std::min<long>(TQ_NW, ((long)n * g + 31) / 32);
  const long sums = ((long)n * g + TQ_NT - 1) / TQ_NT * ((warps + 3) / 4) * (4L * ((nl + g - 1) / g) + 2 * lg);
  const long rows = (nl + TQ_NT / 8 - 1) / (TQ_NT / 8) * ((std::min(nl, TQ_NT / 8) + 15) / 16) * (4L * ((n + 7) / 8) + 6);
  const long parts = ((long)n * 4 + TQ_NT - 1) / TQ_NT * 2L * (ca / 2 + 4);
  const size_t head = tq_head(n) * sizeof(zd), slice = sizeof(zd) * (size_t)nl * (n | 1);
  p.resident = head + slice <= TQ_SMEM_LIMIT;
  p.smem = head + (p.resident ? slice : 0);
  p.cycles = 64 * (sums + rows + parts) + (ca > 1 ? 5000 : 2000);
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

cudaError_t launch_tall_qr(zd* A, int m, int n, int dagger, zd* R, int* status, int* count, int stall, cudaStream_t s) {
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
  return cudaLaunchKernelEx(&cfg, k_tall_qr, A, m, n, dagger, R, status, count, p.resident, stall);
}

void init_tallqr_attributes() {
  cudaFuncSetAttribute(k_tall_qr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TQ_SMEM_LIMIT);
  cudaFuncSetAttribute(k_tall_qr, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

}  // namespace qlb
