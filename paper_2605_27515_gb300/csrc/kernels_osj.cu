// One-sided (Hestenes) Jacobi SVD of the operator builder in one launch: rows of X (m x n)
// are rotated until every pair is orthogonal to working precision, the rotations are
// accumulated in T (m x m), and the truncation rule and the factors follow (Sec. II.B, exact
// operator ranks of Table I).  Always FP64.
//
// Work split: the columns of X and of T are spread over the CTAs of a cluster.  A rotation
// is the same combination of two rows in every column, so nothing but the pairs' inner
// products crosses CTAs: in a round every CTA forms its part of the m / 2 pairs' four sums,
// publishes them, and after one cluster barrier sums all parts in the same order, so that
// every CTA takes the same decisions with the same bits.  The slices stay in shared memory
// from the first sweep to the factors while they fit (in X and T's own storage otherwise).
//
// What bounds it: an FP64 instruction of a warp holds a partition's pipe for 64 clocks, a
// square root or a division some 20 of them.  The rotation's tangent is therefore formed in
// FP32 and corrected once in FP64 (see below), and a group of 4 to 256 lanes takes a pair, so
// that few pairs of long rows and many of short ones both fill the CTA.
//
// Measured on GB300 with the factors (against one CTA of 1,024 threads over global memory with
// FP64 square roots and divisions, and the factors in a launch of their own): 16 x 16, ten sweeps,
// 0.42 ms (1.30); 16 x 56 0.30 ms (0.86); 36 x 72, 13 sweeps, 2.0 ms (11.9, 14 sweeps);
// 8 x 1,024 0.11 ms (0.52); 20 x 16,384 9.0 ms (110).  Admitting an N = 64 cat, 135 such
// solves of 2 to 43 rows, 9.9 ms on the device, and the QRs of its 65 tall matrices
// (kernels_tallqr.cu), 2.8 ms: 47 ms before, 22 now.

#include <algorithm>

#include "cluster.cuh"

namespace qlb {

namespace {

constexpr int OSJ_NT = 256;
constexpr int OSJ_NW = OSJ_NT / 32;
constexpr int OSJ_MAX_M = 512;                    // rows the one-launch kernel takes at most
constexpr size_t OSJ_SMEM_LIMIT = 200 * 1024;

// double times 2^k to float and back, in integer arithmetic: the conversions of the FP64 pipe
// cost its 64 clocks a warp each.  Truncated; zero below FP32's normal range, infinite above.
__device__ __forceinline__ float osj_to_f(double v, int k) {
  const unsigned hi = (unsigned)__double2hiint(v);
  const int ev = (int)((hi >> 20) & 0x7ff);
  const int e = ev ? ev + k - 896 : 0;  // zero (and subnormal) stays zero whatever k
  const unsigned b = (hi & 0x80000000u) | ((unsigned)e << 23) | ((hi & 0xfffffu) << 3) | ((unsigned)__double2loint(v) >> 29);
  return __uint_as_float(e <= 0 ? 0u : e >= 255 ? (hi & 0x80000000u) | 0x7f800000u : b);
}
__device__ __forceinline__ double osj_to_d(float f) {
  const unsigned b = __float_as_uint(f);
  const unsigned hi = (b & 0x80000000u) | (((b >> 3) & 0x0fffffffu) + (896u << 20));
  return (b & 0x7f800000u) == 0u ? 0.0 : __hiloint2double((int)hi, (int)(b << 29));
}
// v 2^k for a normal result (zero below)
__device__ __forceinline__ double osj_scale(double v, int k) {
  const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
  return !e || e + k <= 0 ? 0.0 : __hiloint2double(hi + k * (1 << 20), __double2loint(v));
}

__device__ __forceinline__ int osj_player(int pos, int round, int np) {
  if (pos == 0) return 0;
  const int x = pos - 1 + round;
  return 1 + (x >= np - 1 ? x - (np - 1) : x);
}

// (rows 0..m-1 of) a column slice: nl columns of X from j0, ml columns of T from t0
struct OsjSlice {
  zd* x;
  zd* t;
  long ldx, ldt;
  int j0, nl, t0, ml;
};

// Order of the rows by squared norm w (m entries; ties to the lower row) and the step's
// truncation rule.  On return w[j] is the j-th singular value, ws[j] its reciprocal (0 for 0),
// perm[j] its row.  Called by the CTA.
__device__ int osj_rule(double* w, double* ws, int* perm, int* s_k, int m, double tol, int cap, double gap) {
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    const long long li = __double_as_longlong(w[i]);  // squared norms order like their bit patterns
    int r = 0;
    for (int j = 0; j < m; j++) {
      const long long lj = __double_as_longlong(w[j]);
      r += lj > li || (lj == li && j < i);
    }
    perm[r] = i;
    ws[r] = w[i];
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double total, kept;
    const int k = truncation_count(ws, m, tol, cap > 0 ? cap : m, gap, total, kept);
    if (threadIdx.x == 0) *s_k = total > 0 ? k : 1;
  }
  __syncthreads();
  for (int r = threadIdx.x; r < m; r += blockDim.x) {
    const double s = ::sqrt(ws[r]);
    w[r] = s;
    ws[r] = s > 0 ? 1.0 / s : 0.0;
  }
  __syncthreads();
  return *s_k;
}

// our slice's part of the factors: R[j, :] = X[perm_j, :] / s_j^r_unscale,
// U[i, j] = conj(T[perm_j, i]) * s_j^u_scale; with X the rows of A^dag = T^dag X (A = X^dag T)
// R[j, :] = T[perm_j, :], U[i, j] = conj(X[perm_j, i])
__device__ void osj_write_r(const OsjSlice& c, const double* sv, const double* inv, const int* perm, int m, int n, int k,
                            const OsjOut& o) {
  if (o.dagger) {
    for (long x = threadIdx.x; x < (long)k * c.ml; x += blockDim.x) {
      const int j = (int)(x / c.ml), i = (int)(x - (long)j * c.ml);
      o.Rr[(long)j * m + c.t0 + i] = c.t[perm[j] * c.ldt + i];
    }
    return;
  }
  for (long x = threadIdx.x; x < (long)k * c.nl; x += blockDim.x) {
    const int j = (int)(x / c.nl), i = (int)(x - (long)j * c.nl);
    zd v = c.x[perm[j] * c.ldx + i];
    if (o.r_unscale) v = sv[j] > 0 ? cscale(v, inv[j]) : mk<double>(0, 0);
    o.Rr[(long)j * n + c.j0 + i] = v;
  }
}
__device__ void osj_write_u(const OsjSlice& c, const double* sv, const int* perm, int k, const OsjOut& o) {
  if (o.dagger) {
    for (long x = threadIdx.x; x < (long)c.nl * k; x += blockDim.x) {
      const int i = (int)(x / k), j = (int)(x - (long)i * k);
      o.U[(long)(c.j0 + i) * k + j] = cconj(c.x[perm[j] * c.ldx + i]);
    }
    return;
  }
  for (long x = threadIdx.x; x < (long)c.ml * k; x += blockDim.x) {
    const int i = (int)(x / k), j = (int)(x - (long)i * k);
    zd v = cconj(c.t[perm[j] * c.ldt + i]);
    if (o.u_scale) v = cscale(v, sv[j]);
    o.U[(long)(c.t0 + i) * k + j] = v;
  }
}

struct __align__(16) PairSums {
  double v[4];  // |x_p|^2, |x_q|^2, Re and Im of x_p . conj(x_q)
};

// Lanes of a pair: as many as fill the CTA, at most twice the slice's width.
__host__ __device__ inline int osj_lanes(int m, int width) {
  const int pairs = (m + 1) / 2;
  int g = OSJ_NT;
  while (g > 4 && (pairs * g > OSJ_NT || g >= 2 * width)) g >>= 1;
  return g;
}

// dynamic shared memory: parts of the sums (two sets in turn), the rule's arrays, the slice
__host__ __device__ inline size_t osj_part_count(int m, int g) {
  return (size_t)((m + 1) / 2) * (g > 32 ? g / 32 : 1);
}
__host__ __device__ inline size_t osj_head_bytes(int m, int g) {
  return 2 * osj_part_count(m, g) * sizeof(PairSums) + (((size_t)m * (2 * sizeof(double) + sizeof(int)) + 15) & ~(size_t)15);
}
__host__ __device__ inline int osj_ld(int n, int m, int ca) { return ((n + ca - 1) / ca + (m + ca - 1) / ca) | 1; }

// sweeps_out: the sweeps run, -1 when max_sweeps did not do, -2 when a bounded wait gave up
__global__ void __launch_bounds__(OSJ_NT, 1) k_osj(zd* X, int m, int n, zd* T, int max_sweeps, int* sweeps_out,
                                                   int resident, OsjOut out) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ unsigned long long s_cbar;
  __shared__ double s_f2[OSJ_NW];
  __shared__ double s_mine;  // our part of ||X||_F^2; read by the others
  __shared__ unsigned s_mc, s_ms;
  __shared__ int s_k, s_gave_up;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ca = (int)gridDim.x, rank = (int)cta_rank_in_cluster();
  const int wn = (n + ca - 1) / ca, wm = (m + ca - 1) / ca;
  const int G = osj_lanes(m, wn + wm), GW = G < 32 ? G : 32, nsub = G > 32 ? G / 32 : 1;
  const int pairs = (m + 1) / 2, np = 2 * pairs;
  PairSums* const part = (PairSums*)sm;  // [2][pairs][nsub]; read by the others
  double* const w = (double*)(part + 2 * pairs * nsub);
  double* const ws = w + m;
  int* const perm = (int*)(ws + m);

  if (tid == 0) {
    s_gave_up = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&s_cbar)),
                 "r"(ca + (out.stall == rank + 1))
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // once, with every CTA of the cluster: the barrier above is set up
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  ClusterBarrier cb{&s_cbar, &s_gave_up, ca, 0u, false};

  OsjSlice c;
  c.j0 = min(n, rank * wn);
  c.nl = min(n, c.j0 + wn) - c.j0;
  c.t0 = min(m, rank * wm);
  c.ml = min(m, c.t0 + wm) - c.t0;
  if (resident) {
    c.ldx = c.ldt = osj_ld(n, m, ca);
    c.x = (zd*)(sm + osj_head_bytes(m, G));
    c.t = c.x + c.nl;
  } else {
    c.ldx = n;
    c.ldt = m;
    c.x = X + c.j0;
    c.t = T + c.t0;
  }
  double f2 = 0.0;
  for (int p = warp; p < m; p += OSJ_NW) {
    for (int j = lane; j < c.nl; j += 32) {
      const zd v = X[(long)p * n + c.j0 + j];
      f2 += cabs2(v);
      if (resident) c.x[p * c.ldx + j] = v;
    }
    for (int j = lane; j < c.ml; j += 32) c.t[p * c.ldt + j] = mk<double>(c.t0 + j == p ? 1.0 : 0.0, 0.0);
  }
  for (int o = 16; o > 0; o >>= 1) f2 += __shfl_xor_sync(0xffffffffu, f2, o);
  if (lane == 0) s_f2[warp] = f2;
  __syncthreads();
  if (tid == 0) {
    double s = s_f2[0];
    for (int i = 1; i < OSJ_NW; i++) s += s_f2[i];
    s_mine = s;
    s_mc = s_ms = 0u;
  }
  cb.sync();
  f2 = 0.0;
  for (int r = 0; r < ca && !cb.lost; r++) f2 += *on_cta(&s_mine, r);

  // A pair is rotated only when |x_p . x_q| exceeds both ~sqrt(n) eps |x_p| |x_q| (a length-n
  // dot product carries that much rounding) and 1e-31 ||X||_F^2: without the absolute floor, the
  // excess rows of a rank-deficient matrix keep rotating rounding noise forever.
  const bool usable = ::isfinite(f2) && f2 > 0.0;
  const float rel = 2.220446e-16f * fmaxf(8.f, 4.f * sqrtf((float)n));
  const double thr = 1e-31 * f2;
  const int gid = tid / G, gl = tid % G, ng = OSJ_NT / G;
  const int sub = gl / 32, base = lane & ~(GW - 1);
  int sweep = 0;
  bool converged = !usable || m <= 1;
  for (int par = 0; !converged && !cb.lost && sweep < max_sweeps; sweep++) {
    float mc = 0.f, ms = 0.f;
    for (int round = 0; round < np - 1; round++, par ^= 1) {
      PairSums* const mine = part + par * pairs * nsub;
      for (int k0 = 0; k0 < pairs; k0 += ng) {
        if (k0 + (warp * 32) / G >= pairs) break;  // no pair for this warp
        const int k = k0 + gid;
        double a = 0, b = 0, gr = 0, gi = 0;
        if (k < pairs) {
          const int p = osj_player(k, round, np), q = osj_player(np - 1 - k, round, np);
          if (p < m && q < m) {
            const zd* xp = c.x + min(p, q) * c.ldx;
            const zd* xq = c.x + max(p, q) * c.ldx;
            for (int j = gl; j < c.nl; j += G) {
              const zd u = xp[j], v = xq[j];
              a = fma(u.im, u.im, fma(u.re, u.re, a));
              b = fma(v.im, v.im, fma(v.re, v.re, b));
              gr = fma(u.im, v.im, fma(u.re, v.re, gr));
              gi = fma(-u.re, v.im, fma(u.im, v.re, gi));
            }
          }
        }
        // four sums over the group's lanes, the first two exchanges also splitting them
        const bool h1 = lane & 1, h2 = lane & 2;
        double s0 = h1 ? b : a, s1 = h1 ? gi : gr;
        s0 += __shfl_xor_sync(0xffffffffu, h1 ? a : b, 1);
        s1 += __shfl_xor_sync(0xffffffffu, h1 ? gr : gi, 1);
        double v = h2 ? s1 : s0;
        v += __shfl_xor_sync(0xffffffffu, h2 ? s0 : s1, 2);
        for (int o = 4; o < GW; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (k < pairs && (gl & 31) < 4) mine[k * nsub + sub].v[lane & 3] = v;
      }
      if (!cb.sync()) break;
      for (int k0 = 0; k0 < pairs; k0 += ng) {
        if (k0 + (warp * 32) / G >= pairs) break;
        const int k = k0 + gid;
        int p = m, q = m;
        if (k < pairs) {
          p = osj_player(k, round, np);
          q = osj_player(np - 1 - k, round, np);
          if (p > q) {
            const int x = p;
            p = q;
            q = x;
          }
        }
        // all parts, summed alike in every warp and CTA: lane l of a group has component l & 3
        double v = 0.0;
        if (q < m)
          for (int i = (lane & (GW - 1)) >> 2; i < ca * nsub; i += GW / 4) {
            const int r = i / nsub;
            v += on_cta(&mine[k * nsub + (i - r * nsub)], r)->v[lane & 3];
          }
        for (int o = 4; o < GW; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        const double a = sget(v, base), b = sget(v, base | 1), gr = sget(v, base | 2), gi = sget(v, base | 3);
        // Scaled by a power of two that takes the larger squared norm to [1, 2), the decision and
        // the rotation's tangent in FP32.
        const long long am = max(__double_as_longlong(a), __double_as_longlong(b));
        const int sk = 1023 - (int)(am >> 52);
        const double dd = a - b;
        const float df = osj_to_f(dd, sk), fr = osj_to_f(gr, sk), fi = osj_to_f(gi, sk);
        const float f2x = fmaf(fr, fr, fi * fi);
        const float gm = fmaxf(::fabsf(fr), ::fabsf(fi));
        // |g| without its square's underflow
        const float fx = f2x > 1e-30f ? sqrtf(f2x) : gm * sqrtf(fmaf(fr / gm, fr / gm, (fi / gm) * (fi / gm)));
        const float ra = rsqrtf(osj_to_f(a, sk)), rb = rsqrtf(osj_to_f(b, sk));
        const float cs = fx * ra * rb;  // infinite for a norm below FP32's range
        if (!(q < m && gm > 0.f && cs > rel && fx > osj_to_f(thr, sk))) continue;
        // The rotation [[c, -sp], [conj(sp), c]] with sp = c z zeroes g + z (a - b) - z^2 conj(g).
        // z from FP32, then one Newton step in FP64, whose derivative is real at the root and
        // needs FP32 only: what is left of the coupling is ~1e-13 of it (~1e-7 without the step,
        // a sweep more in most solves of up to 16 rows).
        const float h = fmaf(0.5f, ::fabsf(df), sqrtf(fmaf(0.25f * df, df, f2x)));
        const float iz = __fdividef(df <= 0.f ? 1.f : -1.f, h);
        const float z0r = fr * iz, z0i = fi * iz;
        const double D = osj_scale(dd, sk), Gr = osj_scale(gr, sk), Gi = osj_scale(gi, sk);
        double zr = osj_to_d(z0r), zi = osj_to_d(z0i);
        const double wr = fma(-zi, Gi, fma(-zr, Gr, D)), wi = fma(zr, Gi, -zi * Gr);
        const double er = fma(-zi, wi, fma(zr, wr, Gr)), ei = fma(zi, wr, fma(zr, wi, Gi));
        const double dz = osj_to_d(__fdividef(-1.f, fmaf(-2.f, fmaf(z0r, fr, z0i * fi), df)));
        zr = fma(er, dz, zr);
        zi = fma(ei, dz, zi);
        // 1 / sqrt(1 + |z|^2): FP32 seed and one third-order step
        const double w1 = fma(zi, zi, fma(zr, zr, 1.0));
        const double y = osj_to_d(rsqrtf(fmaf(z0i, z0i, fmaf(z0r, z0r, 1.f))));
        const double e = fma(-w1 * y, y, 1.0);
        const double cc = fma(y * e, fma(0.375, e, 0.5), y);
        const double sr = cc * zr, si = cc * zi;
        // the largest cosine met and the largest tangent of the sweep
        mc = fmaxf(mc, fminf(cs, 1.f));
        ms = fmaxf(ms, sqrtf(fmaf(z0r, z0r, z0i * z0i)));
        auto rotate = [&](zd* xp, zd* xq, int len) {
          for (int j = gl; j < len; j += G) {
            const zd u = xp[j], t = xq[j];
            xp[j] = mk<double>(fma(si, t.im, fma(-sr, t.re, cc * u.re)), fma(-si, t.re, fma(-sr, t.im, cc * u.im)));
            xq[j] = mk<double>(fma(si, u.im, fma(sr, u.re, cc * t.re)), fma(-si, u.re, fma(sr, u.im, cc * t.im)));
          }
        };
        if (resident) {
          rotate(c.x + p * c.ldx, c.x + q * c.ldx, c.nl + c.ml);  // T's slice follows X's
        } else {
          rotate(c.x + p * c.ldx, c.x + q * c.ldx, c.nl);
          rotate(c.t + p * c.ldt, c.t + q * c.ldt, c.ml);
        }
      }
      __syncthreads();
    }
    if (cb.lost) break;
    mc = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(mc)));
    ms = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(ms)));
    if (lane == 0 && mc > 0.f) {
      atomicMax(&s_mc, __float_as_uint(mc));
      atomicMax(&s_ms, __float_as_uint(ms));
    }
    __syncthreads();
    mc = __uint_as_float(s_mc);
    ms = __uint_as_float(s_ms);
    __syncthreads();
    if (tid == 0) s_mc = s_ms = 0u;
    // a sweep that rotated nothing, or whose rotations can have refilled the couplings they met
    // by no more than the largest sine times the largest cosine of the sweep, and left no more
    // than the tangent's error
    converged = mc == 0.f || mc * fmaxf(ms, 1e-12f) * (float)m < 0.1f * rel;
  }

  // row norms, truncation rule (alike in every CTA), our columns of the factors
  if (!cb.lost) {
    for (int p = warp; p < m; p += OSJ_NW) {
      double acc = 0;
      for (int j = lane; j < c.nl; j += 32) acc += cabs2(c.x[p * c.ldx + j]);
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) ws[p] = acc;  // read by the others
    }
    if (cb.sync())
      for (int p = tid; p < m; p += OSJ_NT) {
        double acc = 0;
        for (int r = 0; r < ca; r++) acc += *on_cta(&ws[p], r);
        w[p] = acc;
      }
  }
  const bool gave_up = cb.leave();
  if (rank == 0 && tid == 0) *sweeps_out = gave_up ? -2 : converged ? max(1, sweep) : -1;
  if (gave_up) return;  // no factors
  const int k = osj_rule(w, ws, perm, &s_k, m, out.tol, out.cap, out.gap);
  if (rank == 0 && tid == 0) *out.k_out = k;
  osj_write_r(c, w, ws, perm, m, n, k, out);
  if ((out.U == X || out.U == T) && !resident) {  // U over what R was read from: behind everyone's read
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  }
  osj_write_u(c, w, perm, k, out);
}

// Row norms, rule and factors behind the rounds of separate launches.  One CTA.
__global__ void __launch_bounds__(OSJ_NT) k_osj_finish(zd* X, int m, int n, zd* T, OsjOut out) {
  extern __shared__ __align__(16) unsigned char sm[];
  double* const w = (double*)sm;
  double* const ws = w + m;
  int* const perm = (int*)(ws + m);
  __shared__ int s_k;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int i = warp; i < m; i += nw) {
    double acc = 0;
    for (int j = lane; j < n; j += 32) acc += cabs2(X[(long)i * n + j]);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) w[i] = acc;
  }
  const int k = osj_rule(w, ws, perm, &s_k, m, out.tol, out.cap, out.gap);
  const OsjSlice c{X, T, n, m, 0, n, 0, m};
  if (threadIdx.x == 0) *out.k_out = k;
  osj_write_r(c, w, ws, perm, m, n, k, out);
  __syncthreads();  // U may lie over X or T
  osj_write_u(c, w, perm, k, out);
}

// CTAs (a power of two), whether the slices fit in shared memory, and its size
struct OsjPlan {
  int ca;
  bool resident;
  size_t smem;
  long cycles;  // of a round, by the count of FP64 operations
};

// Cycles of a round on ca CTAs: a warp takes 64 per FP64 instruction, 8 per element of X for
// the sums, 12 per element of X and T for the rotation, ~35 for the rotation's scalars; the
// barrier, the reads between CTAs and what is not FP64 are counted as 2,000 (1,000 on one CTA),
// the fastest over the SVDs of an N = 64 cat's admission (3,500: 2 % slower).
OsjPlan osj_split(int m, int n, int ca) {
  OsjPlan p{};
  p.ca = ca;
  const int wn = (n + ca - 1) / ca, wm = (m + ca - 1) / ca;
  const int g = osj_lanes(m, wn + wm), pairs = (m + 1) / 2;
  const size_t head = osj_head_bytes(m, g), rows = sizeof(zd) * (size_t)m * osj_ld(n, m, ca);
  p.resident = head + rows <= OSJ_SMEM_LIMIT;
  p.smem = head + (p.resident ? rows : 0);
  const long warps = ((long)pairs * g + 31) / 32;
  p.cycles = 64 * ((warps + 3) / 4) * (8L * ((wn + g - 1) / g) + 12L * ((wn + wm + g - 1) / g) + 35) +
             (ca > 1 ? 2000 : 1000);
  return p;
}
OsjPlan osj_plan(int m, int n) {
  OsjPlan best = osj_split(m, n, 1);
  for (int ca = 2; ca <= FC_MAX_C; ca *= 2) {
    const OsjPlan p = osj_split(m, n, ca);
    if (p.cycles < best.cycles || (p.resident && !best.resident)) best = p;
  }
  return best;
}

}  // namespace

// One launch over a cluster, unless a launch per round with a CTA to every pair is faster: that
// takes 10 n + 6 m cycles for its pair and ~12,000 for the launch, the block sums and the
// square roots.
bool osj_serves(int m, int n) {
  if (m > OSJ_MAX_M) return false;
  return osj_plan(m, n).cycles <= 10L * n + 6L * m + 12000;
}

cudaError_t launch_osj(zd* X, int m, int n, zd* T, int max_sweeps, int* sweeps_out, const OsjOut& out, cudaStream_t s) {
  const OsjPlan p = osj_plan(m, n);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.ca, 1, 1);
  cfg.blockDim = dim3(OSJ_NT, 1, 1);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = p.ca;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_osj, X, m, n, T, max_sweeps, sweeps_out, (int)p.resident, out);
}

cudaError_t launch_osj_finish(zd* X, int m, int n, zd* T, const OsjOut& out, cudaStream_t s) {
  const size_t smem = (size_t)m * (2 * sizeof(double) + sizeof(int));
  if (smem > 48 * 1024) cudaFuncSetAttribute(k_osj_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_osj_finish<<<1, OSJ_NT, smem, s>>>(X, m, n, T, out);
  return cudaGetLastError();
}

void init_osj_attributes() {
  cudaFuncSetAttribute(k_osj, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OSJ_SMEM_LIMIT);
  cudaFuncSetAttribute(k_osj, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

}  // namespace qlb
