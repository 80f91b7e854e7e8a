// Range basis of a zip-up bond without an eigen-solve, for planned sizes up to 256.
//
// The zip-up (Sec. III.A MPO.MPS product, Sec. V.A) cuts its bonds at a relative weight
// tol * zip_tol_factor, far below the final truncation: it needs an orthonormal U (n x r)
// with || (1 - U U^dag) M ||_F^2 <= tol' ||M||_F^2, not the eigen-decomposition of
// G = M M^dag.  This kernel builds U by column-pivoted Gram-Schmidt on the columns of G,
// each new basis vector re-orthogonalised against the basis so far (a second time when
// the first pass cancels more than three quarters of the squared norm: "twice is enough",
// Giraud, Langou & Rozloznik 2005).
//
// With W = (1 - Q Q^dag) G the residual of G's columns after j basis vectors, the
// discarded weight is Tr((1 - Q Q^dag) G) = sum_k Re W_kk, and the columns already chosen
// contribute zero, so the weight is known at every step from the diagonal of the columns
// still open.  Step j:
//   (a) stop with r = j when that weight <= tol * Tr G;
//   (b) stop with r = j when the largest residual column norm, or that column's residual
//       after re-orthogonalisation, is at the rounding level of the working precision
//       (<= eps ||G||_F): only rounding is left;
//   (c) at j = cap the cut would drop real weight: the best rank-cap subspace is the top
//       eigenvectors of G, so the kernel sets the gate and leaves the bond to the
//       eigen-solve launched behind it (which runs only when gated in);
//   else the column p with the largest residual norm, to FP32's precision (ties go to the lower
//   column), becomes
//       q_j = normalise((1 - Q Q^dag) w_p)
//   and every open column k loses its component: w_k -= q_j (q_j^dag w_k).
//
// Work split: the columns of W, and with them the basis vectors that they become, are
// spread over C CTAs of a cluster (range_ctas).  A step's O(n^2) column sweep is local;
// between CTAs go the pivot candidates, the pivot column and the re-orthogonalisation's
// partial sums (summed over the CTAs in a fixed order, deterministic).  One CTA
// spends a step on ~10 n^2 FMAs at two FP64 operations per clock; with C of them a step
// is bound by its two or three barriers and the latency of what is read between them.
//
// Measured on GB300, a cold G of rank r with weights over 1e-12 (against one CTA of 512
// threads sweeping all columns, the kernel of the sizes above 256): FP64 n = 32, r = 16
// 102 us (360), n = 64, r = 32 268 us (987), n = 128, r = 64 0.85 ms (4.47); double-float
// 81 us (124), 229 us (348), 0.72 ms (2.25).  FP64 runs on four warps instead of eight, with
// its comparisons off the FP64 pipe (n = 64 333 us and n = 128 0.94 ms on eight): what every
// warp computes for itself held the pipes for ~6,000 of a step's ~20,000 cycles.
//
// R = double (the FP64 form) or df64 (the mixed forms).  G and U are FP64 in both.

#include <algorithm>

#include "cluster.cuh"

namespace qlb {

namespace {

template <typename R>
struct RangeEps;
template <>
struct RangeEps<double> {
  static constexpr double v = 2.220446049250313e-16;
};
template <>
struct RangeEps<df64> {
  static constexpr double v = 3.552713678800501e-15;  // 2^-48
};

constexpr int RB_LOCAL = 48;  // columns of one CTA at most
// Up to this many parts of rows, on up to eight CTAs, every CTA reads and sums all of them;
// beyond, each sums a slice of the rows and hands it on (a barrier and a trip more): FP64 n = 32,
// eight CTAs, 102 us against 110, n = 64 266 against 274; double-float n = 64, four CTAs, 227
// against 239, but n = 128, eight CTAs, 757 against 707.
constexpr int RB_ALL_PARTS = 512;
constexpr int RB_ALL = 8;

// CTAs that work on a problem of size n (a power of two).  One CTA needs no exchange (three
// barriers and four reads across CTAs, ~5,000 cycles a step) and takes ~5 n^2 cycles for the
// sweep in FP64, an eighth of that in double-float.  The lines lie where the times of two
// splits cross (r = n / 2): FP64 n = 24 92 us on one CTA and 88 on four, n = 32 143 on one,
// 114 on four, 110 on eight, n = 64 337, 274, 270 on 4, 8, 16, n = 80 511 on eight, 432 on
// 16; double-float n = 40 131 on one, 130 on eight, n = 64 270, 247, 239, 272 on 1, 2, 4, 8,
// n = 80 530, 448, 368, 383, n = 128 724 on four, 707 on eight.
template <typename R>
__host__ __device__ inline int range_ctas(int n) {
  if (std::is_same<R, double>::value) return n <= 24 ? 1 : n <= 64 ? 8 : 16;
  return n <= 48 ? 1 : n <= 96 ? 4 : n <= 128 ? 8 : 16;
}

// a pivot candidate (key: FP32 bits of the squared residual norm above the complement of
// the column's index, 0 for none) and the residual weight of the open columns
template <typename R>
struct __align__(16) Candidate {
  unsigned lo, hi;
  R best, weight;
};

template <typename R, bool GRP>
__global__ void __launch_bounds__(ClThreads<R>::v, 1) k_range(EigDesc e, int* d, double* prof,
                                                 const EigDesc* __restrict__ grp) {
  constexpr int NT = ClThreads<R>::v, NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  if constexpr (GRP) {  // grouped launch: one cluster per member (blockIdx.y; the cluster spans x)
    e = grp[blockIdx.y];
    d = e.dims;
  }
  const int n = dev_eval(e.n, d);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cta_rank_in_cluster();
  if (n <= 0) {
    if (rank == 0 && tid == 0) {
      d[e.dim_out] = 0;
      if (e.gate) *e.gate = 0;
    }
    return;
  }
  const int ca = range_ctas<R>(n);
  int cap = dev_eval(e.cap, d);
  if (cap < 1) cap = 1;
  const R zero = pzero(R());
  typedef Candidate<R> Cand;
  // (raw storage: double-float has a constructor)
  __shared__ __align__(16) unsigned char v_raw[FC_MAX_N * sizeof(cx<R>)];
  __shared__ __align__(16) unsigned char y_raw[2 * FC_MAX_N * sizeof(cx<R>)];
  __shared__ __align__(16) unsigned char z_raw[32 * sizeof(cx<R>)];
  __shared__ __align__(16) unsigned char c_raw[RB_LOCAL * sizeof(cx<R>)];
  __shared__ __align__(16) unsigned char part_raw[NW * sizeof(Cand)];
  __shared__ __align__(16) unsigned char pub_raw[2 * sizeof(Cand)];
  __shared__ __align__(16) unsigned char red_raw[NW * 2 * sizeof(R)];
  __shared__ __align__(16) unsigned char sums_raw[2 * sizeof(R)];
  cx<R>* const s_v = (cx<R>*)v_raw;      // the pivot column, then the new basis vector (a copy in every CTA)
  cx<R>* s_y = (cx<R>*)y_raw;            // our basis vectors' part of Q Q^dag v, two in turn; read by the others
  cx<R>* const s_z = (cx<R>*)z_raw;      // our slice of the projected column; read by the others
  cx<R>* const s_c = (cx<R>*)c_raw;      // q_i^dag v of our basis vectors
  Cand* const s_part = (Cand*)part_raw;  // per warp
  Cand* const s_pub = (Cand*)pub_raw;    // ours, two in turn; read by the others
  R* const s_red = (R*)red_raw;
  R* const s_sums = (R*)sums_raw;        // trace and squared norm of our columns; read by the others
  __shared__ unsigned char s_done[RB_LOCAL];
  __shared__ short s_slot[RB_LOCAL], s_idx[RB_LOCAL];  // our basis vectors: column slot, index j
  __shared__ unsigned long long s_cbar;
  __shared__ int s_bad, s_gave_up;

  if (tid == 0) {
    s_bad = 0;
    s_gave_up = 0;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&s_cbar)),
                 "r"(ca + (e.stall == rank + 1))
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // once, with every CTA of the cluster: the barrier above is set up
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  if (rank >= ca) return;
  ClusterBarrier cb{&s_cbar, &s_gave_up, ca, 0u, false};

  const int cpb = (n + ca - 1) / ca;  // columns (and rows of a slice) per CTA
  const bool all_rows = ca <= RB_ALL && ca * n <= RB_ALL_PARTS;
  const int k0c = rank * cpb;
  const int ncl = max(0, min(n, k0c + cpb) - k0c);
  cx<R>* W = (cx<R>*)smem_raw;  // our columns, each contiguous
  const zd* G = (const zd*)e.G;

  // power-of-two scale from the trace, then W = G column by column: column k of a Hermitian
  // G is the conjugate of row k
  double trd = 0.0;
  for (int i = tid; i < n; i += NT) trd += ::fabs(G[(long)i * n + i].re);
  for (int o = 16; o > 0; o >>= 1) trd += __shfl_xor_sync(0xffffffffu, trd, o);
  if (lane == 0) ((double*)red_raw)[warp] = trd;
  __syncthreads();
  trd = ((double*)red_raw)[0];
  for (int w = 1; w < NW; w++) trd += ((double*)red_raw)[w];
  const int ex = ::isfinite(trd) && trd > 0.0 ? max(-1000, min(1000, ilogb(trd))) : 0;
  const double up = ldexp(1.0, -ex);
  bool bad = !::isfinite(trd);
  Acc<R> fr_a, tr_a;
  for (int x = tid; x < ncl * n; x += NT) {
    const int lk = x / n, i = x - lk * n;
    const zd g = G[(long)k0c * n + x];
    bad = bad || !::isfinite(g.re) || !::isfinite(g.im);
    const cx<R> w = mk<R>(R(g.re * up), R(i == k0c + lk ? 0.0 : -g.im * up));
    W[x] = w;
    fr_a.mac(w.re, w.re);
    fr_a.mac(w.im, w.im);
    if (i == k0c + lk) tr_a.mac(w.re, from_f(R(), 1.f));
  }
  for (int i = tid; i < RB_LOCAL; i += NT) s_done[i] = 0;
  if (bad) s_bad = 1;
  __syncthreads();
  // sums of two values over the CTA, the same in every thread
  auto cta_sum2 = [&](Acc<R> a, Acc<R> b, R& sa, R& sb) {
    const R h = csum(a, b, 32);
    if (lane < 2) s_red[2 * warp + lane] = h;
    __syncthreads();
    R v = s_red[lane & (2 * NW - 1)];
    for (int o = 2; o < 2 * NW; o <<= 1) v = v + sx(v, o);
    sa = sget(v, 0);
    sb = sget(v, 1);
    __syncthreads();
  };
  R fr, tr;
  cta_sum2(fr_a, tr_a, fr, tr);

  // lanes per column of the sweep: enough warps to fill the SM's four partitions (FP64: one
  // warp each, as every warp-wide FP64 instruction costs the same however many lanes it serves)
  const int want = std::is_same<R, double>::value ? 4 : 8;
  int LG = 32;
  while (LG > 4 && ((cpb * LG + 31) / 32 > want || LG >= 2 * n)) LG >>= 1;
  const int g = tid / LG, gl = tid % LG, ng = NT / LG;
  const int base = lane & ~(LG - 1);
  // One sweep over our open columns: w_k -= q (q^dag w_k) if q; then the candidate with the
  // largest squared residual norm (ties to the lower column) and the residual weight.
  auto column_sweep = [&](const cx<R>* q, int par) {
    unsigned hi = 0, lo = 0;
    R best = zero, wsum = zero;
    for (int kk = 0; kk < ncl; kk += ng) {
      if (kk + (warp * 32) / LG >= ncl) break;  // no column for this warp
      const int k = kk + g;
      const bool act = k < ncl && !s_done[k];
      cx<R>* wk = W + (long)(act ? k : 0) * n;
      cx<R> a = mk<R>(zero, zero);
      if (q) {
        Acc<R> re, im;
        if (act)
          for (int i = gl; i < n; i += LG) {
            const cx<R> x = q[i], w = wk[i];
            re.mac(x.re, w.re);
            re.mac(x.im, w.im);
            im.mac(x.re, w.im);
            im.mac(-x.im, w.re);
          }
        const R h = csum(re, im, LG);
        a.re = sget(h, base);
        a.im = sget(h, base | 1);
      }
      Acc<R> nu, none;
      R dk = zero;
      if (act)
        for (int i = gl; i < n; i += LG) {
          cx<R> w = wk[i];
          if (q) {
            const cx<R> x = q[i];
            w.re = pmac(pmac(w.re, -x.re, a.re), x.im, a.im);
            w.im = pmac(pmac(w.im, -x.re, a.im), -x.im, a.re);
            wk[i] = w;
          }
          nu.mac(w.re, w.re);
          nu.mac(w.im, w.im);
          if (i == k0c + k) dk = w.re;
        }
      const R nuv = sget(csum(nu, none, LG), base);
      const R dkv = sget(dk, base | ((k0c + k) & (LG - 1)));  // the lane of row k
      if (act && gl == 0) {
        const unsigned h2 = __float_as_uint(to_f(nuv)), l2 = 0xffffffffu - (unsigned)(k0c + k);
        if (lo == 0 || h2 > hi || (h2 == hi && l2 > lo)) {
          hi = h2;
          lo = l2;
          best = nuv;
        }
        wsum = wsum + dkv;
      }
    }
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const unsigned who = __ballot_sync(0xffffffffu, hi == mh && lo == ml);
    best = sget(best, __ffs(who) - 1);
    for (int o = LG; o < 32; o <<= 1) wsum = wsum + sx(wsum, o);
    if (lane == 0) {
      Cand c;
      c.lo = ml;
      c.hi = mh;
      c.best = best;
      c.weight = wsum;
      s_part[warp] = c;
    }
    if (ca > 1) {
      __syncthreads();
      if (warp == 0) {
        const Cand c = s_part[lane & (NW - 1)];
        const unsigned h = __reduce_max_sync(0xffffffffu, c.hi);
        const unsigned l = __reduce_max_sync(0xffffffffu, c.hi == h ? c.lo : 0u);
        const unsigned w = __ballot_sync(0xffffffffu, c.hi == h && c.lo == l);
        R ws = c.weight;
        for (int o = 1; o < NW; o <<= 1) ws = ws + sx(ws, o);
        const R bv = sget(c.best, __ffs(w) - 1);
        if (lane == 0) {
          Cand p;
          p.lo = l;
          p.hi = h;
          p.best = bv;
          p.weight = ws;
          s_pub[par] = p;
        }
      }
    }
  };

  if (tid == 0) {
    s_sums[0] = fr;
    s_sums[1] = tr;
  }
  column_sweep(nullptr, 0);
  cb.sync();
  bool any_bad = s_bad != 0;
  if (ca > 1 && !cb.lost) {
    fr = zero;
    tr = zero;
    any_bad = false;
    for (int c = 0; c < ca; c++) {
      fr = fr + *on_cta(&s_sums[0], c);
      tr = tr + *on_cta(&s_sums[1], c);
      any_bad = any_bad || *on_cta(&s_bad, c) != 0;
    }
  }
  // thresholds of the stop tests, as squared norms in the working type
  const R thr_w = R(e.tol) * tr;
  const R floor2 = R(RangeEps<R>::v * RangeEps<R>::v) * fr;
  const R quarter = from_f(R(), 0.25f);
  bool usable = !any_bad && fr > zero;
  double flops = 0.0;  // thread 0 only
  int j = 0, jl = 0;   // basis vectors, ours of them
  bool fallback = false;
  if (usable && !cb.lost) {
    for (int par = 0;; j++, par ^= 1) {
      // the candidates, reduced alike in every warp of every CTA
      Cand c;
      const int ne = ca == 1 ? NW : ca;
      if (ca == 1)
        c = s_part[lane & (NW - 1)];
      else
        c = *on_cta(&s_pub[par], lane & (ca - 1));
      const unsigned h = __reduce_max_sync(0xffffffffu, c.hi);
      const unsigned l = __reduce_max_sync(0xffffffffu, c.hi == h ? c.lo : 0u);
      const unsigned w = __ballot_sync(0xffffffffu, c.hi == h && c.lo == l);
      const R best = sget(c.best, __ffs(w) - 1);
      R wres = c.weight;
      for (int o = 1; o < ne; o <<= 1) wres = wres + sx(wres, o);
      if (j == n || l == 0u) break;  // l = 0: no open column
      if (j >= 1 && (le_nn(wres, thr_w) || le_nn(best, floor2))) break;
      if (j >= cap) {
        fallback = true;
        break;
      }
      const int p = (int)(0xffffffffu - l);
      const int op = p / cpb, lp = p - op * cpb;
      {
        const cx<R>* src = on_cta(W + (long)lp * n, op);
        for (int i = tid; i < n; i += NT) s_v[i] = src[i];
      }
      __syncthreads();
      R nrm2 = best;
      for (int pass = 0; j > 0 && pass < 2; pass++) {
        // c_i = q_i^dag v, a lane group per basis vector of ours
        for (int i0 = 0; i0 < jl; i0 += ng) {
          if (i0 + (warp * 32) / LG >= jl) break;
          const int i = i0 + g;
          Acc<R> re, im;
          if (i < jl) {
            const cx<R>* qi = W + (long)s_slot[i] * n;
            for (int r = gl; r < n; r += LG) {
              const cx<R> x = qi[r], y = s_v[r];
              re.mac(x.re, y.re);
              re.mac(x.im, y.im);
              im.mac(x.re, y.im);
              im.mac(-x.im, y.re);
            }
          }
          const R h2 = csum(re, im, LG);
          if (i < jl && gl == 0) s_c[i].re = h2;
          if (i < jl && gl == 1) s_c[i].im = h2;
        }
        __syncthreads();
        // our part of Q c, two lanes per row
        for (int r0 = 0; r0 < n; r0 += NT / 2) {
          const int row = r0 + tid / 2, half = tid & 1;
          Acc<R> re, im;
          if (row < n)
            for (int i = half; i < jl; i += 2) {
              const cx<R> x = s_c[i], q = W[(long)s_slot[i] * n + row];
              re.mac(x.re, q.re);
              re.mac(-x.im, q.im);
              im.mac(x.re, q.im);
              im.mac(x.im, q.re);
            }
          re.add_from(re, 1);
          im.add_from(im, 1);
          if (row < n && half == 0) {
            const cx<R> y = mk<R>(re.value(), im.value());
            if (ca == 1)
              s_v[row] = csub_r(s_v[row], y);
            else
              s_y[row] = y;
          }
        }
        if (!cb.sync()) break;
        if (ca > 1 && all_rows) {
          // v - the CTAs' parts, every row in every CTA, two lanes per row: one barrier and
          // one trip between CTAs fewer than by slices, for ca n reads (the same sums in the
          // same order)
          for (int r0 = 0; r0 < n; r0 += NT / 2) {
            if (r0 + warp * 16 >= n) break;  // no row for this warp
            const int row = r0 + tid / 2, half = (tid & 1) * (ca / 2);
            cx<R> y[RB_ALL / 2];
#pragma unroll
            for (int c = 0; c < RB_ALL / 2; c++)
              y[c] = c < ca / 2 && row < n ? *on_cta(&s_y[row], half + c) : mk<R>(zero, zero);
#pragma unroll
            for (int o = 1; o < RB_ALL / 2; o <<= 1)
#pragma unroll
              for (int c = 0; c < RB_ALL / 2; c += 2 * o) y[c] = mk<R>(y[c].re + y[c + o].re, y[c].im + y[c + o].im);
            y[0].re = y[0].re + sx(y[0].re, 1);
            y[0].im = y[0].im + sx(y[0].im, 1);
            if (row < n && !(tid & 1)) s_v[row] = csub_r(s_v[row], y[0]);
          }
          __syncthreads();
        } else if (ca > 1) {
          // our slice of rows: v - the CTAs' parts, ca lanes per row
          for (int s0 = 0; s0 < ncl; s0 += NT / ca) {
            const int sr = s0 + tid / ca, sc = tid & (ca - 1), srow = k0c + sr;
            if (s0 + (warp * 32) / ca >= ncl) break;  // no row for this warp
            cx<R> y = mk<R>(zero, zero);
            if (sr < ncl) y = *on_cta(&s_y[srow], sc);
            for (int o = 1; o < ca; o <<= 1) {
              y.re = y.re + sx(y.re, o);
              y.im = y.im + sx(y.im, o);
            }
            if (sr < ncl && sc == 0) s_z[sr] = csub_r(s_v[srow], y);
          }
          if (!cb.sync()) break;
          for (int i = tid; i < n; i += NT) s_v[i] = *on_cta(&s_z[i % cpb], i / cpb);
          __syncthreads();
        }
        s_y = (cx<R>*)y_raw + (s_y == (cx<R>*)y_raw ? FC_MAX_N : 0);
        const R prev = nrm2;
        {
          Acc<R> re, im;
          for (int i = tid; i < n; i += NT) {
            const cx<R> x = s_v[i];
            re.mac(x.re, x.re);
            im.mac(x.im, x.im);
          }
          R sa, sb;
          cta_sum2(re, im, sa, sb);
          nrm2 = sa + sb;
        }
        if (tid == 0) flops += 16.0 * n * j;
        if (le_nn(quarter * prev, nrm2)) break;
      }
      if (cb.lost) break;
      // the pivot's true residual is at the rounding level: what the tracked norms still
      // show is rounding of earlier projections, and the range is complete
      if (j >= 1 && le_nn(nrm2, floor2)) break;
      if (j == 0 && !cb.sync()) break;  // every CTA has read the column that becomes q_0
      {
        const R inv = rsqrt_r(nrm2);
        for (int i = tid; i < n; i += NT) {
          const cx<R> q = mk<R>(s_v[i].re * inv, s_v[i].im * inv);
          s_v[i] = q;
          if (rank == op) W[(long)lp * n + i] = q;
        }
      }
      if (rank == op) {
        if (tid == 0) {
          s_done[lp] = 1;
          s_slot[jl] = (short)lp;
          s_idx[jl] = (short)j;
        }
        jl++;
      }
      __syncthreads();
      column_sweep(s_v, par ^ 1);
      if (tid == 0) flops += 20.0 * n * (n - j - 1);
      if (!cb.sync()) break;
    }
  }
  const bool gave_up = cb.leave();
  let_next_start();
  if (gave_up) usable = fallback = false;  // one unit vector and the flag
  const int r = usable ? j : 1;
  if (rank == 0 && tid == 0) {
    if (gave_up && e.err) atomicOr(e.err, 4);
    if (e.gate) *e.gate = fallback ? 1 : 0;
    if (!fallback) {
      d[e.dim_out] = r;
      if (any_bad && e.err) atomicOr(e.err, 2);
    }
    if (e.solver_stats) {
      atomicAdd(e.solver_stats + 7, 1.0);
      if (fallback) {
        atomicAdd(e.solver_stats + 8, 1.0);
      } else {
        atomicAdd(e.solver_stats + 0, 1.0);
        atomicAdd(e.solver_stats + 2, (double)n);
        atomicAdd(e.solver_stats + 3, (double)r);
        atomicMax((unsigned long long*)(e.solver_stats + 6), (unsigned long long)__double_as_longlong((double)n));
      }
    }
    if (prof) {
      atomicAdd(prof, flops);
      if (!fallback) atomicAdd(prof + QLB_K_COUNT, sizeof(zd) * ((double)n * n + (double)n * r));
    }
  }
  if (fallback) return;
  zd* out = (zd*)e.out;
  auto put = [&](int i, int jj, double re, double im) {
    if (e.out_mode == 0)
      out[(long)i * r + jj] = mk<double>(re, im);
    else if (e.out_mode == 1)
      out[(long)jj * n + i] = mk<double>(re, -im);
  };
  if (!usable) {  // G = 0, non-finite entries or a lost wait: one unit vector
    if (rank == 0)
      for (int i = tid; i < n; i += NT) put(i, 0, i == 0 ? 1.0 : 0.0, 0.0);
    return;
  }
  for (int x = tid; x < jl * n; x += NT) {
    const int q = x / n, i = x - q * n;
    const cx<R> u = W[(long)s_slot[q] * n + i];
    put(i, s_idx[q], (double)u.re, (double)u.im);
  }
}

// dynamic shared memory of a launch for sizes up to n_max
template <typename R>
size_t range_smem(int n_max) {
  int m = 1;
  for (int n = 1; n <= n_max; n++) {
    const int c = range_ctas<R>(n);
    m = std::max(m, ((n + c - 1) / c) * n);
  }
  return (size_t)m * sizeof(cx<R>);
}

constexpr size_t RB_SMEM_LIMIT = 80 * 1024;  // n = 256 over 16 CTAs: 64 KB

template <typename R>
cudaError_t launch_range(int n_max, const EigDesc& e, const int* d_dims, cudaStream_t s, double* prof,
                         const EigDesc* grp, int members) {
  cudaLaunchConfig_t cfg = {};
  const int c = range_ctas<R>(n_max);
  cfg.gridDim = dim3(c, members, 1);
  cfg.blockDim = dim3(ClThreads<R>::v, 1, 1);
  cfg.dynamicSmemBytes = range_smem<R>(n_max);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  if (grp) return cudaLaunchKernelEx(&cfg, k_range<R, true>, e, (int*)d_dims, prof, grp);
  return cudaLaunchKernelEx(&cfg, k_range<R, false>, e, (int*)d_dims, prof, grp);
}

template <typename K>
void range_attr(K* k) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RB_SMEM_LIMIT);
  cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

}  // namespace

size_t zipqr_workspace_elems(int n_max) { return n_max > FC_MAX_N ? zipqr_large_workspace_elems(n_max) : 1; }

// A member of a group launched with the kernel of a larger co-member's planned size needs
// that kernel's workspace for its own planned size.
size_t zipqr_group_workspace_elems(int n_max, int group_n_max) {
  return group_n_max > FC_MAX_N ? zipqr_large_workspace_elems(n_max) : 1;
}

template <typename R>
cudaError_t launch_zipqr(const EigDesc& e, const int* d_dims, cudaStream_t s, void* work, double* prof) {
  if (e.n_max > FC_MAX_N) return launch_zipqr_large<R>(e.n_max, e, d_dims, s, work, prof, nullptr, 1);
  return launch_range<R>(e.n_max, e, d_dims, s, prof, nullptr, 1);
}
template cudaError_t launch_zipqr<double>(const EigDesc&, const int*, cudaStream_t, void*, double*);
template cudaError_t launch_zipqr<df64>(const EigDesc&, const int*, cudaStream_t, void*, double*);

// The range bases of S states' zip-up bonds in one launch (one cluster per member);
// n_max is the largest planned size over the members.
template <typename R>
cudaError_t launch_zipqr_group(int n_max, const EigDesc* d_grp, int S, cudaStream_t s, double* prof) {
  if (S <= 0) return cudaSuccess;
  if (n_max > FC_MAX_N) return launch_zipqr_large<R>(n_max, EigDesc{}, nullptr, s, nullptr, prof, d_grp, S);
  return launch_range<R>(n_max, EigDesc{}, nullptr, s, prof, d_grp, S);
}
template cudaError_t launch_zipqr_group<double>(int, const EigDesc*, int, cudaStream_t, double*);
template cudaError_t launch_zipqr_group<df64>(int, const EigDesc*, int, cudaStream_t, double*);

void init_range_attributes() {
  range_attr(k_range<double, false>);
  range_attr(k_range<double, true>);
  range_attr(k_range<df64, false>);
  range_attr(k_range<df64, true>);
}

}  // namespace qlb
