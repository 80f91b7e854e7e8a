// Truncation eigen-solve of a Hermitian positive semi-definite (Gram) matrix for
// planned sizes up to 256: pivoted Cholesky followed by one-sided Jacobi, spread over
// a thread-block cluster, ending with the truncation decision of the bond it serves.
//
//   1. G = L L^dag with complete (diagonal) pivoting, L of n x r (Higham, "Analysis of
//      the Cholesky decomposition of a semi-definite matrix", 1990).  A pivot is
//      taken while its residual stands above eps times that diagonal entry of G; what
//      is left then is the rounding G itself carries.
//   2. One-sided cyclic Jacobi on the columns of L (Hestenes 1958; Veselic & Hari,
//      "A note on a one-sided Jacobi algorithm", 1989): L V = U Sigma, so that
//      G = U Sigma^2 U^dag.  A pair of columns is rotated while
//      |a_p^dag a_q| > n eps |a_p| |a_q|, which keeps the small eigenvalues and their
//      vectors to the relative accuracy that G's own entries allow.
//   3. Weights, kept count (relative discarded weight, cap, degenerate clusters) and
//      the kept vectors U.
//
// Against a two-sided Jacobi solve (rows and columns of G and the columns of V
// per rotation), a rotation touches two columns once, no eigenvector matrix is
// accumulated, only the r columns above rounding take part, and the pivoted factor is
// already close to orthogonal columns.
//
// The rotation [[c, sp], [-conj(sp), c]] is formed from a complex tangent z held in
// FP32 and c = 1 / sqrt(1 + |z|^2), sp = c z in the working precision: it is unitary to
// the working precision whatever the error of z, which only leaves 1e-7 of the coupling
// for the next sweep.  That keeps square roots and divisions off the FP64 pipe, which
// retires two operations per clock and SM here, so that a warp-wide instruction holds
// it for 64 clocks.
//
// Work split: with C active CTAs the factor's columns form 2 C blocks of b columns.  A
// CTA holds two blocks, rotates the b x b pairs between them (in its first turn of a
// sweep also the pairs inside each block) with one barrier per round of b pairs, then
// hands the blocks on in the round-robin order of Brent & Luk (1985) through
// distributed shared memory: 2 C - 1 exchanges per sweep.  In the
// factorisation a CTA holds n / C rows, one cluster barrier per pivot.  C follows the
// run-time size (pj_ctas), so that a problem takes the same split, and gives the same
// bits, whatever larger size it was launched for; CTAs beyond C leave at once.
//
// Measured on GB300, cold Gram matrices of rank n with weights over 1e-12 (against the
// two-sided Jacobi solves of kernels_eig.cu): FP64 n = 16 192 us (698), n = 32 458 us
// (1,925), n = 64 1.31 ms (6.03), n = 128 4.21 ms (38.8); double-float n = 16 100 us (388),
// n = 32 266 us (1,251), n = 64 0.69 ms (3.83), n = 128 2.05 ms (23.8).  At n = 64 an FP64 round of
// four pairs to a CTA takes 4,700 cycles, ~3,500 of them the FP64 pipe; a double-float
// round 2,100, the latency of its chain.
//
// R = double (the FP64 form) or df64 (the mixed forms); G and the vectors are FP64.

#include <algorithm>

#include "cluster.cuh"

namespace qlb {

namespace {

constexpr int PJ_MAX_NW = 8;  // warps per CTA at most
constexpr int PJ_MAX_N = FC_MAX_N;
constexpr int PJ_MAX_C = FC_MAX_C;
constexpr int PJ_SLOTS = PJ_MAX_N + 2 * PJ_MAX_C;  // columns with the padding of the last block

// CTAs that work on a problem of size n (a power of two).  An FP64 round costs its ~50
// warp-wide instructions at 64 clocks whatever its pairs, so four pairs to a CTA (one warp to
// each partition) is the fastest split until the 16 CTAs of a cluster run out.  In
// double-float a round of n = 24 takes 2,600 cycles on one CTA and an exchange of blocks
// 2,000, so small problems stay on one.
template <typename R>
__host__ __device__ inline int pj_ctas(int n) {
  if (std::is_same<R, double>::value) return n <= 8 ? 1 : n <= 16 ? 2 : n <= 32 ? 4 : n <= 64 ? 8 : 16;
  return n <= 24 ? 1 : n <= 48 ? 4 : n <= 96 ? 8 : 16;
}

// complex elements of one of the two column buffers for a problem of size n
__host__ __device__ inline int pj_region(int n, int c) {
  return 2 * ((n + 2 * c - 1) / (2 * c)) * (n + 1);
}

// ------------------------------------------------------------------ pivoted Cholesky

// The factorisation's own shared memory.  key, d and bad are read by the other CTAs after
// a barrier; key has three sets in turn, as a set is written again only after the
// barrier that follows its reads.
struct __align__(16) FactorSmem {
  unsigned char row[FC_MAX_N * 16];  // the pivot's row of L
  unsigned char d[FC_MAX_N * 8];     // residual diagonal of our rows
  unsigned char floor[FC_MAX_N * 8]; // below it only rounding is left
  unsigned char open[FC_MAX_N];      // our rows not taken as pivots yet
  double red[PJ_MAX_NW];
  unsigned long long cbar;           // every working CTA has arrived
  unsigned key[3];                   // our best pivot candidate
  int bad;
  int gave_up;                       // a CTA lost a wait
};

struct Factor {
  int r;         // columns
  bool bad;      // non-finite entries
  double tr;     // trace of G
  double down;   // the power of two that undoes the scale of L L^dag
};

// Sets up fs, the barrier over the ca CTAs that work on the problem and the one of the
// exchanges (`more`); false for the other CTAs, which leave.  Every thread of every CTA of the
// cluster calls it.
__device__ __forceinline__ bool factor_begin(FactorSmem& fs, unsigned long long* more, int ca, int rank, int stall) {
  if (threadIdx.x == 0) {
    fs.bad = 0;
    fs.gave_up = 0;
    fs.key[0] = fs.key[1] = fs.key[2] = 0u;
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(more)), "r"(1 + (stall == -rank - 1))
                 : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&fs.cbar)), "r"(ca + (stall == rank + 1))
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // once, with every CTA of the cluster: the barriers above are set up
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  return rank < ca;
}

// G = L L^dag with complete (diagonal) pivoting (Higham, "Analysis of the Cholesky
// decomposition of a semi-definite matrix", 1990).  CTA `rank` of ca works on rows
// [rank * rpb, (rank + 1) * rpb): Gl and Ll are theirs, row-major with stride n, G scaled by
// a power of two to a trace in [1, 2).  A pivot is taken while its residual stands above
// eps times its diagonal entry of G.  One barrier per pivot; ends with one.  When a wait is
// lost (cb.lost) there is no factor.
template <typename R>
__device__ Factor pivoted_cholesky(FactorSmem& fs, ClusterBarrier& cb, const zd* G, int n, int ca, int rank,
                                   cx<R>* Gl, cx<R>* Ll) {
  constexpr int NT = ClThreads<R>::v, NW = NT / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const R zero = pzero(R());
  cx<R>* const s_row = (cx<R>*)fs.row;
  R* const s_d = (R*)fs.d;
  R* const s_floor = (R*)fs.floor;
  const int rpb = (n + ca - 1) / ca;
  const int r0 = rank * rpb;
  const int nl = max(0, min(n, r0 + rpb) - r0);
  Factor out{};

  // trace, scale, our rows
  double tr = 0.0;
  for (int i = tid; i < n; i += NT) tr += ::fabs(G[(long)i * n + i].re);
  for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
  if (lane == 0) fs.red[warp] = tr;
  __syncthreads();
  tr = fs.red[0];
  for (int w = 1; w < NW; w++) tr += fs.red[w];
  const bool tr_ok = ::isfinite(tr) && tr > 0.0;
  const int ex = tr_ok ? max(-1000, min(1000, ilogb(tr))) : 0;
  const double up = ldexp(1.0, -ex);
  out.tr = tr;
  out.down = ldexp(1.0, ex);
  const R eps = R(FcEps<R>::pivot);
  bool bad = !::isfinite(tr);
  for (int x = tid; x < nl * n; x += NT) {
    const int li = x / n, j = x - li * n;
    const zd v = G[(long)r0 * n + x];
    bad = bad || !::isfinite(v.re) || !::isfinite(v.im);
    Gl[x] = mk<R>(R(v.re * up), R(v.im * up));
    if (r0 + li == j) {
      const R g = R(v.re * up);
      s_d[li] = g;
      s_floor[li] = g * eps;
      fs.open[li] = 1;
    }
  }
  if (bad) fs.bad = 1;
  __syncthreads();

  // lanes per row: enough warps to fill the SM's four partitions (FP64: one warp each, as
  // every warp-wide FP64 instruction costs the same however many lanes it serves)
  const int want = std::is_same<R, double>::value ? 4 : 8;
  int LR = 32;
  while (LR > 4 && (rpb * LR + 31) / 32 > want) LR >>= 1;
  const int rg = tid / LR, rl = tid % LR, nrg = NT / LR;
  // a candidate pivot: FP32 bits of its residual with the low byte replaced by the
  // index's complement (the pivot is the largest to 2^-15, ties to the lower row)
  auto key_of = [&](int li) -> unsigned {
    const R v = s_d[li];
    const float f = to_f(v);
    if (!fs.open[li] || !(f > FC_TINY) || !(v > s_floor[li])) return 0u;
    return (__float_as_uint(f) & ~0xffu) | (unsigned)(0xff - (r0 + li));
  };
  {
    unsigned key = 0;
    for (int li = tid; li < nl; li += NT) key = max(key, key_of(li));
    key = __reduce_max_sync(0xffffffffu, key);
    if (lane == 0 && key) atomicMax(&fs.key[0], key);
  }
  if (!cb.sync()) return out;
  for (int c = 0; c < ca; c++) out.bad = out.bad || *on_cta(&fs.bad, c) != 0;
  int r = 0;
  if (!out.bad && tr_ok) {
    for (int set = 0; r < n; r++) {
      // the pivot, the same in every thread
      unsigned key = lane < ca ? *on_cta(&fs.key[set], lane) : 0u;
      key = __reduce_max_sync(0xffffffffu, key);
      if (key == 0u) break;
      set = set == 2 ? 0 : set + 1;
      // last read by others before this step's barrier, written next after its own
      if (tid == 0) fs.key[set == 2 ? 0 : set + 1] = 0u;
      const int p = 0xff - (int)(key & 0xffu);
      const int op = p / rpb, lp = p - op * rpb;
      const cx<R>* row = Ll + (long)lp * n;
      const R dp = *on_cta(&s_d[lp], op);  // stays as it is while its row is the pivot's
      if (ca > 1) {
        const cx<R>* rem = on_cta(row, op);
        for (int t = tid; t < r; t += NT) s_row[t] = rem[t];
        row = s_row;
        __syncthreads();
      }
      unsigned best = 0;
      for (int i0 = 0; i0 < nl; i0 += nrg) {
        if (i0 + (warp * 32) / LR >= nl) break;  // no row for this warp
        const R inv = rsqrt_r(dp);
        const int li = i0 + rg;
        const bool act = li < nl;
        Acc<R> cr, ci;
        if (act) {
          const cx<R>* Li = Ll + (long)li * n;
          for (int t = rl; t < r; t += LR) {  // L_it conj(L_pt)
            const cx<R> x = Li[t], y = row[t];
            cr.mac(x.re, y.re);
            cr.mac(x.im, y.im);
            ci.mac(x.im, y.re);
            ci.mac(-x.re, y.im);
          }
        }
        const R ar = csum(cr, ci, LR), ai = sx(ar, 1);
        if (act && rl == 0) {
          cx<R> l = mk<R>(zero, zero);
          if (fs.open[li]) {
            if (r0 + li == p) {
              l.re = dp * inv;
              fs.open[li] = 0;
            } else {
              const cx<R> g = Gl[(long)li * n + p];
              l = mk<R>((g.re - ar) * inv, (g.im - ai) * inv);
              const R dn = pmac(pmac(s_d[li], -l.re, l.re), -l.im, l.im);
              s_d[li] = dn;
              best = max(best, key_of(li));
            }
          }
          Ll[(long)li * n + r] = l;
        }
      }
      best = __reduce_max_sync(0xffffffffu, best);
      if (lane == 0 && best) atomicMax(&fs.key[set], best);
      if (!cb.sync()) return out;
    }
  }
  cb.sync();  // nobody reads another CTA's candidates any more
  out.r = r;
  return out;
}

// the rotations of a sweep in one warp's pairs
struct __align__(16) PjSweep {
  int nrot;
  float mc, ms;  // largest |cos| rotated, largest |s|
  float pad;
};

// ------------------------------------------------------------------ the kernel

template <typename R, bool GRP>
__global__ void __launch_bounds__(ClThreads<R>::v, 1) k_pj(EigDesc e, int* d, double* prof,
                                             const EigDesc* __restrict__ grp) {
  constexpr int NT = ClThreads<R>::v, NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  after_previous();
  if constexpr (GRP) {  // grouped launch: one cluster per member (blockIdx.y; the cluster spans x)
    e = grp[blockIdx.y];
    d = e.dims;
  }
  if (e.gate && *e.gate == 0) return;  // the zip-up range basis already served this bond
  const int n = dev_eval(e.n, d);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cta_rank_in_cluster();
  if (n <= 0) {
    if (rank == 0 && tid == 0) d[e.dim_out] = 0;
    return;
  }
  const int ca = pj_ctas<R>(n);
  int cap = dev_eval(e.cap, d);
  if (cap < 1) cap = 1;
  const R zero = pzero(R());

  __shared__ FactorSmem fs;
  // read by the other CTAs after a barrier; two sets in turn, as a set is written again
  // only after the barrier that follows their reads
  __shared__ PjSweep s_sweep[2][NW];
  __shared__ double s_off[NW];
  __shared__ double s_own[PJ_MAX_N + 2];  // squared norms of our columns
  __shared__ double s_lam[PJ_SLOTS], s_w[PJ_SLOTS];
  __shared__ short s_rank[PJ_SLOTS];
  __shared__ int s_bad, s_k;
  __shared__ __align__(8) unsigned long long s_bar;  // the two blocks of an exchange have arrived

  if (!factor_begin(fs, &s_bar, ca, rank, e.stall)) return;
  ClusterBarrier cb{&fs.cbar, &fs.gave_up, ca, 0u, false};

  // ---- 1. pivoted Cholesky
  const int rpb = (n + ca - 1) / ca;
  cx<R>* buf0 = (cx<R>*)smem_raw;
  cx<R>* buf1 = buf0 + pj_region(n, ca);
  cx<R>* Ll = buf1;
  const Factor f = pivoted_cholesky<R>(fs, cb, (const zd*)e.G, n, ca, rank, buf0, Ll);
  int r = f.r;
  const bool any_bad = f.bad;
  const double tr = f.tr, down = f.down;

  // ---- 2. one-sided Jacobi.  Columns of L go to the CTAs' blocks.
  const int b = max(1, (r + 2 * ca - 1) / (2 * ca));
  const int nc = 2 * b;
  const int ld = n + 1;  // a column and its squared norm
  cx<R>* cur = buf0;
  cx<R>* nxt = buf1;
  // blocks may be sent to us from the barrier below on
  const bool exchanging = ca > 1 && !cb.lost;
  bool armed = false;  // s_bar expects this turn's blocks
  for (int x = tid; x < nc * n && !cb.lost; x += NT) {
    const int i = x / nc, s = x - i * nc;
    const int t = s < b ? rank * b + s : (ca + rank) * b + (s - b);
    const int o = i / rpb;
    cx<R> v = mk<R>(zero, zero);
    if (t < r) v = on_cta(Ll, o)[(long)(i - o * rpb) * n + t];
    cur[(long)s * ld + i] = v;
  }
  if (!cb.lost) cb.sync();  // every CTA has read the factor before its rows become the next column buffer

  // lanes per pair: enough warps to fill the SM's four partitions, as in the factorisation
  const int want = std::is_same<R, double>::value ? 4 : 8;
  int LP = 32;
  while (LP > 4 && ((b * LP + 31) / 32 > want || LP >= 2 * n)) LP >>= 1;
  const int pg = tid / LP, pl = tid % LP, npg = NT / LP;
  const unsigned gmask = (LP == 32 ? 0xffffffffu : ((1u << LP) - 1u) << (lane & ~(LP - 1)));
  const float tol_f = (float)(FcEps<R>::v * (double)(n > 8 ? n : 8));
  auto norm2 = [&](int k) {  // squared norm of column k, in every lane of its group
    Acc<R> re, im;
    if (k < nc)
      for (int i = pl; i < n; i += LP) {
        const cx<R> x = cur[(long)k * ld + i];
        re.mac(x.re, x.re);
        im.mac(x.im, x.im);
      }
    const R h = csum(re, im, LP);
    return h + sx(h, 1);
  };
  int sweep = 0;
  long total_rot = 0;
  int turn = 0;
  bool converged = false, measure = false, pending = false;
  double off2 = 0.0;
  for (; !cb.lost; sweep++) {
    int nrot = 0;
    float mc = 0.f, ms = 0.f;
    double off_l = 0.0;
    for (int k0 = 0; k0 < nc; k0 += npg) {  // squared norms, afresh every sweep
      if (k0 + (warp * 32) / LP >= nc) break;
      const R na = norm2(k0 + pg);
      if (pl == 0 && k0 + pg < nc) *(df64*)(cur + (long)(k0 + pg) * ld + n) = to_df(na);
    }
    __syncthreads();
    for (int o = 0; o < 2 * ca - 1; o++) {
      const int rounds = o == 0 ? nc - 1 : b;
      for (int rd = 0; rd < rounds; rd++) {
        for (int k0 = 0; k0 < b; k0 += npg) {
          if (k0 + (warp * 32) / LP >= b) break;  // no pair for this warp
          const int k = k0 + pg;
          const bool act = k < b;
          int p = 0, q = 0;
          if (act) {
            if (o == 0) {  // round robin over all columns of the CTA
              p = k - 1 + rd;
              p = k == 0 ? 0 : 1 + (p >= nc - 1 ? p - (nc - 1) : p);
              q = nc - 2 - k + rd;
              q = 1 + (q >= nc - 1 ? q - (nc - 1) : q);
            } else {
              p = k;
              q = k + rd;
              q = b + (q >= b ? q - b : q);
            }
          }
          cx<R>* X = cur + (long)p * ld;
          cx<R>* Y = cur + (long)q * ld;
          const df64 na = *(const df64*)(X + n), nb = *(const df64*)(Y + n);
          Acc<R> tr_, ti_;
          if (act)
            for (int i = pl; i < n; i += LP) {
              const cx<R> x = X[i], y = Y[i];
              tr_.mac(x.re, y.re);
              tr_.mac(x.im, y.im);
              ti_.mac(x.re, y.im);
              ti_.mac(-x.im, y.re);
            }
          // from the pair's first two lanes: every lane takes the same decision and rotation
          const float half = to_f(csum(tr_, ti_, LP));
          const float gr = __shfl_sync(0xffffffffu, half, lane & ~(LP - 1));
          const float gi = __shfl_sync(0xffffffffu, half, (lane & ~(LP - 1)) | 1);
          if (measure) {
            if (act && pl == 0) off_l += (double)gr * (double)gr + (double)gi * (double)gi;
            continue;
          }
          // FP32 tangent of the rotation
          const float ra = rsqrtf(na.hi), rb = rsqrtf(nb.hi);
          const float cr = gr * ra * rb, ci = gi * ra * rb;
          const float c2 = fmaf(cr, cr, ci * ci), rcs = rsqrtf(c2), cs = c2 * rcs;
          if (!(act && na.hi > 0.f && nb.hi > 0.f && cs > tol_f)) continue;
          const float tau = (nb - na).hi * ra * rb * (0.5f * rcs);
          const float at = ::fabsf(tau), hy = fmaf(at, at, 1.f);
          float t = at > 1e9f ? __fdividef(0.5f, at) : __fdividef(1.f, at + hy * rsqrtf(hy));
          if (tau < 0.f) t = -t;
          const float tz = t * rcs;
          const R zr = from_f(R(), tz * cr), zi = from_f(R(), tz * ci);
          const R c = rsqrt_r(pmac(pmac(from_f(R(), 1.f), zr, zr), zi, zi));
          const R sr = c * zr, si = c * zi;
          __syncwarp(gmask);  // every lane of the pair has its norms
          if (pl == 0) {
            const df64 move = df64(__fdividef(t * cs, ra * rb), 0.f);  // t |g|
            *(df64*)(X + n) = na - move;
            *(df64*)(Y + n) = nb + move;
            nrot++;
            mc = fmaxf(mc, cs);
            ms = fmaxf(ms, ::fabsf(t));
          }
          // x' = c x - conj(sp) y,  y' = sp x + c y
          for (int i = pl; i < n; i += LP) {
            const cx<R> x = X[i], y = Y[i];
            X[i] = mk<R>(mul3(c, x.re, -sr, y.re, -si, y.im), mul3(c, x.im, -sr, y.im, si, y.re));
            Y[i] = mk<R>(mul3(c, y.re, sr, x.re, -si, x.im), mul3(c, y.im, sr, x.im, si, x.re));
          }
        }
        __syncthreads();
      }
      if (o == 2 * ca - 2) {
        // the sweep's rotations, before the barrier below
        for (int s = 16; s > 0; s >>= 1) {
          nrot += __shfl_xor_sync(0xffffffffu, nrot, s);
          mc = fmaxf(mc, __shfl_xor_sync(0xffffffffu, mc, s));
          ms = fmaxf(ms, __shfl_xor_sync(0xffffffffu, ms, s));
        }
        PjSweep v;
        v.nrot = nrot;
        v.mc = mc;
        v.ms = ms;
        v.pad = 0.f;
        if (lane == 0) s_sweep[sweep & 1][warp] = v;
      }
      if (ca > 1) {
        // top block to the next CTA's top (the last one's to its own bottom, the first
        // one's stays its top), bottom block to the previous CTA's bottom (the first one's
        // to the second's top), by the bulk-copy engine: remote stores take 4,300 cycles an
        // exchange at n = 64 over 8 CTAs (10,200 at n = 128 over 16), remote loads 5,300
        // (6,500), most of it their acknowledgement.
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (!pending)
          __syncthreads();
        else if (!cb.wait())  // every CTA's next buffer has been sent on
          break;
        if (tid == 0) {
          const unsigned bytes = (unsigned)(b * ld * sizeof(cx<R>));
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&s_bar)),
                       "r"(2 * bytes)
                       : "memory");
          const int tc = rank == 0 ? 0 : rank == ca - 1 ? rank : rank + 1;
          const int ts = rank > 0 && rank == ca - 1 ? b : 0;
          send_block(tc, nxt + (long)ts * ld, cur, bytes, &s_bar);
          send_block(rank == 0 ? 1 : rank - 1, nxt + (rank == 0 ? 0 : (long)b * ld), cur + (long)b * ld, bytes, &s_bar);
        }
        armed = true;
        if (!cb.agree(bounded_wait(&s_bar, turn & 1))) break;
        armed = false;
        turn++;
        cb.post();  // our two blocks are here, so their senders' buffers are free
        pending = o < 2 * ca - 2;
        if (!pending && !cb.wait()) break;  // the sweep's rotations of every CTA are there
        cx<R>* t = cur;
        cur = nxt;
        nxt = t;
      } else if (o == 2 * ca - 2) {
        __syncthreads();
      }
    }
    if (cb.lost) break;
    if (measure) {
      for (int s = 16; s > 0; s >>= 1) off_l += __shfl_xor_sync(0xffffffffu, off_l, s);
      if (lane == 0) s_off[warp] = off_l;
      if (!cb.sync()) break;
      for (int c = 0; c < ca * NW; c++) off2 += *on_cta(&s_off[c % NW], c / NW);
      break;
    }
    int all = 0;
    float amc = 0.f, ams = 0.f;
    for (int c = lane; c < ca * NW; c += 32) {
      const PjSweep v = *on_cta(&s_sweep[sweep & 1][c % NW], c / NW);
      all += v.nrot;
      amc = fmaxf(amc, v.mc);
      ams = fmaxf(ams, v.ms);
    }
    for (int s = 16; s > 0; s >>= 1) {
      all += __shfl_xor_sync(0xffffffffu, all, s);
      amc = fmaxf(amc, __shfl_xor_sync(0xffffffffu, amc, s));
      ams = fmaxf(ams, __shfl_xor_sync(0xffffffffu, ams, s));
    }
    total_rot += all;
    // a sweep that rotated nothing, or whose rotations can have refilled the couplings
    // they met by no more than the largest sine times the largest cosine of the sweep,
    // and left no more than FP32's rounding of the tangent
    if (all == 0 || amc * fmaxf(ams, 1e-6f) * (float)r < 0.1f * tol_f) {
      converged = true;
      break;
    }
    if (sweep + 1 >= e.max_sweeps) measure = true;  // one pass that only sums the couplings left
  }

  // ---- 3. weights, kept count, vectors
  const int ns = nc * ca;
  if (!cb.lost) {
    for (int k0 = 0; k0 < nc; k0 += npg) {
      if (k0 + (warp * 32) / LP >= nc) break;
      const int k = k0 + pg;
      const R na = norm2(k);
      if (k < nc && pl == 0) s_own[k] = (double)na * down;
    }
    if (cb.sync())
      for (int i = tid; i < ns; i += NT) s_lam[i] = *on_cta(&s_own[i % nc], i / nc);
  }
  // blocks that the others have sent us by now land before anyone leaves: a sender is at
  // most one turn ahead of us, and waits in leave() meanwhile
  if (cb.lost && exchanging) {
    if (!armed && tid == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&s_bar)),
                   "r"((unsigned)(2 * b * ld * sizeof(cx<R>)))
                   : "memory");
    bounded_wait(&s_bar, turn & 1);
  }
  const bool gave_up = cb.leave();
  let_next_start();
  if (gave_up) {  // one unit vector and the flag
    r = 0;
    for (int i = tid; i < ns; i += NT) s_lam[i] = 0.0;
  }
  if (tid == 0) s_bad = any_bad ? 1 : 0;
  __syncthreads();
  for (int i = tid; i < ns; i += NT) {
    // squared norms order like their bit patterns
    const long long li = __double_as_longlong(s_lam[i]);
    if (!::isfinite(s_lam[i])) s_bad = 1;
    int rk = 0;
    for (int j = 0; j < ns; j++) {
      const long long lj = __double_as_longlong(s_lam[j]);
      rk += lj > li || (lj == li && j < i);
    }
    s_rank[i] = (short)rk;
    s_w[rk] = s_lam[i];
  }
  __syncthreads();
  if (warp == 0) {
    // weights beyond the factor's rank are zero: the rule sees the first r, and the zeros
    // behind them change neither its sums nor its decision
    const int m = max(1, min(r, n));
    double total = 0.0, kept = 0.0;
    const int k = !s_bad && r > 0 ? truncation_count(s_w, m, e.tol, cap, e.gap, total, kept) : 1;
    if (lane == 0) s_k = k;
    if (rank == 0 && lane == 0) {
      d[e.dim_out] = k;
      if (e.kept_weight) *e.kept_weight = kept;
      if (e.total_weight) *e.total_weight = total;
      if (e.disc_stat && total > 0.0) {
        const double dr = (total - kept) / total;
        if (dr > *e.disc_stat) *e.disc_stat = dr;
      }
      if (e.err) {
        if (gave_up) atomicOr(e.err, 4);
        if (!gave_up && !converged && !s_bad && !(::sqrt(off2) * down <= (double)n * FcEps<R>::v * tr)) atomicOr(e.err, 1);
        if (s_bad) atomicOr(e.err, 2);
      }
      if (e.solver_stats) {
        atomicAdd(e.solver_stats + 0, 1.0);
        atomicAdd(e.solver_stats + 1, (double)(converged ? sweep + 1 : e.max_sweeps));
        atomicAdd(e.solver_stats + 2, (double)n);
        atomicAdd(e.solver_stats + 3, (double)k);
        if (!converged && !gave_up) atomicAdd(e.solver_stats + 4, 1.0);
        if (ca > 1) atomicAdd(e.solver_stats + 5, 1.0);  // a multi-SM solve
        atomicMax((unsigned long long*)(e.solver_stats + 6), (unsigned long long)__double_as_longlong((double)n));
      }
      if (prof) {
        atomicAdd(prof, 28.0 * (double)n * (double)total_rot + 4.0 * (double)n * (double)r * (double)r);
        atomicAdd(prof + QLB_K_COUNT, 2.0 * sizeof(zd) * (double)n * (double)n);
      }
    }
  }
  __syncthreads();
  const int k = s_k;
  if (rank == 0 && e.lam)
    for (int i = tid; i < n; i += NT) e.lam[i] = r > 0 && i < ns ? s_w[i] : 0.0;
  zd* out = (zd*)e.out;
  if (e.out_mode != 0 && e.out_mode != 1) return;
  if (r == 0) {  // nothing above rounding (or non-finite entries, a lost wait): one unit vector
    if (rank == 0)
      for (int i = tid; i < n; i += NT) out[i] = mk<double>(i == 0 ? 1.0 : 0.0, 0.0);
    return;
  }
  for (int s = warp; s < nc; s += NW) {
    const int rk = s_rank[rank * nc + s];
    if (rk >= k) continue;
    // the norm again in the working precision (a scaled weight may have left its range)
    R na = zero;
    const cx<R>* X = cur + (long)s * ld;
    for (int i = lane; i < n; i += 32) na = pmac(pmac(na, X[i].re, X[i].re), X[i].im, X[i].im);
    for (int o = 16; o > 0; o >>= 1) na = na + sx(na, o);
    const R inv = na > zero ? from_f(R(), 1.f) / sqrt(na) : zero;
    for (int i = lane; i < n; i += 32) {
      const double vr = (double)(X[i].re * inv), vi = (double)(X[i].im * inv);
      if (e.out_mode == 0)
        out[(long)i * k + rk] = mk<double>(vr, vi);
      else
        out[(long)rk * n + i] = mk<double>(vr, -vi);
    }
  }
}

template <typename R>
size_t pj_smem(int n_max) {
  int m = 1;
  for (int n = 1; n <= n_max; n++) m = std::max(m, pj_region(n, pj_ctas<R>(n)));
  return 2 * (size_t)m * sizeof(cx<R>);
}

constexpr size_t PJ_SMEM_LIMIT = 160 * 1024;  // n = 256 over 16 CTAs needs 128 KB

}  // namespace

bool pj_serves(int n_max) { return n_max <= PJ_MAX_N; }

// grp: the solves of S states in one launch, one cluster per member, n_max their largest
// planned size
template <typename R>
cudaError_t launch_pj(int n_max, const EigDesc& e, const int* d_dims, cudaStream_t s, double* prof,
                      const EigDesc* grp, int S) {
  cudaLaunchConfig_t cfg = {};
  const int c = pj_ctas<R>(n_max);
  cfg.gridDim = dim3(c, S, 1);
  cfg.blockDim = dim3(ClThreads<R>::v, 1, 1);
  cfg.dynamicSmemBytes = pj_smem<R>(n_max);
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
  if (grp) return cudaLaunchKernelEx(&cfg, k_pj<R, true>, e, (int*)d_dims, prof, grp);
  return cudaLaunchKernelEx(&cfg, k_pj<R, false>, e, (int*)d_dims, prof, grp);
}
template cudaError_t launch_pj<double>(int, const EigDesc&, const int*, cudaStream_t, double*, const EigDesc*, int);
template cudaError_t launch_pj<df64>(int, const EigDesc&, const int*, cudaStream_t, double*, const EigDesc*, int);

template <typename K>
static void pj_attr(K* k) {
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PJ_SMEM_LIMIT);
  cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
void init_pj_attributes() {
  pj_attr(k_pj<double, false>);
  pj_attr(k_pj<double, true>);
  pj_attr(k_pj<df64, false>);
  pj_attr(k_pj<df64, true>);
}

}  // namespace qlb
