// Batched complex GEMM of the step whose shapes are read from device memory, in FP64 or,
// for the mixed forms, multiplied and summed in double-float with FP64 operands and results.
//
// The step's GEMMs are small and their sizes change every step (bond dimensions
// live in device memory), while the launch configuration is fixed when the step is
// captured as a CUDA graph.  On this GPU one SM retires ~2 FP64 FMAs per clock, so what
// counts is how evenly the products are spread over the SMs: a 32 x 32 x 16 block of
// complex products takes one SM 16 us, a 16 x 16 x 16 block 4 us, an 8 x 8 x 16 block 1 us.
// The kernel is persistent over a grid decided for four CTAs per SM (its registers let three
// be resident at a time; a step launches fewer, step_gemm_ctas) and decides the decomposition
// at run time from the actual sizes: output tiles of 16 x 16 or 8 x 8 (the eight warps of a CTA
// take a quarter of the K chunk each), whichever finishes first, or takes less work in all, with
// its padding counted, and, with a workspace, a split of the K range into s parts while tiles are fewer than CTAs and a part still outweighs what adding the parts costs.  Each
// (tile, part) item writes its partial tile to the workspace; the CTA that finishes a
// tile last (a per-tile counter, no waiting) adds the s partials in part order and applies
// alpha and beta, so the result does not depend on timing.
//
// Measured on GB300 (C = A B, m x n x k; before: 32 x 32 tiles on two CTAs per SM, parts of 16
// upwards): FP64 16 x 16 x 16 9 us (16), 20 x 32 x 14 9 us (19), 30 x 30 x 30 10 us (28),
// 64^3 12 us (30), 60 x 60 x 2600 94 us (164), 128 x 128 x 600 89 us (100, of which the FP64
// pipe needs 62), 512^3 0.94 ms (1.05); double-float 9 us (12), 8 us (16), 9 us (22), 11 us (21),
// 45 us (91), 42 us (52), 0.35 ms (0.43).  What is left of the small ones is the launch and a chain
// of three trips to L2.

#include <algorithm>
#include <type_traits>

#include "df64.cuh"
#include "qlb_internal.cuh"

namespace qlb {

namespace {

constexpr int G_THREADS = 256;
constexpr int GB_K = 32;                  // K chunk in shared memory
constexpr int GB_TILE = 16 * 16;          // entries of a partial tile in the workspace
constexpr int GB_SPLIT_CAP = 64;          // default cap on the K split
constexpr int GB_SMEM = 2 * GB_K * 17;    // operand chunks (complex entries)

// FP64 -> double-float without the FP64 pipe: hi is the high half of the significand
// rounded to nearest (an integer addition on the bit pattern carries into the exponent as
// rounding should), lo the signed rest, an integer below 2^28 units of the last place.
// Values outside FP32's range for either half take the conversions (out of line: inlined,
// the compiler executes them for every value beside the selection, on the FP64 pipe).
__device__ __noinline__ df64 split_df_slow(double x) { return df64(x); }
__device__ __forceinline__ df64 split_df(double x) {
  const long long u = __double_as_longlong(x);
  const long long mag = u & 0x7fffffffffffffffll;
  const int e = (int)(mag >> 52);
  if (mag == 0) return df64(0.f, 0.f);
  if (e < 1023 - 73 || e > 1023 + 126) return split_df_slow(x);
  const long long hb = (mag + (1ll << 28)) & ~((1ll << 29) - 1);
  const int rest = (int)(mag - hb);
  const unsigned sign = (unsigned)((unsigned long long)u >> 32) & 0x80000000u;
  const float hi = __uint_as_float(((unsigned)(hb >> 29) - ((1023u - 127u) << 23)) | sign);
  const float ulp = __uint_as_float(((unsigned)(e - 1023 - 52 + 127) << 23) | sign);
  return df64(hi, __fmul_rn(__int2float_rn(rest), ulp));
}
__device__ __forceinline__ cx<double> to_c(cx<double>*, zd v) { return v; }
__device__ __forceinline__ cx<df64> to_c(cx<df64>*, zd v) { return mk<df64>(split_df(v.re), split_df(v.im)); }

// a partial tile entry written by another CTA of this launch (past L1)
__device__ __forceinline__ cx<double> ldcg_cx(const cx<double>* p) {
  const double2 v = __ldcg((const double2*)p);
  return mk<double>(v.x, v.y);
}
__device__ __forceinline__ cx<df64> ldcg_cx(const cx<df64>* p) {
  const float4 v = __ldcg((const float4*)p);
  return mk<df64>(df64(v.x, v.y), df64(v.z, v.w));
}

// Running sum of products.  Double-float: a two-sum of each product into the high word, its
// error terms into one FP32 word, renormalised every second product (settle): the chain
// from product to product is one FP32 addition, and the error word stays at the rounding
// level of the sum.
template <typename C>
struct GAcc;
template <>
struct GAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void mac(double a, double b) { s = fma(a, b, s); }
  __device__ __forceinline__ void settle() {}
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct GAcc<df64> {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void mac(df64 a, df64 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p), t;
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    df_two_sum(s, p, s, t);
    c = __fadd_rn(c, __fadd_rn(e, t));
  }
  __device__ __forceinline__ void settle() { df_quick_two_sum(s, c, s, c); }
  __device__ __forceinline__ df64 value() const {
    df64 r;
    df_two_sum(s, c, r.hi, r.lo);
    return r;
  }
};

__device__ __forceinline__ zd gemm_alpha(const GemmDesc& g) {
  zd alpha = mk<double>(g.alpha_re, g.alpha_im);
  if (g.alpha_scale) {
    double s = *g.alpha_scale;
    if (g.alpha_scale_rsqrt) s = (s > 0.0) ? 1.0 / sqrt(s) : 0.0;
    alpha = cscale(alpha, s);
  }
  return alpha;
}

// cycles that one SM spends on a K of `k` for one tile of TS x TS outputs: ~2 per complex
// product in FP64 (four FMAs at two per clock), ~0.4 in double-float (~50 FP32
// instructions at 128 lanes), and what an item costs besides
template <typename Cm>
__device__ __forceinline__ float tile_cycles(int ts, int k) {
  return (std::is_same<Cm, double>::value ? 2.0f : 0.4f) * (float)(ts * ts) * (float)k +
         600.f;
}

struct GemmPlan {
  int m, n, K, nb1, nb2;
  int tm, tn, ks, chunk;
  long ntiles;
};

// One launch's work items with TS x TS tiles.
template <typename Cm, int TS>
__device__ void gemm_items(const GemmDesc& g, const int* d, const GemmPlan& P, int gnom, unsigned char* sm,
                          int* s_last) {
  constexpr int SL = G_THREADS / (TS * TS);  // K slices of a chunk (1 or 4)
  constexpr int LD = TS + 1;
  constexpr int NL = TS * GB_K / G_THREADS;  // loads per thread and operand
  cx<Cm>* As = (cx<Cm>*)sm;                  // [k][row]
  cx<Cm>* Bs = As + GB_K * LD;               // [k][column]
  const int tid = threadIdx.x;
  const int slice = tid / (TS * TS), o = tid % (TS * TS);
  const int tx = o % TS, ty = o / TS;
  const int lda = dev_eval(g.lda, d), ldb = dev_eval(g.ldb, d);
  cx<Cm>* part_ws = (cx<Cm>*)g.ws;
  int* counters = g.ws ? (int*)(part_ws + (long)gnom * GB_TILE) : nullptr;
  const long items = P.ntiles * P.ks;
  for (long it = blockIdx.x; it < items; it += gridDim.x) {
    const long tile = it / P.ks;
    const int kp = (int)(it - tile * P.ks);
    const int bz = (int)(tile / ((long)P.tm * P.tn));
    const int t2 = (int)(tile - (long)bz * P.tm * P.tn);
    const int row0 = (t2 / P.tn) * TS, col0 = (t2 % P.tn) * TS;
    const int b1 = bz / P.nb2, b2 = bz - b1 * P.nb2;
    const zd* A = (const zd*)g.A + (long)b1 * dev_eval(g.sA1, d) + (long)b2 * dev_eval(g.sA2, d);
    const zd* B = (const zd*)g.B + (long)b1 * dev_eval(g.sB1, d) + (long)b2 * dev_eval(g.sB2, d);
    const int kbeg = kp * P.chunk, kend = min(P.K, kbeg + P.chunk);
    // the products of padding rows are skipped where a whole warp would form only those
    const int wrow = row0 + (TS == 16 ? 2 * ((tid >> 5) & 7) : 4 * ((tid >> 5) & 1));
    const bool work = wrow < P.m;
    cx<Cm> acc = mk<Cm>(GAcc<Cm>().value(), GAcc<Cm>().value());
    for (int k0 = kbeg; k0 < kend; k0 += GB_K) {
      // All loads of a chunk in flight.  Up to three CTAs per SM cover their latency for each other;
      // where a launch has one (most of a step's), nothing does.
      zd v[2 * NL];
#pragma unroll
      for (int q = 0; q < NL; q++) {
        const int e = tid + q * G_THREADS;
        // op(A)(i, k): OP_N A[i lda + k]; OP_T, OP_C A[k lda + i] (lanes along the rows of memory)
        const int kk = g.opA == OP_N ? e % GB_K : e / TS, i = g.opA == OP_N ? e / GB_K : e % TS;
        const int gi = row0 + i, gk = k0 + kk;
        v[q] = mk<double>(0.0, 0.0);
        if (gi < P.m && gk < kend) v[q] = g.opA == OP_N ? A[(long)gi * lda + gk] : A[(long)gk * lda + gi];
        // op(B)(k, j): OP_N B[k ldb + j]; OP_T, OP_C B[j ldb + k]
        const int k2 = g.opB == OP_N ? e / TS : e % GB_K, j = g.opB == OP_N ? e % TS : e / GB_K;
        const int gj = col0 + j, gl = k0 + k2;
        v[NL + q] = mk<double>(0.0, 0.0);
        if (gj < P.n && gl < kend) v[NL + q] = g.opB == OP_N ? B[(long)gl * ldb + gj] : B[(long)gj * ldb + gl];
      }
#pragma unroll
      for (int q = 0; q < NL; q++) {
        const int e = tid + q * G_THREADS;
        const int kk = g.opA == OP_N ? e % GB_K : e / TS, i = g.opA == OP_N ? e / GB_K : e % TS;
        if (g.opA == OP_C) v[q].im = -v[q].im;
        As[kk * LD + i] = to_c((cx<Cm>*)nullptr, v[q]);
        const int k2 = g.opB == OP_N ? e / TS : e % GB_K, j = g.opB == OP_N ? e % TS : e / GB_K;
        if (g.opB == OP_C) v[NL + q].im = -v[NL + q].im;
        Bs[k2 * LD + j] = to_c((cx<Cm>*)nullptr, v[NL + q]);
      }
      __syncthreads();
      const int kn = min(GB_K, kend - k0);
      // slice s takes the k of its residue modulo SL
      auto step = [&](int kk, GAcc<Cm>& re, GAcc<Cm>& im) {
        const cx<Cm> a = As[kk * LD + ty], b = Bs[kk * LD + tx];
        re.mac(a.re, b.re);
        re.mac(-a.im, b.im);
        im.mac(a.re, b.im);
        im.mac(a.im, b.re);
        re.settle();
        im.settle();
      };
      if (work) {
        // even and odd steps apart and a sum of its own for every chunk: shorter chains, and
        // less rounding (errors grow with the chain's length)
        GAcc<Cm> re0, im0, re1, im1;
        int kk = slice;
#pragma unroll 2
        for (; kk + SL < kn; kk += 2 * SL) {
          step(kk, re0, im0);
          step(kk + SL, re1, im1);
        }
        if (kk < kn) step(kk, re0, im0);
        acc = mk<Cm>(acc.re + (re0.value() + re1.value()), acc.im + (im0.value() + im1.value()));
      }
      __syncthreads();
    }
    if (SL > 1) {
      // the slices' sums, in slice order
      As[slice * TS * TS + o] = acc;
      __syncthreads();
      if (slice == 0) {
#pragma unroll
        for (int q = 1; q < SL; q++) acc = cadd(acc, As[q * TS * TS + o]);
      }
      __syncthreads();
    }
    const bool mine = slice == 0 && row0 + ty < P.m && col0 + tx < P.n;
    if (P.ks > 1) {
      // partial tile of this K part; the last CTA of the tile adds them in order
      if (mine) part_ws[((long)kp * P.ntiles + tile) * GB_TILE + o] = acc;
      __threadfence();
      __syncthreads();
      if (tid == 0) *s_last = atomicAdd(counters + tile, 1) == P.ks - 1;
      __syncthreads();
      const bool last = *s_last != 0;
      __syncthreads();
      if (!last) continue;
      __threadfence();
      if (mine) {
        const long pstride = P.ntiles * GB_TILE;
        const cx<Cm>* P0 = part_ws + tile * GB_TILE + o;
        cx<Cm> sum = ldcg_cx(P0);
        int q = 1;
        // four independent loads in flight, added in part order
        for (; q + 4 <= P.ks; q += 4) {
          const cx<Cm> v0 = ldcg_cx(P0 + q * pstride), v1 = ldcg_cx(P0 + (q + 1) * pstride);
          const cx<Cm> v2 = ldcg_cx(P0 + (q + 2) * pstride), v3 = ldcg_cx(P0 + (q + 3) * pstride);
          sum = cadd(cadd(cadd(cadd(sum, v0), v1), v2), v3);
        }
        for (; q < P.ks; q++) sum = cadd(sum, ldcg_cx(P0 + q * pstride));
        acc = sum;
      }
      if (tid == 0) counters[tile] = 0;  // ready for the next launch on this workspace
    }
    if (mine) {
      const zd v = cmul(gemm_alpha(g), mk<double>((double)acc.re, (double)acc.im));
      zd* dst = (zd*)g.C + (long)b1 * dev_eval(g.sC1, d) + (long)b2 * dev_eval(g.sC2, d) +
                (long)(row0 + ty) * dev_eval(g.ldc, d) + col0 + tx;
      *dst = g.beta ? cadd(v, *dst) : v;
    }
  }
}

// Cm: the type the products are formed and summed in (double, or double-float in the
// mixed forms)
template <typename Cm, bool GRP>
__global__ void __launch_bounds__(G_THREADS, 3) k_gemm(const GemmDesc g_in, const int* d_in, double* prof,
                                                       const GemmDesc* __restrict__ grp) {
  // grouped launch: this CTA works on member blockIdx.y, whose descriptor (and dims)
  // come from the group's table (kept in shared memory, not registers); the tile and the K
  // split are decided on the member's nominal grid
  __shared__ GemmDesc s_g;
  __shared__ __align__(16) unsigned char sm[GB_SMEM * sizeof(cx<Cm>)];
  __shared__ int s_last;
  if constexpr (GRP) {
    const int* src = (const int*)(grp + blockIdx.y);
    for (int i = threadIdx.x; i < (int)(sizeof(GemmDesc) / sizeof(int)); i += G_THREADS) ((int*)&s_g)[i] = src[i];
    __syncthreads();
  }
  const GemmDesc& g = GRP ? s_g : g_in;
  const int* d = GRP ? s_g.dims : d_in;
  after_previous();
  let_next_start();
  const int gnom = g.split_grid > 0 ? g.split_grid : (int)gridDim.x;
  GemmPlan P;
  P.m = dev_eval(g.m, d);
  P.n = dev_eval(g.n, d);
  P.K = dev_eval(g.k, d);
  P.nb1 = dev_eval(g.nb1, d);
  P.nb2 = dev_eval(g.nb2, d);
  const int nb = P.nb1 * P.nb2;
  if (P.m <= 0 || P.n <= 0 || nb <= 0) return;
  // Most CTAs of a small product find no work however it is cut (parts are of 32 in K at least) and
  // leave before the plan: 16 cats of N = 32 at bonds of 1, on their own streams, are bound by it.
  const long t8 = (long)((P.m + 7) / 8) * ((P.n + 7) / 8) * nb;
  if (blockIdx.x && (long)blockIdx.x >= t8 * max(1, (P.K + 31) / 32)) return;
  // the tile: both counts of tiles in waves over the SMs (a quarter of the nominal grid)
  const long t16 = (long)((P.m + 15) / 16) * ((P.n + 15) / 16) * nb;
  const int sms = max(1, gnom / 4);
  // Products that keep the chip busy however they are cut go by their work with its padding: a
  // product takes an SM 2.0 cycles in tiles of 16 and 2.4 in tiles of 8, which read shared memory
  // twice as often, in double-float 0.75 and 1.2 (768^3).  The others go by waves over the SMs.
  // About the line, tiles of 16 against 8: 150^3 41 us against 44, double-float 30 against 25;
  // 128 x 128 x 600 90 against 102, 40 against 57; 256^3 146 against 148, 64 against 74; 512^3 0.94 ms
  // against 1.10, 0.35 against 0.53.  A Gram matrix's line lies higher: in a step, behind the
  // launch that wrote its operand, 162 x 162 x 496 is 50 us slower in tiles of 16.
  const float products = (float)P.m * (float)P.n * (float)P.K * (float)nb;
  const bool large = products >= (g.kclass == QLB_K_GRAM ? 1.6e7f : 8.0e6f);
  const float c16 = large ? (std::is_same<Cm, double>::value ? 4.f * 0.83f : 4.f * 0.63f) * (float)t16
                          : (float)((t16 + sms - 1) / sms) * tile_cycles<Cm>(16, P.K);
  const float c8 = large ? (float)t8 : (float)((t8 + sms - 1) / sms) * tile_cycles<Cm>(8, P.K);
  const bool small = c8 < c16;
  P.ntiles = small ? t8 : t16;
  P.tm = small ? (P.m + 7) / 8 : (P.m + 15) / 16;
  P.tn = small ? (P.n + 7) / 8 : (P.n + 15) / 16;
  // the K split (the same in every CTA): parts of at least ~8,000 cycles, about twice what
  // the partial tiles' round trip through L2 costs
  P.ks = 1;
  const int least = GB_K * (std::is_same<Cm, double>::value ? (small ? 2 : 1) : (small ? 8 : 2));
  if (g.ws && P.K > least && P.ntiles < (long)gnom) {
    const int cap = g.ksplit >= 1 ? g.ksplit : GB_SPLIT_CAP;
    P.ks = (int)min((long)cap, (long)gnom / P.ntiles);
    if (large) {
      // Three of the nominal four CTAs per SM are resident: parts that fill their places leave no
      // second wave (192 x 192 x 2048: 568 us in 3 parts, 680 in 4), but a grid part empty is spread
      // unevenly (162 x 162 x 496, 121 tiles: 165 us in 3 parts, 113 in 4).
      const int slots = 3 * sms, per = slots / (int)P.ntiles;
      if (16 * per * (int)P.ntiles >= 15 * slots) P.ks = min(P.ks, per);
    }
    P.ks = max(1, min(P.ks, (P.K + least - 1) / least));
  }
  P.chunk = P.ks > 1 ? (((P.K + P.ks - 1) / P.ks + GB_K - 1) / GB_K) * GB_K : P.K;
  if (P.ks > 1) P.ks = (P.K + P.chunk - 1) / P.chunk;
  if (prof && blockIdx.x == 0 && threadIdx.x == 0) {
    atomicAdd(prof, 8.0 * (double)P.m * (double)P.n * (double)P.K * nb);
    atomicAdd(prof + QLB_K_COUNT,
              (double)sizeof(zd) * ((double)P.m * P.K + (double)P.K * P.n + (double)P.m * P.n) * nb);
  }
  if ((long)blockIdx.x >= P.ntiles * P.ks) return;
  if (small)
    gemm_items<Cm, 8>(g, d, P, gnom, sm, &s_last);
  else
    gemm_items<Cm, 16>(g, d, P, gnom, sm, &s_last);
}

}  // namespace

size_t gemm_workspace_elems(int grid) {
  // grid partial tiles, then one counter (int) per tile, rounded up to whole elements
  return (size_t)grid * GB_TILE + ((size_t)grid * sizeof(int) + sizeof(zd) - 1) / sizeof(zd);
}

int gemm_grid_default() {
  static int grid = 0;
  if (!grid) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
      cudaGetLastError();
      sms = 148;
    }
    grid = 4 * sms;
  }
  return grid;
}

// CTAs that a step launches for a GEMM of m_max planned rows (GemmDesc::ctas): one per SM, four
// for a Gram matrix planned above 64.  The sizes that a launch meets are mostly far below the
// planned ones, and states on their own streams share the SMs: sixteen cats of N = 32 at bonds of 1
// took 0.97 ms a step of all with four for every GEMM, 0.55 with this rule, and 0.49 now that CTAs
// without work leave before the plan.  One for the large Grams costs 6 % of their time in the
// transmon at chi 128 (6.21 ms in two steps against 5.85) and 12 % in the coupled cats (4.31
// against 3.84), two cost 4 and 7 %.  The tiles and the K split stay those of the full grid.
int step_gemm_ctas(int kclass, int m_max) {
  return kclass == QLB_K_GRAM && m_max > 64 ? 0 : gemm_grid_default() / 4;
}

cudaError_t launch_gemm(const GemmDesc& g, const int* d_dims, cudaStream_t s, double* prof) {
  const long planned =
      (long)((g.m_max + 7) / 8) * ((g.n_max + 7) / 8) * (g.nb_max > 0 ? g.nb_max : 1);
  if (planned <= 0) return cudaSuccess;
  // a fixed grid that the run-time decomposition fills; without a workspace (no K split)
  // no more CTAs than planned tiles
  GemmDesc gg = g;
  const int full = g.ws && g.grid > 0 ? g.grid : gemm_grid_default();
  const int grid = g.ws ? full : (int)std::min<long>(planned, full);
  gg.split_grid = full;
  const int ctas = g.ctas > 0 ? std::min(grid, g.ctas) : grid;
  if (g.df64)
    return launch_after(k_gemm<df64, false>, dim3(ctas), G_THREADS, s, gg, d_dims, prof, nullptr);
  return launch_after(k_gemm<double, false>, dim3(ctas), G_THREADS, s, gg, d_dims, prof, nullptr);
}

// The same GEMM of S states in one launch: grid (per-member CTAs, S).  Every member
// descriptor in d_grp carries its dims, a workspace for the default grid and
// split_grid = the default grid, so each member is tiled, split and summed exactly as in
// its own launch; the per-member CTA count only changes how the work items are
// shared out (S x per-member CTAs ~ four per SM over the whole group).
cudaError_t launch_gemm_group(const GemmDesc* d_grp, int S, int use_df, cudaStream_t s, double* prof) {
  if (S <= 0) return cudaSuccess;
  const int full = gemm_grid_default();
  const int per = std::max(8, std::min(full, (full + S - 1) / S));
  GemmDesc dummy{};
  if (use_df)
    return launch_after(k_gemm<df64, true>, dim3(per, S), G_THREADS, s, dummy, nullptr, prof, d_grp);
  return launch_after(k_gemm<double, true>, dim3(per, S), G_THREADS, s, dummy, nullptr, prof, d_grp);
}

}  // namespace qlb
