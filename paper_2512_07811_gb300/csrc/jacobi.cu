// One-sided Jacobi SVD of small dense matrices by one thread-block cluster per
// matrix, with the truncation rule at its end.
//
// G (p x q, columns rotated to mutual orthogonality) gives the left singular
// vectors of G as normalised rotated columns.  The columns, padded with zero
// columns to 2 NC bs, form NB = 2 NC blocks of bs, two per CTA: position i
// ("top") and NB - 1 - i ("bottom") of the round-robin tournament of the
// blocks.  In a block-round a CTA rotates the bs x bs cross pairs of its two
// blocks in bs rounds of bs disjoint pairs, one warp per pair, the top column
// in registers throughout; in the first block-round of a sweep also the pairs
// inside each block.  In the last round the rotated columns are written straight
// from registers to the shared memory of the CTA that holds them next, so a
// block exchange costs one cluster barrier.
//
// What bounds it: a sweep is a chain of about q rounds, each the latency of one
// pair (dot product, warp reduction, rotation scalars, rotation, barrier), in
// FP64 also the FP64 pipe (a warp instruction holds it 16 cycles, a dependent
// one takes 75).  Hence
//   * the squared column norms are carried along, |a|^2 -+ |g|^2 / w, and summed
//     anew once a sweep and after a drop below a twentieth, which leaves one
//     inner product per pair instead of three;
//   * the rotation needs two reciprocal square roots and no division (see
//     rotate_pair);
//   * a sweep in which every rotation was small is the last one: the next
//     would only confirm it (see `big2`).
// The caller sorts and QR-factors the matrix first (jacobi on R^H), which cuts
// the sweeps from 14-21 to 6-7 on the roundings' matrices.
//
// FP64 matrices get all but the last two or three sweeps in FP32 (PRE): a sweep
// costs a fifth there (68 x 68: 45 us against 224 us).  The FP32 kernel rotates
// an identity along and returns V; two Newton-Schulz steps make V unitary to
// FP64 rounding, G V is formed in FP64, and the FP64 kernel goes on from there
// to its own tolerance, so the result is as before: V only chooses a basis.
// The columns of G V keep the accuracy of the small ones, since V is graded as
// G is.  Clusters of values equal to FP32 still take the full number.  us of a
// rounding with one such SVD (values over 12 decades) without / with it: 68 x 68
// 2640 / 1627, 80 x 48 1682 / 1100, 256 x 128 9054 / 5167; errors against 64-bit
// references unchanged.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "dense.cuh"
#include "kernels.h"

namespace {

namespace cg = cooperative_groups;
using dense::Lim;

template <class R>
struct JacArgs {
  const cplx<R>* G;       // p x q row-major, matrices p*q apart
  const int* perm;        // row i of G is component perm[i] of the vectors (p apart), or null
  cplx<R>* Vh;            // q x p row-major: row j the conjugate of vector j, by decreasing singular value
  R* sigma;               // q, or null
  int* trunc;             // 4 per matrix: rank kept, 1 if max_rank cut it, discarded tail (double); or null
  double delta;           // threshold of the tail
  const double* deltas;   // per matrix instead of delta, or null
  int max_rank;           // 0: no cap
  int mask;               // rows of Vh from the kept rank on are zeroed
  int p, q, bs, bsx, adapt, max_sweeps;  // bsx: the most columns a block may get; adapt: columns may be left out
  int* sweeps;
  // rotations only (PRE): the matrix in FP64, the accumulated rotations transposed (row j: the column of the j-th
  // largest norm, q x q), followed by two identity matrices of that size
  const zc* Gd;
  zc* Vt;
};

// most threads of a CTA: 256 where a pair's two columns take more than the 128
// registers that 512 leave (up to 256 rows or columns, which sixteen CTAs of
// eight warps hold)
template <class R, int RT, bool PRE>
struct JacThreads {
  static constexpr int value = sizeof(R) == 8 || PRE || (RT > 4 && RT <= 8) ? 256 : 512;
};

// cycles of a sweep, see jac_plan
template <class R>
__host__ __device__ inline float jac_cost(int nc, int bs, int lp, int rows) {
  const int queue = ((bs * lp + 31) / 32 + 3) / 4;
  float c, e = nc > 1 ? 600.f : 60.f;
  if (sizeof(R) == 4) {
    const float lat = 540.f + 22.f * rows, issue = queue * (150.f + 28.f * rows);
    c = lat > issue ? lat : issue;
    if (nc > 1) e += 100.f + 30.f * bs * lp * rows / 32;
  } else {
    c = queue * 64.f * (16.f * rows + 27.f) + 300.f;
    if (nc > 1) e += 60.f * bs * lp * rows / 32;
  }
  return (2 * nc - 1) * (bs * c + e) + (bs + (bs & 1)) * c;
}

// sum over the LP lanes that share a pair (all lanes of the warp take part)
template <int LP, class R>
__device__ __forceinline__ R gsum(R v) {
#pragma unroll
  for (int o = LP / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// FP64: half of the lanes sum the real part, half the imaginary one, one addition a level
template <int LP, class R>
__device__ __forceinline__ cplx<R> gsum_c(cplx<R> w, int lane) {
  if constexpr (sizeof(R) == 4) {
#pragma unroll
    for (int o = LP / 2; o > 0; o >>= 1) {
      w.re += __shfl_xor_sync(0xffffffffu, w.re, o);
      w.im += __shfl_xor_sync(0xffffffffu, w.im, o);
    }
    return w;
  } else {
    const bool up = lane & (LP / 2);
    R v = (up ? w.im : w.re) + __shfl_xor_sync(0xffffffffu, up ? w.re : w.im, LP / 2);
#pragma unroll
    for (int o = LP / 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const R o = __shfl_xor_sync(0xffffffffu, v, LP / 2);
    return up ? cplx<R>(o, v) : cplx<R>(v, o);
  }
}

// FP64 helpers without FP64 instructions
__device__ __forceinline__ double times2(double x, int k) {  // x 2^k, x normal
  return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
}
__device__ __forceinline__ int ilogb_c(double x) { return (__double2hiint(x) >> 20) - 1023; }  // x > 0 normal
constexpr int kHiMin = 0x05e00000;  // squares of inner products below 1e-280 count as zero

// whether a squared norm has dropped to less than about a sixteenth of its old value
__device__ __forceinline__ bool dropped(float v, float old) { return !(v > 0.0625f * old); }
__device__ __forceinline__ bool dropped(double v, double old) {
  return __double2hiint(v) < __double2hiint(old) - (4 << 20);  // by the exponents: no FP64 instruction
}

// (a column's first RPL slices are the matrix's, the other RT - RPL follow its rotations)
template <int LP, int RPL, class R, int RT>
__device__ __forceinline__ R col_norm2(const cplx<R> (&x)[RT]) {
  R s = 0, s1 = 0;
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    if (u & 1) s1 += abs2(x[u]); else s += abs2(x[u]);
  }
  return gsum<LP>(s + s1);
}

// Rotates columns x, y (rows on the LP lanes of a group) to orthogonality; al,
// be their squared norms.  With g = x^H y, d = (be - al) / 2, h = sqrt(d^2 +
// |g|^2) and w = |d| + h, the smaller root has tan = |g| / w and w^2 + |g|^2 =
// 2 h w, so with r = 1 / sqrt(w^2 + |g|^2): cos = w r, sin e^{i arg g} = g r
// (signed by d), and the norms change by |g|^2 / w = 2 |g|^2 h r^2.  cos^2 +
// sin^2 = 1 to the accuracy of r, whatever h is.  Returns 0 (`act` false,
// orthogonal to tol, or |g|^2 below the normal range), 1 (rotated) or 3 (rotated, not
// small: the sine weighted by the norms' ratio above sqrt(big2); that weighted
// sine is at least about half the cosine of the angle between x and y).
// FP32 rotations alone (RT > RPL): a pair's norms are brought to 2^40, so that the
// noise columns of a rank-deficient matrix (1e-16 of the largest) are rotated
// too: they take as many FP64 sweeps as the others.
template <int LP, int RPL, class R, int RT>
__device__ __forceinline__ int rotate_pair(cplx<R> (&x)[RT], cplx<R> (&y)[RT], R& al, R& be, R tol2, R big2,
                                           int lane, bool act) {
  cplx<R> g(0, 0), g1(0, 0);
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    if (u & 1) cfma_conj(g1, x[u], y[u]); else cfma_conj(g, x[u], y[u]);
  }
  g = gsum_c<LP>(g + g1, lane);
  const R al0 = al, be0 = be;
  R unscale = 1;
  if constexpr (RT > RPL) {
    const int e = max(__float_as_int(fmax(al, be)) >> 23, 60);
    const R k = __int_as_float((294 - e) << 23);
    g = k * g;
    al *= k;
    be *= k;
    unscale = __int_as_float((e - 40) << 23);
  }
  const R ag2 = abs2(g);
  R cs, dl;
  cplx<R> f;
  int code;
  bool rot, up;
  if constexpr (sizeof(R) == 4) {
    rot = act && ag2 > tol2 * (al * be) && ag2 >= FLT_MIN;
    if (LP == 32 ? !rot : !__any_sync(0xffffffffu, rot)) {
      al = al0;
      be = be0;
      return 0;
    }
    const R d = R(0.5) * (be - al), h2 = fma(d, d, ag2);
    const R h = h2 * rsqrtf(h2), w = fabs(d) + h;
    const R r = dense::rsqrt_nr(fma(w, w, ag2));
    up = d >= R(0);  // be >= al
    cs = w * r;
    const R sr = up ? r : -r;
    f = cplx<R>(sr * g.re, sr * g.im);
    const R s2 = ag2 * (r * r);
    dl = (h + h) * s2;
    code = s2 * (up ? be : al) > big2 * (up ? al : be) ? 3 : 1;
  } else {
    // a warp instruction holds its quarter's FP64 unit for 64 cycles: comparisons
    // by exponents (integer), factors of 2 and 4 by adding to them, h from the
    // hardware's 20-bit reciprocal square root.  The threshold then lies between
    // tol / sqrt(2) and sqrt(2) tol.
    const int hg = __double2hiint(ag2), ea = __double2hiint(al) >> 20, eb = __double2hiint(be) >> 20;
    rot = act && (hg >> 20) + 1023 > ea + eb + ilogb_c(tol2) && hg >= kHiMin && hg < 0x7ff00000;
    if (LP == 32 ? !rot : !__any_sync(0xffffffffu, rot)) return 0;
    const R D = be - al, q4 = times2(ag2, 2), h2 = fma(D, D, q4);
    // 2 h by one Newton step of the square root from 20 bits (without it a rotation leaves
    // up to 2^-21 of its cosine, which the rule for the last sweep takes for nothing), 2 w
    const R yh = dense::rsqrt_approx(h2), H0 = h2 * yh, H = fma(fma(-H0, H0, h2), times2(yh, -1), H0), W = fabs(D) + H;
    const R x4 = fma(W, W, q4);
    const R r2 = dense::rsqrt_third_order(x4, dense::rsqrt_approx(x4));  // r / 2
    const R r = times2(r2, 1);
    up = __double2hiint(D) >= 0;
    cs = W * r2;
    const R sr = up ? r : -r;
    f = cplx<R>(sr * g.re, sr * g.im);
    const R s2 = ag2 * (r * r);
    dl = H * s2;
    const int es = (__double2hiint(s2) >> 20) + (up ? eb - ea : ea - eb);
    code = es >= ilogb_c(big2) + 1022 ? 3 : 1;
  }
  if (LP < 32 && !rot) {  // another group of the warp rotates
    cs = R(1);
    f = cplx<R>(0, 0);
    dl = R(0);
    code = 0;
  }
#pragma unroll
  for (int u = 0; u < RT; ++u) {
    const cplx<R> a = x[u], b = y[u];
    x[u].re = fma(cs, a.re, fma(-f.re, b.re, -f.im * b.im));
    x[u].im = fma(cs, a.im, fma(-f.re, b.im, f.im * b.re));
    y[u].re = fma(cs, b.re, fma(f.re, a.re, -f.im * a.im));
    y[u].im = fma(cs, b.im, fma(f.re, a.im, f.im * a.re));
  }
  if constexpr (RT > RPL) dl *= unscale;
  if (!up) dl = -dl;
  al = al0 - dl;
  be = be0 + dl;
  const bool da = dropped(al, al0), db = dropped(be, be0);
  if (LP == 32 ? da || db : __any_sync(0xffffffffu, da || db)) {
    const R na = col_norm2<LP, RPL>(x), nb = col_norm2<LP, RPL>(y);
    if (da) al = na;
    if (db) be = nb;
  }
  return code;
}

template <class R, int LP, int RPL, bool PRE>
__global__ void __launch_bounds__(JacThreads<R, RPL, PRE>::value, 1)
jacobi_cluster2_kernel(const __grid_constant__ JacArgs<R> a) {
  typedef cplx<R> C;
  cg::cluster_group cluster = cg::this_cluster();
  typedef typename std::conditional<PRE, double, R>::type S;  // type of the matrix
  const int rank = (int)cluster.block_rank(), p = a.p, q = a.q;
  // active CTAs of the cluster, columns of a block, columns worked on
  int NC = (int)cluster.num_blocks(), bs = a.bs, qa = q;
  constexpr int RT = PRE ? 2 * RPL : RPL, LD = LP * RT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int nthr = blockDim.x;
  // a pair is worked on by a group of LP lanes: group w of ng, lane gl of it
  const int gl = lane % LP, w = threadIdx.x / LP;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* slots = reinterpret_cast<C*>(smem_raw);                 // [4][bs][LD]
  double* scan = reinterpret_cast<double*>(slots + (size_t)4 * a.bsx * LD);  // [0] squared norm of the dropped columns
  R* nrm = reinterpret_cast<R*>(scan + 2);                   // [4][bs] squared norms
  R* norms = nrm + 4 * a.bsx;                                // [qp] final norms
  R* sorted = norms + q + 64;                                // [qp]
  int* flags = reinterpret_cast<int*>(sorted + q + 64);      // [2][NC] sweep flags, then [NC] exponents
  int* s_int = flags + 3 * 16;                               // [0] sweep flags of this CTA, [1] kept rank, [2..4] plan
  const int64_t bt = blockIdx.y;
  auto col = [&](int slot, int j) { return slots + (slot * a.bsx + j) * LD; };
  int top = 0, bot = 1, in_top = 2, in_bot = 3;
  if (threadIdx.x == 0) s_int[0] = 0;
  cluster.sync();
  const cplx<S>* G;
  if constexpr (PRE) G = a.Gd; else G = a.G;
  G += bt * (int64_t)p * q;
  // blocks of this CTA: rank on top, 2 NC - 1 - rank below
  auto blocks = [&](auto&& f) {
    for (int e = threadIdx.x; e < 2 * bs * LD; e += nthr) {
      const int i = e / (2 * bs), jj = e - i * 2 * bs, half = jj / bs, j = jj - half * bs;
      const int c = (half == 0 ? rank : 2 * NC - 1 - rank) * bs + j;
      f(c, i, col(half == 0 ? top : bot, j) + i);
    }
  };
  // the power of two that brings the largest component near 1 (FP32: near
  // 2^14, so that squares of squared norms of columns down to 1e-14 of the
  // largest stay normal)
  const bool whole = PRE || a.adapt;  // the matrix is read before its columns are dealt out
  S amax = 0;
  // (rows dealt to the CTAs, a CTA's rows to groups of qg threads)
  const int qg = min((q + 31) & ~31, nthr), ngr = nthr / qg, grp = threadIdx.x / qg, c0 = threadIdx.x - grp * qg;
  if (whole) {
    if (grp < ngr)
      for (int c = c0; c < q; c += qg) {
#pragma unroll 8
        for (int i = rank + NC * grp; i < p; i += NC * ngr) {
          const cplx<S> v = G[(int64_t)i * q + c];
          amax = fmax(amax, fmax(fabs(v.re), fabs(v.im)));
        }
      }
  } else if constexpr (!PRE) {
    blocks([&](int c, int i, C* d) {
      C v(0, 0);
      if (c < q && i < p) v = G[(int64_t)i * q + c];
      *d = v;
      amax = fmax(amax, fmax(fabs(v.re), fabs(v.im)));
    });
  }
  {
    const int ex = __reduce_max_sync(0xffffffffu, dense::exponent_of(amax, sizeof(S) == 4 ? -110 : -1000));
    int* wex = reinterpret_cast<int*>(sorted);
    if (lane == 0) wex[warp] = ex;
    __syncthreads();
    if (warp == 0) {
      const int t = __reduce_max_sync(0xffffffffu, lane < (nthr >> 5) ? wex[lane] : -1000);
      if (lane < NC) cluster.map_shared_rank(flags, lane)[32 + rank] = t;
    }
    cluster.sync();
  }
  int esc = flags[32];
  for (int i = 1; i < NC; ++i) esc = max(esc, flags[32 + i]);
  if (sizeof(R) == 4) esc -= 14;
  const S sg = dense::pow2(S(0), -esc);
  if (a.adapt) {
    // Trailing columns whose whole norm is at most eps ||G|| (one rounding of G)
    // and a quarter of the truncation threshold are left out: in a rounding
    // of a train with superfluous rank they are the noise of the QR, half of
    // the columns.  Their norm counts as discarded, so the tail's bound holds.
    // us without / with: 118 x 118 of rank 59 453 / 227, 172 x 172 of rank 85 852 /
    // 412, FP64 68 x 68 of rank 33 475 / 356; where all columns stay 5 more.
    R* parts = reinterpret_cast<R*>(slots);  // [NC][q] partial sums of the CTAs' rows, then [q] squared norms
    R* cn = parts + NC * q;
    R* own = cn + q;  // [ngr][q]
    if (grp < ngr)
      for (int c = c0; c < q; c += qg) {
        R t = 0;
#pragma unroll 8
        for (int i = rank + NC * grp; i < p; i += NC * ngr) {
          const cplx<S> v = G[(int64_t)i * q + c];
          t += abs2(C((R)(sg * v.re), (R)(sg * v.im)));
        }
        own[grp * q + c] = t;
      }
    __syncthreads();
    for (int c = threadIdx.x; c < q; c += nthr) {
      R t = 0;
      for (int g = 0; g < ngr; ++g) t += own[g * q + c];
      for (int k = 0; k < NC; ++k) cluster.map_shared_rank(parts, k)[rank * q + c] = t;
    }
    cluster.sync();
    for (int c = threadIdx.x; c < q; c += nthr) {
      R t = 0;
      for (int k = 0; k < NC; ++k) t += parts[k * q + c];
      cn[c] = t;
    }
    __syncthreads();
    if (warp == 0) {
      double tot = 0;
      for (int j = lane; j < q; j += 32) tot += (double)cn[j];
      tot = dense::wsum(tot);
      constexpr double eps = sizeof(S) == 4 ? (double)FLT_EPSILON : DBL_EPSILON;
      const double ds = 0.25 * (a.deltas ? a.deltas[bt] : a.delta) * dense::pow2(0.0, -esc);
      double thr2 = eps * eps * tot;
      if (!(ds * ds >= thr2)) thr2 = ds * ds;  // (a NaN drops nothing)
      double out = 0;
      int t = q;
      for (int hi = q; hi > 1; hi -= 32) {
        const int j = hi - 1 - lane;
        double v = j >= 1 ? (double)cn[j] : 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double u = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += u;
        }
        v += out;
        const unsigned ok = __ballot_sync(0xffffffffu, j >= 1 && v <= thr2);
        const int n = __ffs(~ok) - 1, cnt = n < 0 ? 32 : n;  // leading lanes that may go
        t -= cnt;
        if (cnt > 0) out = __shfl_sync(0xffffffffu, v, cnt - 1);
        if (cnt < 32) break;
      }
      // the cheapest tournament of t columns on at most NC CTAs
      const int nc = lane + 1, b = (t + 2 * nc - 1) / (2 * nc);
      float cost = FLT_MAX;
      if (nc <= NC && b <= a.bsx && (nc == 1 || (2 * nc - 2) * b < t)) cost = jac_cost<R>(nc, b, LP, RT);
      int best = nc;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float oc = __shfl_xor_sync(0xffffffffu, cost, o);
        const int on = __shfl_xor_sync(0xffffffffu, best, o);
        if (oc < cost || (oc == cost && on < best)) {
          cost = oc;
          best = on;
        }
      }
      if (lane == 0) {
        scan[0] = out;
        s_int[2] = best;
        s_int[3] = (t + 2 * best - 1) / (2 * best);
        s_int[4] = t;
      }
    }
    __syncthreads();
    NC = s_int[2];
    bs = s_int[3];
    qa = s_int[4];
    nthr = (bs * LP + 31) & ~31;
    if (rank >= NC || threadIdx.x >= nthr) return;  // (the barriers wait for the threads that are left)
  }
  const int ng = nthr / LP;
  const int NB = 2 * NC;
  const bool act = w < bs;       // this group has a column of either block
  const int wc = act ? w : 0;
  if (whole) {
    blocks([&](int c, int i, C* d) {
      C v(0, 0);
      if (c < qa && i < p) {
        const cplx<S> g = G[(int64_t)i * q + c];
        v = C((R)(sg * g.re), (R)(sg * g.im));
      } else if (PRE && c < qa && i == LP * RPL + c) {
        v = C(1, 0);
      }
      *d = v;
    });
    // (the partial sums lay where another CTA's columns arrive)
    if (NC > 1) cluster.sync(); else __syncthreads();
  } else {
    for (int e = threadIdx.x; e < 2 * bs * LD; e += nthr) slots[e] = (R)sg * slots[e];  // (bsx = bs)
    __syncthreads();
  }
  // Pairs are rotated down to a cosine of eps / 2, in FP64 at most 0.7 eps (the inner product's own
  // rounding is below that): what is left of the cosines is the vectors'
  // non-orthogonality, which the truncated train inherits once per bond (a
  // tolerance of eps sqrt(p) made it the largest error of a rounding, 1e-5 at
  // 128 columns).
  // (Rotations alone stop where the FP64 sweeps after them take two: what they
  // leave, about 1e-6, is squared by the first of them.)
  const R tol = PRE ? R(4) * Lim<R>::eps : R(0.5) * Lim<R>::eps, tol2 = tol * tol;
  // Quadratic regime: a rotation by sin s_ij of a pair (i, j) puts back s_ij g_jk
  // into an annihilated g_ik.  With c the largest cosine and s the largest
  // sine weighted by the norms' ratio of a sweep, the cosines after it are at
  // most about sqrt(qa) s c; with both at most sqrt(tol / sqrt(qa)) they are at
  // most tol, and the next sweep would rotate nothing.
  const R big2 = tol / sqrt(R(qa));
  C x[RT], y[RT];
  auto load = [&](C(&v)[RT], const C* s) {
#pragma unroll
    for (int u = 0; u < RT; ++u) v[u] = s[gl + LP * u];
  };
  auto store = [&](const C(&v)[RT], C* s) {
#pragma unroll
    for (int u = 0; u < RT; ++u) s[gl + LP * u] = v[u];
  };
  const int posn[2] = {rank, NB - 1 - rank};
  int dst_cta[2], dst_top[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int np = posn[h] == 0 ? 0 : (posn[h] == 1 ? NB - 1 : posn[h] - 1);
    dst_top[h] = np < NC;
    dst_cta[h] = np < NC ? np : NB - 1 - np;
  }
  int sweep = 0;
  for (; sweep < a.max_sweeps; ++sweep) {
    int wf = 0;
    // fresh norms of both blocks
    load(x, col(top, wc));
    load(y, col(bot, wc));
    {
      const R na = col_norm2<LP, RPL>(x), nb = col_norm2<LP, RPL>(y);
      if (gl == 0 && act) {
        nrm[top * a.bsx + w] = na;
        nrm[bot * a.bsx + w] = nb;
      }
    }
    __syncthreads();
    // pairs inside each block (round-robin of bs columns, one bye if bs is odd)
    const int be_ = bs + (bs & 1), half = be_ / 2;
    for (int s = 0; s + 1 < be_; ++s) {
      for (int k0 = 0; k0 < 2 * half; k0 += ng) {
        const int kk = min(k0 + w, 2 * half - 1);
        const int slot = kk < half ? top : bot, k = kk < half ? kk : kk - half;
        const int j0 = k == 0 ? 0 : 1 + (k - 1 + s) % (be_ - 1);
        const int k1 = be_ - 1 - k;
        const int j1 = 1 + (k1 - 1 + s) % (be_ - 1);
        const bool on = k0 + w < 2 * half && j0 < bs && j1 < bs;
        const int i0 = on ? j0 : 0, i1 = on ? j1 : 0;
        if (on) {
          load(x, col(slot, i0));
          load(y, col(slot, i1));
        }
        R al = nrm[slot * a.bsx + i0], be = nrm[slot * a.bsx + i1];
        const int f = rotate_pair<LP, RPL>(x, y, al, be, tol2, big2, lane, on);
        if (f) {
          wf |= f;
          store(x, col(slot, j0));
          store(y, col(slot, j1));
          if (gl == 0) {
            nrm[slot * a.bsx + j0] = al;
            nrm[slot * a.bsx + j1] = be;
          }
        }
      }
      __syncthreads();
    }
    for (int br = 0; br < NB - 1; ++br) {
      load(x, col(top, wc));
      R al = nrm[top * a.bsx + wc];
      int c = wc;
      for (int s = 0; s < bs; ++s) {
        if (act) load(y, col(bot, c));  // (an idle group's values are not used)
        R be = nrm[bot * a.bsx + c];
        const int f = rotate_pair<LP, RPL>(x, y, al, be, tol2, big2, lane, act);
        wf |= f;
        if (s + 1 < bs) {
          if (f) {
            store(y, col(bot, c));
            if (gl == 0) nrm[bot * a.bsx + c] = be;
          }
          __syncthreads();
          c = c + 1 == bs ? 0 : c + 1;
        } else if (!act) {
        } else if (NC > 1) {
          // both blocks to their next CTA, straight from the registers
          const int st = dst_top[0] ? in_top : in_bot, sb = dst_top[1] ? in_top : in_bot;
          C* rs = cluster.map_shared_rank(slots, dst_cta[0]);
          store(x, rs + (st * a.bsx + w) * LD);
          C* rb = cluster.map_shared_rank(slots, dst_cta[1]);
          store(y, rb + (sb * a.bsx + c) * LD);
          if (gl == 0) {
            cluster.map_shared_rank(nrm, dst_cta[0])[st * a.bsx + w] = al;
            cluster.map_shared_rank(nrm, dst_cta[1])[sb * a.bsx + c] = be;
          }
        } else {
          store(x, col(top, w));
          store(y, col(bot, c));
          if (gl == 0) {
            nrm[top * a.bsx + w] = al;
            nrm[bot * a.bsx + c] = be;
          }
        }
      }
      if (br == NB - 2) {
        if (gl == 0 && wf) atomicOr(&s_int[0], wf);
        __syncthreads();
        if (threadIdx.x < NC) cluster.map_shared_rank(flags, threadIdx.x)[(sweep & 1) * 16 + rank] = s_int[0];
      }
      if (NC > 1) {
        cluster.sync();
        int t = top;
        top = in_top;
        in_top = t;
        t = bot;
        bot = in_bot;
        in_bot = t;
      } else {
        __syncthreads();
      }
    }
    int any = 0;
    for (int i = 0; i < NC; ++i) any |= flags[(sweep & 1) * 16 + i];
    if (threadIdx.x == 0) s_int[0] = 0;  // next written after this sweep's barriers
    __syncthreads();
    if (!(any & 2)) {
      ++sweep;
      break;
    }
  }
  if (bt == 0 && rank == 0 && threadIdx.x == 0 && a.sweeps) *a.sweeps = sweep;
  // column norms (whole columns are local), gathered in every CTA
  load(x, col(top, wc));
  load(y, col(bot, wc));
  const R nx = sqrt(col_norm2<LP, RPL>(x)), ny = sqrt(col_norm2<LP, RPL>(y));
  const int cx = rank * bs + wc, cy = (NB - 1 - rank) * bs + wc;
  if (act)
    for (int i = gl; i < NC; i += LP) {
      R* rn = cluster.map_shared_rank(norms, i);
      rn[cx] = nx;
      rn[cy] = ny;
    }
  cluster.sync();
  // order by decreasing norm (ties by index; a NaN first, so that it stays a permutation)
  auto key = [&](int i) {
    const R v = norms[i];
    return v == v ? v : Lim<R>::big;
  };
  auto place = [&](int c) {
    const R v = key(c);
    int rk = 0;
    for (int i = gl; i < qa; i += LP) {
      const R u = key(i);
      rk += (u > v) || (u == v && i < c);
    }
    return gsum<LP>(rk);
  };
  if constexpr (PRE) {
    zc* Vt = a.Vt + bt * (int64_t)q * q;
    const int64_t eye = (int64_t)gridDim.y * q * q;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = h == 0 ? cx : cy;
      const int rk = place(min(c, qa - 1));
      if (c >= qa || !act) continue;
#pragma unroll
      for (int u = 0; u < RPL; ++u) {
        const int i = gl + LP * u;
        if (i >= q) continue;
        const C g = h == 0 ? x[RPL + u] : y[RPL + u];
        const int64_t o = (int64_t)rk * q + i;
        Vt[o] = zc(g.re, g.im);
        Vt[eye + o] = Vt[2 * eye + o] = zc(i == rk ? 1.0 : 0.0, 0.0);
      }
    }
    for (int e = rank * nthr + threadIdx.x; e < (q - qa) * q; e += NC * nthr) {  // dropped columns stay
      const int64_t o = (int64_t)qa * q + e;
      Vt[o] = Vt[eye + o] = Vt[2 * eye + o] = zc(o / q == o % q ? 1.0 : 0.0, 0.0);
    }
    return;
  }
  const R sb = dense::pow2(R(0), esc);
  for (int k0 = 0; k0 < qa; k0 += ng) {
    const int c = min(k0 + w, qa - 1), rk = place(c);
    if (gl == 0 && k0 + w < qa) sorted[rk] = norms[c] * sb;
  }
  __syncthreads();
  if (a.sigma && rank == 0)
    for (int i = threadIdx.x; i < q; i += nthr)  // (the dropped columns' norm as one value)
      a.sigma[bt * q + i] = i < qa ? sorted[i] : i == qa ? (R)(sqrt(scan[0]) * dense::pow2(0.0, esc)) : R(0);
  int keep = qa;
  if (a.trunc) {
    // smallest t >= 1 with sqrt(sum_{j >= t} s_j^2) <= delta, sums in double
    // by a suffix scan over the lanes, 32 values at a time from the end
    if (threadIdx.x < 32) {
      const double delta = a.deltas ? a.deltas[bt] : a.delta;
      const double sq = dense::pow2(0.0, esc);
      double tail = qa < q ? scan[0] * sq * sq : 0.0;
      int t = qa;
      bool stop = false;
      for (int hi = qa; hi > 1 && !stop; hi -= 32) {
        const int j = hi - 1 - lane;  // lane 0 the last value
        const double v = j >= 1 ? (double)sorted[j] : 0.0;
        double s = v * v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double u = __shfl_up_sync(0xffffffffu, s, o);
          if (lane >= o) s += u;
        }
        s += tail;
        const unsigned ok = __ballot_sync(0xffffffffu, j >= 1 && sqrt(s) <= delta);
        const int n = __ffs(~ok) - 1;  // leading lanes whose sums stay within delta (-1: all 32)
        const int cnt = n < 0 ? 32 : n;
        t -= cnt;
        if (cnt > 0) tail = __shfl_sync(0xffffffffu, s, cnt - 1);
        stop = cnt < 32;
      }
      int capped = 0;
      if (a.max_rank > 0 && t > a.max_rank) {
        double s = 0.0;
        for (int j = a.max_rank + lane; j < t; j += 32) s += (double)sorted[j] * (double)sorted[j];
        tail += dense::wsum(s);
        t = a.max_rank;
        capped = 1;
      }
      if (lane == 0) {
        s_int[1] = t;
        if (rank == 0) {
          int* o = a.trunc + 4 * bt;
          o[0] = t;
          o[1] = capped;
          *reinterpret_cast<double*>(o + 2) = sqrt(tail);
        }
      }
    }
    __syncthreads();
    keep = s_int[1];
  }
  // vectors, conjugated, one per row; columns with a subnormal norm carry no usable direction
  const int* perm = a.perm ? a.perm + bt * p : nullptr;
  C* Vh = a.Vh + bt * (int64_t)p * q;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = h == 0 ? cx : cy;
    const int rk = place(min(c, qa - 1));
    if (c >= qa || !act) continue;
    const R v = h == 0 ? nx : ny;
    R f = v > Lim<R>::tiny * R(4) ? R(1) / v : R(0);
    if (a.mask && rk >= keep) f = 0;
    C o[RPL];
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
      const C g = h == 0 ? x[u] : y[u];
      o[u] = f == R(0) ? C(0, 0) : C(g.re * f, -g.im * f);
    }
    if constexpr (sizeof(R) == 4) dense::unit_norm(o);
#pragma unroll
    for (int u = 0; u < RPL; ++u) {
      const int i = gl + LP * u;
      if (i < p) Vh[(int64_t)rk * p + (perm ? perm[i] : i)] = o[u];
    }
  }
  for (int e = rank * nthr + threadIdx.x; e < (q - qa) * p; e += NC * nthr) Vh[(int64_t)qa * p + e] = C(0, 0);
}

struct JacPlan {
  int nc, bs, lp, rpl, warps, bsx, adapt;
  size_t smem;
  double cost;  // cycles of a sweep
};

// instances: rows held by a group of lp lanes, rpl each
template <class R>
bool jac_rows(int p, int lp, int* rpl) {
  const int need = (p + lp - 1) / lp;
  auto first = [&](std::initializer_list<int> l) {
    for (int v : l)
      if (v >= need) {
        *rpl = v;
        return true;
      }
    return false;
  };
  if (sizeof(R) == 4) {
    return lp == 32 && first({1, 2, 3, 4, 5, 6, 8, 12, 16});
  }
  if (lp == 32) return first({1, 2, 3, 4, 5, 6, 8, 12, 16});
  return first({1, 2, 4});
}

template <class R>
size_t jac_smem(int q, int bs, int ld) {
  return (size_t)4 * bs * ld * sizeof(cplx<R>) + 16 + (4 * bs + (size_t)2 * (q + 64)) * sizeof(R) + 56 * sizeof(int) + 16;
}

// Cluster size, lanes per pair and column width, by the cost of a sweep in
// cycles: (2 nc - 1) block-rounds of bs rounds and one exchange, bs rounds inside
// the blocks.  A round costs its latency, or where that is more what its warps
// queue for: FP32 the issue slots; FP64 the FP64 unit of their quarter of the
// SM, which a warp instruction holds for 64 cycles (16 rows' worth per slice and
// about 27 for the scalars), so that four pairs an SM, one per quarter, are
// the most that run side by side.  An exchange costs a cluster barrier and two
// blocks through distributed shared memory at about 17 bytes a clock.
// Constants from clock readings inside the kernel (FP32 620 cycles a round at
// 118 rows, 720 at 256).  (FP32 gains nothing from two pairs a warp: 690 cycles
// a round at 16 rows against 650.)  us per sweep with powers of two of at most 8
// columns a block, and with this choice: 118 x 118 FP32 59.7 / 54.2, 256 x 136
// FP32 103.6 / 88.1, 128 x 72 FP32 39.9 / 32.8; FP64, with the FP64 instructions
// of the scalars cut from about 45 to 27, 68 x 68 376 / 224, 124 x 124 597 / 467.
template <class R>
bool jac_plan(int p, int q, int batch, JacPlan* pl, bool pre = false) {
  if (p < 1 || q < 1 || p > 512 || q > 512 || batch < 1 || batch > 65535) return false;
  int ncmax = 16;
  while (ncmax > 1 && ncmax * batch > 160) ncmax /= 2;
  double best = 1e300;
  for (int pass = 0; pass < 2 && best > 1e299; ++pass)  // second pass: whatever fits shared memory
    for (int lp : {32, 16}) {
      int rpl;
      if (!jac_rows<R>(p, lp, &rpl) || (pre && rpl > 8)) continue;
      const int wmax = sizeof(R) == 8 || pre || (rpl > 4 && rpl <= 8) ? 8 : 16;
      if (pre) rpl *= 2;
      for (int nc = 1; nc <= (pass ? 16 : ncmax); ++nc) {
        const int bs = (q + 2 * nc - 1) / (2 * nc), warps = (bs * lp + 31) / 32;
        if (nc > 1 && (2 * nc - 2) * bs >= q) continue;  // a CTA less would hold them
        const size_t sm = jac_smem<R>(q, bs, lp * rpl);
        if (warps > wmax || sm > 200 * 1024) continue;
        const double cost = jac_cost<R>(nc, bs, lp, rpl);
        if (cost < best) {
          best = cost;
          *pl = JacPlan{nc, bs, lp, pre ? rpl / 2 : rpl, warps, bs, 0, sm, cost};
        }
      }
    }
  return best < 1e299;
}

// Columns may be left out (see the kernel) where that can save more than the 5 us
// it takes to look for them (a sweep of 48 FP32 columns takes 19 us); a block may then be wider, since fewer CTAs can be
// quicker for fewer columns.
template <class R>
void jac_adapt(JacPlan* pl, int q, bool pre) {
  if (q < (sizeof(R) == 4 && !pre ? 48 : 24)) return;
  const int ld = pl->lp * pl->rpl * (pre ? 2 : 1), b = std::max(pl->bs, sizeof(R) == 4 ? 8 : 4);
  const size_t sm = jac_smem<R>(q, b, ld);
  const int threads = (b * pl->lp + 31) / 32 * 32;  // (a partial sum each, or per column)
  if (sm > 200 * 1024 ||
      ((size_t)(pl->nc + 1) * q + std::max(threads, q)) * sizeof(R) > (size_t)4 * b * ld * sizeof(cplx<R>))
    return;
  pl->bsx = b;
  pl->adapt = 1;
  pl->smem = sm;
  pl->warps = (b * pl->lp + 31) / 32;
}

template <class R, int LP, int RPL, bool PRE = false>
int launch(const JacArgs<R>& a, const JacPlan& pl, int batch, cudaStream_t s) {
  const void* fn = (const void*)jacobi_cluster2_kernel<R, LP, RPL, PRE>;
  if (qtt_allow_max_smem(fn) != QTT_OK) return QTT_ERR_CUDA;
  if (pl.nc > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return QTT_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)pl.nc, (unsigned)batch, 1);
  cfg.blockDim = dim3(32 * pl.warps, 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)pl.nc;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, jacobi_cluster2_kernel<R, LP, RPL, PRE>, a) == cudaSuccess ? QTT_OK : QTT_ERR_CUDA;
}

}  // namespace

template <class R>
bool qtt_svd_fits(int p, int q, int batch) {
  JacPlan pl;
  return jac_plan<R>(p, q, batch, &pl);
}

template <class R>
int qtt_svd(const cplx<R>* G, const int* perm, cplx<R>* Vh, R* sigma, int* trunc, double delta, const double* deltas,
            int max_rank, int mask, int p, int q, int batch, int max_sweeps, int* sweeps, cudaStream_t s) {
  JacPlan pl;
  if (!jac_plan<R>(p, q, batch, &pl)) return QTT_ERR_UNSUPPORTED;
  if (deltas || delta >= 0) jac_adapt<R>(&pl, q, false);
  const JacArgs<R> a{G, perm,  Vh,     sigma,    trunc,      delta,  deltas,  max_rank, mask,
                     p, q,     pl.bs,  pl.bsx,   pl.adapt,   max_sweeps, sweeps, nullptr, nullptr};
#define QTT_J(LP, RPL) \
  if (pl.lp == LP && pl.rpl == RPL) return launch<R, LP, RPL>(a, pl, batch, s)
  if constexpr (sizeof(R) == 4) {
    QTT_J(32, 1); QTT_J(32, 2); QTT_J(32, 3); QTT_J(32, 4); QTT_J(32, 5); QTT_J(32, 6); QTT_J(32, 8); QTT_J(32, 12);
    QTT_J(32, 16);
  } else {
    QTT_J(32, 1); QTT_J(32, 2); QTT_J(32, 3); QTT_J(32, 4); QTT_J(32, 5); QTT_J(32, 6); QTT_J(32, 8); QTT_J(32, 12);
    QTT_J(32, 16); QTT_J(16, 1); QTT_J(16, 2); QTT_J(16, 4);
  }
#undef QTT_J
  return QTT_ERR_UNSUPPORTED;
}

// FP32 rotations first where seven FP32 sweeps and the five products (about 80
// us at 70 columns) cost less than the 4.5 sweeps that they save; this is so from
// about 16 columns on (us of a rounding, without / with: 24 x 24 602 / 518, 16 x
// 16 378 / 349, 12 x 12 293 / 279, 16 x 8 212 / 224, 8 x 8 197 / 210).
bool qtt_svd_pre_fits(int p, int q, int batch) {
  JacPlan pd, pf;
  if (p < q || !jac_plan<double>(p, q, batch, &pd) || !jac_plan<float>(p, q, batch, &pf, true)) return false;
  return 4.5 * pd.cost > 7.0 * pf.cost + 1.5e5;
}

int qtt_svd_pre(const zc* G, zc* Vt, double delta, const double* deltas, int p, int q, int batch,
                int* sweeps, cudaStream_t s) {
  JacPlan pl;
  if (p < q || !jac_plan<float>(p, q, batch, &pl, true)) return QTT_ERR_UNSUPPORTED;
  if (deltas || delta >= 0) jac_adapt<float>(&pl, q, true);
  const JacArgs<float> a{nullptr, nullptr, nullptr, nullptr, nullptr,  delta, deltas, 0, 0,
                         p,       q,       pl.bs,   pl.bsx,  pl.adapt, 30,    sweeps, G, Vt};
#define QTT_J(RPL) \
  if (pl.rpl == RPL) return launch<float, 32, RPL, true>(a, pl, batch, s)
  QTT_J(1); QTT_J(2); QTT_J(3); QTT_J(4); QTT_J(5); QTT_J(6); QTT_J(8);
#undef QTT_J
  return QTT_ERR_UNSUPPORTED;
}

template bool qtt_svd_fits<float>(int, int, int);
template bool qtt_svd_fits<double>(int, int, int);
template int qtt_svd<float>(const cc*, const int*, cc*, float*, int*, double, const double*, int, int, int, int, int, int,
                            int*, cudaStream_t);
template int qtt_svd<double>(const zc*, const int*, zc*, double*, int*, double, const double*, int, int, int, int, int,
                             int, int*, cudaStream_t);
