// Householder QR of small dense matrices by one thread-block cluster per
// matrix.
//
// What bounds it: the columns form a chain (reflector j needs column j after
// reflectors 0 .. j-1), so time = columns x latency of one column step, plus,
// in FP64, the arithmetic itself (two FP64 FMAs per clock and SM on this
// part).  One SM working alone (blocked FP32 / panel FP64 kernel of linalg.cu)
// against this kernel, us per matrix: 272 x 136 FP32 with Q 660 / 194, 256 x
// 128 FP32 R only 470 / 135, 512 x 256 FP32 R only 2450 / 410, 144 x 72 FP64
// with Q 1765 / 537, 148 x 74 FP64 R only 2800 / 418.  Here the
// columns are dealt to the CTAs of a cluster in panels of `b` columns
// (panel p to CTA p mod NC, slot p / NC) and stay in that CTA's shared memory:
//   * the CTA that owns panel p factors it, one warp per column with the
//     column in registers.  Reflectors are kept unscaled, v = (v0, x_{j+1}, ...)
//     with v0 = x_j - alpha, so the later columns' products with the raw column
//     run while its own warp still forms the norm and the two scalars (in FP64
//     a chain of dependent operations of 75 cycles each);
//   * the reflectors go to the workspace V (column-major), one cluster barrier
//     publishes the panel, every CTA stages it in shared memory and its warps
//     apply the b reflectors to their later columns in registers;
//   * the explicit Q is formed at the end, columns dealt round-robin over the
//     CTAs, one warp per column holding Q e_c = H_0 ... H_c e_c in registers
//     while the panels are staged once more, last first.
// The panel width trades the per-panel cost (cluster barrier, staging) against
// the work that one SM does alone: see plan().
// Optionally the columns are taken in the order of decreasing norm (perm),
// which is what lets the Jacobi SVD of R^H converge in a third of the sweeps.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "dense.cuh"
#include "kernels.h"

namespace {

namespace cg = cooperative_groups;
using dense::Lim;

// threads per CTA (a panel has at most one column per warp): two FP64 columns of
// up to 512 rows need more than the 128 registers that 16 warps leave a thread
template <class R>
struct QrThreads {
  static constexpr int value = sizeof(R) == 8 ? 256 : 512;
};

template <class R>
struct QrArgs {
  const cplx<R>* in;
  MIdx inB, rowI, colI;
  int conj_in, m, n, b, slots;
  int64_t rows_total, rows_per_batch;
  cplx<R>* V;  // min(m, n) columns of m per matrix: rows > j of reflector j, v0 at row j
  R* taus;     // n per matrix
  cplx<R>* out;
  int64_t out_bstride, ldr;
  int out_rh;  // 1: out = R^H (n x min(m, n), leading dimension ldr) instead of R
  int* perm;   // non-null: columns by decreasing norm, perm[c] = the input column at place c
  cplx<R>* Q;
  int64_t q_bstride, ldq;
};

// sum of w over the warp, in every lane.  FP64: the halves of the warp sum the
// real and the imaginary part, which takes five additions instead of ten (one
// holds the FP64 pipe for 16 cycles).
template <class R>
__device__ __forceinline__ cplx<R> wsum_c(cplx<R> w, int lane) {
  if constexpr (sizeof(R) == 4) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      w.re += __shfl_xor_sync(0xffffffffu, w.re, o);
      w.im += __shfl_xor_sync(0xffffffffu, w.im, o);
    }
    return w;
  } else {
    const bool up = lane & 16;
    R v = (up ? w.im : w.re) + __shfl_xor_sync(0xffffffffu, up ? w.re : w.im, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return cplx<R>(__shfl_sync(0xffffffffu, v, 0), __shfl_sync(0xffffffffu, v, 16));
  }
}

// 32-row slices above `us` hold zeros of the reflectors: FP64 skips them, FP32
// (bound by latency) runs faster without the branches
template <class R>
__device__ __forceinline__ bool skip(int u, int us) {
  return sizeof(R) == 8 && u < us;
}

// v^H x over the warp, v (in shared memory) left in vv
template <class R, int RPL>
__device__ __forceinline__ cplx<R> vhx(cplx<R> (&vv)[RPL], const cplx<R>* v, const cplx<R> (&x)[RPL], int us, int lane) {
  cplx<R> w(0, 0), w1(0, 0);
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    if (skip<R>(u, us)) continue;
    vv[u] = v[lane + 32 * u];
    if (u & 1) cfma_conj(w1, vv[u], x[u]); else cfma_conj(w, vv[u], x[u]);
  }
  return wsum_c(w + w1, lane);
}

// x -= vv w
template <class R, int RPL>
__device__ __forceinline__ void sub_vw(cplx<R> (&x)[RPL], const cplx<R> (&vv)[RPL], cplx<R> w, int us) {
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    if (skip<R>(u, us)) continue;
    x[u].re = fma(-vv[u].re, w.re, fma(vv[u].im, w.im, x[u].re));
    x[u].im = fma(-vv[u].re, w.im, fma(-vv[u].im, w.re, x[u].im));
  }
}

template <class R, int RPL>
__device__ __forceinline__ void reflect(cplx<R> (&x)[RPL], const cplx<R>* v, R tau, int us, int lane) {
  cplx<R> vv[RPL];
  const cplx<R> w = tau * vhx<R, RPL>(vv, v, x, us, lane);
  sub_vw<R, RPL>(x, vv, w, us);
}

// Scalars of reflector j of the column in x (rows on the lanes): v0 = x_j - alpha
// with alpha = -e^{i arg x_j} ||x_{j:}||, tau = 2 / (|v0|^2 + ||x_{j+1:}||^2).  A
// column whose norm, or whose part below row j, is at most zero2 (the square
// of eps ||A||_F) gets tau = 0.  Row j of x becomes the diagonal of R.
// FP32 sums the squares with compensation (a plain FP32 sum raised the
// solver's error threefold).
template <class R, int RPL>
__device__ __forceinline__ R reflector_scalars(cplx<R> (&x)[RPL], int j, R zero2, int lane, cplx<R>* v0_out) {
  R hi = 0, lo = 0, hi1 = 0, lo1 = 0;
  cplx<R> x0(0, 0);
  const int js = j >> 5;
#pragma unroll
  for (int u = 0; u < RPL; ++u) {
    if (skip<R>(u, js)) continue;
    const R a2 = lane + 32 * u > j ? abs2(x[u]) : R(0);
    if constexpr (sizeof(R) == 4) {
      if (u & 1) dense::add_comp(hi1, lo1, a2); else dense::add_comp(hi, lo, a2);
    } else {
      if (u & 1) hi1 += a2; else hi += a2;
    }
    if (lane + 32 * u == j) x0 = x[u];
  }
  x0.re = __shfl_sync(0xffffffffu, x0.re, j & 31);
  x0.im = __shfl_sync(0xffffffffu, x0.im, j & 31);
  if constexpr (sizeof(R) == 4) {
    lo += lo1;
    dense::add_comp(hi, lo, hi1);
    dense::wsum_comp(hi, lo);
    hi += lo;
  } else {
    hi = dense::wsum(hi + hi1);
  }
  const R below = hi, ax2 = abs2(x0), nrm2 = below + ax2;
  const bool zero = nrm2 <= zero2 || below <= zero2;  // false for a NaN, which then spreads
  R tau = 0;
  cplx<R> v0(0, 0), diag = nrm2 <= zero2 ? cplx<R>(0, 0) : x0;
  if (!zero) {
    const R nrm = nrm2 * dense::rsqrt_nr(nrm2);
    cplx<R> ph(1, 0);
    if (ax2 >= Lim<R>::tiny) {
      const R ra = dense::rsqrt_nr(ax2);
      ph = cplx<R>(x0.re * ra, x0.im * ra);
    }
    diag = cplx<R>(-ph.re * nrm, -ph.im * nrm);
    v0 = x0 - diag;
    tau = R(2) * dense::rcp_nr(below + abs2(v0));
  }
#pragma unroll
  for (int u = 0; u < RPL; ++u)
    if (lane + 32 * u == j) x[u] = diag;
  *v0_out = v0;
  return tau;
}

template <class R>
__device__ __forceinline__ cplx<R> load_l2(const cplx<R>* p) {
  if constexpr (sizeof(R) == 4) {
    const float2 t = __ldcg(reinterpret_cast<const float2*>(p));
    return cplx<R>(t.x, t.y);
  } else {
    const double2 t = __ldcg(reinterpret_cast<const double2*>(p));
    return cplx<R>(t.x, t.y);
  }
}

template <class R, int RPL>
__global__ void __launch_bounds__(QrThreads<R>::value, 1)
qr_cluster_kernel(const __grid_constant__ QrArgs<R> a) {
  typedef cplx<R> C;
  cg::cluster_group cluster = cg::this_cluster();
  const int NC = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int m = a.m, n = a.n, b = a.b, kmax = min(m, n);
  constexpr int LD = 32 * RPL;  // rows, padded with zeros
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int QT = QrThreads<R>::value, NW = QT / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* cols = reinterpret_cast<C*>(smem_raw);            // slots * b columns of LD
  C* Vs = cols + (size_t)a.slots * b * LD;             // the panel being applied
  C* v0s = Vs + (size_t)b * LD;                        // 16
  R* taus = reinterpret_cast<R*>(v0s + 16);            // 16
  R* parts = taus + 16;                                // 16 warp partials, then 16 CTA sums
  int* exps = reinterpret_cast<int*>(parts + 32);      // 16 CTA exponents, then 1 of this CTA
  int* perm = exps + 20;                               // n (sorted columns only)
  R* keys = reinterpret_cast<R*>(perm + (a.perm ? (n + 3) / 4 * 4 : 0));  // n (sorted columns only)
  const int64_t bt = blockIdx.y;
  const C* in = a.in + midx_off(a.inB, bt);
  C* V = a.V + bt * (int64_t)m * n;
  R* tg = a.taus + bt * n;
  int64_t valid = a.rows_total - bt * a.rows_per_batch;
  if (valid > m) valid = m;
  // CTAs of a cluster may touch each other's shared memory once all have started
  cluster.sync();
  if (a.perm) {
    // key of a column: the sum of |re| + |im| (no squares, which could leave the range)
    for (int c = rank + NC * warp; c < n; c += NC * NW) {
      const int64_t co = midx_off(a.colI, c);
      R s = 0;
      for (int i = lane; i < valid; i += 32) {
        const C v = in[midx_off(a.rowI, i) + co];
        s += fabs(v.re) + fabs(v.im);
      }
      s = dense::wsum(s);
      if (!(s <= Lim<R>::big)) s = Lim<R>::big;  // NaN or infinity first: the order stays a permutation
      if (lane < NC) cluster.map_shared_rank(keys, lane)[c] = s;
    }
    cluster.sync();
    for (int c = threadIdx.x; c < n; c += QT) {
      const R v = keys[c];
      int rk = 0;
      for (int i = 0; i < n; ++i) {
        const R u = keys[i];
        rk += (u > v) || (u == v && i < c);
      }
      perm[rk] = c;
    }
    __syncthreads();
    if (rank == 0)
      for (int c = threadIdx.x; c < n; c += QT) a.perm[bt * n + c] = perm[c];
  }
  // This CTA's columns, scaled by a power of two so that the largest component
  // of the matrix is in [1, 2): squares and reciprocals then stay in range
  // whatever the matrix's norm.  One exchange: every CTA sums its squares at
  // its own scale.
  int esc;
  R zero2;
  {
    const int tot = a.slots * b;
    const bool cfast = (a.colI.n2 == 1 ? a.colI.s1 : a.colI.s2) == 1;
    R amax = 0;
    for (int e = threadIdx.x; e < tot * LD; e += QT) {
      int lc, i;
      if (cfast) {
        i = e / tot;
        lc = e - i * tot;
      } else {
        lc = e / LD;
        i = e - lc * LD;
      }
      const int sl = lc / b, c = (sl * NC + rank) * b + (lc - sl * b);
      C v(0, 0);
      if (c < n && i < valid) {
        v = in[midx_off(a.rowI, i) + midx_off(a.colI, a.perm ? perm[c] : c)];
        if (a.conj_in) v.im = -v.im;
      }
      cols[(size_t)lc * LD + i] = v;
      amax = fmax(amax, fmax(fabs(v.re), fabs(v.im)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (lane == 0) parts[warp] = amax;
    __syncthreads();
    if (warp == 0) {
      R t = lane < NW ? parts[lane] : R(0);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t = fmax(t, __shfl_xor_sync(0xffffffffu, t, o));
      if (lane == 0) exps[16] = dense::exponent_of(t, sizeof(R) == 4 ? -120 : -1000);
    }
    __syncthreads();
    const int el = exps[16];
    const R sl = dense::pow2(R(0), -el);
    R part = 0;
    for (int e = threadIdx.x; e < tot * LD; e += QT) part += abs2(sl * cols[e]);
    part = dense::wsum(part);
    if (lane == 0) parts[warp] = part;
    __syncthreads();
    if (warp == 0) {
      R s = lane < NW ? parts[lane] : R(0);
      s = dense::wsum(s);
      if (lane < NC) {
        cluster.map_shared_rank(parts, lane)[16 + rank] = s;
        cluster.map_shared_rank(exps, lane)[rank] = el;
      }
    }
    cluster.sync();
    esc = exps[0];
    for (int i = 1; i < NC; ++i) esc = max(esc, exps[i]);
    R fro2 = 0;
    for (int i = 0; i < NC; ++i) fro2 += parts[16 + i] * dense::pow2(R(0), max(2 * (exps[i] - esc), sizeof(R) == 4 ? -120 : -1000));
    zero2 = Lim<R>::eps * Lim<R>::eps * fro2;
    const R sg = dense::pow2(R(0), -esc);
    for (int e = threadIdx.x; e < tot * LD; e += QT) cols[e] = sg * cols[e];
    __syncthreads();
  }
  C x[RPL];
  auto load_col = [&](int lc) {
#pragma unroll
    for (int u = 0; u < RPL; ++u) x[u] = cols[(size_t)lc * LD + lane + 32 * u];
  };
  auto store_col = [&](int lc) {
#pragma unroll
    for (int u = 0; u < RPL; ++u) cols[(size_t)lc * LD + lane + 32 * u] = x[u];
  };
  // reflectors c0 .. c0+pw-1 from the workspace (written by another SM: read from L2)
  auto stage = [&](int c0, int pw) {
    for (int jj = warp; jj < pw; jj += NW) {
      const int j = c0 + jj;
#pragma unroll
      for (int u = 0; u < RPL; ++u) {
        const int i = lane + 32 * u;
        Vs[(size_t)jj * LD + i] = i >= j && i < m ? load_l2(V + (size_t)j * m + i) : C(0, 0);
      }
      if (lane == 0) taus[jj] = __ldcg(tg + j);
    }
  };
  // ------------------------------------------------------------- R
  const int npan = (kmax + b - 1) / b;
  for (int p = 0; p < npan; ++p) {
    const int c0 = p * b, pw = min(b, kmax - c0), pc = min(b, n - c0), us = c0 >> 5;
    const bool owner = rank == p % NC;
    if (owner && warp < pc) {
      // one warp per column.  Per column: its warp writes the raw column below
      // row j; the dot products of the later columns with it and the
      // reflector's scalars are then formed at the same time, two barriers a step
      const int lc = (p / NC) * b + warp;
      load_col(lc);
      for (int jj = 0; jj < pw; ++jj) {
        const int j = c0 + jj;
        C* v = Vs + (size_t)jj * LD;
        if (warp == jj) {
#pragma unroll
          for (int u = 0; u < RPL; ++u) v[lane + 32 * u] = lane + 32 * u > j ? x[u] : C(0, 0);
        }
        asm volatile("bar.sync 1, %0;" ::"r"(32 * pc) : "memory");
        C vv[RPL], w(0, 0), xj(0, 0);
        if (warp == jj) {
          C v0;
          const R tau = reflector_scalars<R, RPL>(x, j, zero2, lane, &v0);
          if (lane == 0) {
            taus[jj] = tau;
            v0s[jj] = v0;
          }
        } else if (warp > jj) {
          w = vhx<R, RPL>(vv, v, x, us, lane);
#pragma unroll
          for (int u = 0; u < RPL; ++u)
            if (lane + 32 * u == j) xj = x[u];
          xj.re = __shfl_sync(0xffffffffu, xj.re, j & 31);
          xj.im = __shfl_sync(0xffffffffu, xj.im, j & 31);
        }
        asm volatile("bar.sync 1, %0;" ::"r"(32 * pc) : "memory");
        if (warp > jj) {
          const R tau = taus[jj];
          if (tau != R(0)) {
            const C v0 = v0s[jj];
            cfma_conj(w, v0, xj);
            w = tau * w;
#pragma unroll
            for (int u = 0; u < RPL; ++u) {
              if (skip<R>(u, us)) vv[u] = C(0, 0);
              if (lane + 32 * u == j) vv[u] = v0;
            }
            sub_vw<R, RPL>(x, vv, w, us);
          }
        } else if (warp == jj) {
          // row j completed (the products above read it as zero), and the
          // reflector to the workspace, for the other CTAs
#pragma unroll
          for (int u = 0; u < RPL; ++u) {
            const int i = lane + 32 * u;
            if (i > j && i < m) V[(size_t)j * m + i] = x[u];
          }
          if (lane == 0) {
            v[j] = v0s[jj];
            V[(size_t)j * m + j] = v0s[jj];
            tg[j] = taus[jj];
          }
        }
      }
      store_col(lc);
    }
    if (c0 + b >= n) break;  // nothing to the right
    if (NC > 1) cluster.sync(); else __syncthreads();
    // later columns of this CTA: slots s with panel s * NC + rank > p
    const int s0 = rank > p % NC ? p / NC : p / NC + 1;
    if ((s0 * NC + rank) * b < n) {
      if (!owner) stage(c0, pw);
      __syncthreads();
      for (int lc = s0 * b + warp; lc < a.slots * b; lc += NW) {
        const int sl = lc / b, c = (sl * NC + rank) * b + (lc - sl * b);
        if (c >= n) continue;
        load_col(lc);
        for (int jj = 0; jj < pw; ++jj) {
          const R tau = taus[jj];
          if (tau != R(0)) reflect<R, RPL>(x, Vs + (size_t)jj * LD, tau, us, lane);
        }
        store_col(lc);
      }
      __syncthreads();
    }
  }
  if (a.out) {
    __syncthreads();
    const R sb = dense::pow2(R(0), esc);
    C* o = a.out + bt * a.out_bstride;
    for (int lc = warp; lc < a.slots * b; lc += NW) {
      const int sl = lc / b, c = (sl * NC + rank) * b + (lc - sl * b);
      if (c >= n) continue;
      for (int i = lane; i < kmax; i += 32) {
        const C v = i <= c ? sb * cols[(size_t)lc * LD + i] : C(0, 0);
        if (a.out_rh)
          o[(int64_t)c * a.ldr + i] = conjg(v);
        else
          o[(int64_t)i * a.ldr + c] = v;
      }
    }
  }
  if (!a.Q) return;
  // ------------------------------------------------------------- explicit Q
  if (NC > 1) cluster.sync();  // every panel is in V
  C* Q = a.Q + bt * a.q_bstride;
  for (int g0 = 0; g0 < kmax; g0 += NC * NW) {
    const int c = g0 + warp * NC + rank;
    const int cmax = min(kmax, g0 + NC * NW) - 1;
#pragma unroll
    for (int u = 0; u < RPL; ++u) x[u] = C(lane + 32 * u == c ? R(1) : R(0), R(0));
    for (int p = cmax / b; p >= 0; --p) {
      const int c0 = p * b, pw = min(b, kmax - c0), us = c0 >> 5;
      __syncthreads();
      stage(c0, pw);
      __syncthreads();
      if (c < kmax && c >= c0)
        for (int jj = min(pw - 1, c - c0); jj >= 0; --jj) {
          const R tau = taus[jj];
          if (tau != R(0)) reflect<R, RPL>(x, Vs + (size_t)jj * LD, tau, us, lane);
        }
    }
    if (c < kmax) {
      if constexpr (sizeof(R) == 4) dense::unit_norm(x);
#pragma unroll
      for (int u = 0; u < RPL; ++u) {
        const int i = lane + 32 * u;
        if (i < m) Q[(int64_t)i * a.ldq + c] = x[u];
      }
    }
  }
}

struct QrPlan {
  int nc, b, slots;
  size_t smem;
};

// Cluster size and panel width for an m x n matrix, `batch` of them.
//   * n <= 16: one CTA holds every column; a cluster's barriers would cost
//     more than they save.
//   * FP32: panels of 8 columns.  A panel costs its chain of column steps
//     (1250 cycles each at 256 rows), then barrier, staging and update (about
//     6 500 together); 256 x 128 took 154 / 135 / 148 us with 4 / 8 / 16.
//   * FP64: panels of 4 (2 up to 32 columns).  The update of a panel holds the
//     SM's FP64 pipe, so narrow panels spread over more SMs: 148 x 74 took
//     420 / 418 / 533 us with 2 / 4 / 8.
//   * Many matrices share the device: at most about one CTA per SM in all.
// 32-row slices of the instance that takes m rows
int qr_slices(int m) {
  const int nu = (m + 31) / 32;
  return nu <= 6 ? nu : nu <= 8 ? 8 : nu <= 9 ? 9 : nu <= 12 ? 12 : 16;
}

template <class R>
bool qr_plan(int64_t m, int64_t n, int64_t batch, bool sort, QrPlan* pl) {
  if (m < 1 || n < 1 || m > 512) return false;
  const int ldm = 32 * qr_slices((int)m);
  int ncmax = 16;
  while (ncmax > 1 && ncmax * batch > 160) ncmax /= 2;
  for (int nc = 1; nc <= 16; nc *= 2) {
    // smallest cluster that the columns ask for, larger only to fit shared memory
    int b, want;
    if (n <= 16) {
      b = (int)std::min<int64_t>(n, sizeof(R) == 8 ? 8 : 16);
      want = 1;
    } else if (sizeof(R) == 4) {
      b = 8;
      want = (int)std::min<int64_t>(ncmax, (n + b - 1) / b);
    } else {
      b = n <= 32 ? 2 : 4;
      want = (int)std::min<int64_t>(ncmax, (n + b - 1) / b);
    }
    int w2 = 1;
    while (w2 < want) w2 *= 2;
    const int use = std::max(nc, w2);
    const int pans = (int)((n + b - 1) / b), slots = (pans + use - 1) / use;
    const size_t sm = (((size_t)slots * b + b) * ldm + 16) * sizeof(cplx<R>) + (48 + (sort ? n : 0)) * sizeof(R) +
                      (24 + (sort ? n : 0)) * sizeof(int) + 32;
    if (sm <= 200 * 1024) {
      *pl = QrPlan{use, b, slots, sm};
      return true;
    }
  }
  return false;
}

template <class R, int RPL>
int launch(const QrArgs<R>& a, const QrPlan& pl, int64_t batch, cudaStream_t s) {
  const void* fn = (const void*)qr_cluster_kernel<R, RPL>;
  if (qtt_allow_max_smem(fn) != QTT_OK) return QTT_ERR_CUDA;
  if (pl.nc > 8 && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return QTT_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)pl.nc, (unsigned)batch, 1);
  cfg.blockDim = dim3(QrThreads<R>::value, 1, 1);
  cfg.dynamicSmemBytes = pl.smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)pl.nc;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, qr_cluster_kernel<R, RPL>, a) == cudaSuccess ? QTT_OK : QTT_ERR_CUDA;
}

}  // namespace

template <class R>
bool qtt_qr_cluster_fits(int64_t m, int64_t n, int64_t batch) {
  QrPlan pl;
  return batch >= 1 && batch <= 65535 && qr_plan<R>(m, n, batch, true, &pl);
}
template bool qtt_qr_cluster_fits<float>(int64_t, int64_t, int64_t);
template bool qtt_qr_cluster_fits<double>(int64_t, int64_t, int64_t);

template <class R>
int qtt_qr_cluster(const cplx<R>* in, MIdx inB, MIdx rowI, MIdx colI, int conj_in, int64_t m, int64_t n,
                   int64_t rows_total, int64_t rows_per_batch, int64_t batch, cplx<R>* V, cplx<R>* out,
                   int64_t out_bstride, int64_t ldr, int out_rh, int* perm, cplx<R>* Qout, int64_t q_bstride,
                   int64_t ldq, cudaStream_t s) {
  QrPlan pl;
  if (batch < 1 || batch > 65535 || !qr_plan<R>(m, n, batch, perm != nullptr, &pl)) return QTT_ERR_UNSUPPORTED;
  QrArgs<R> a;
  a.in = in;
  a.inB = inB;
  a.rowI = rowI;
  a.colI = colI;
  a.conj_in = conj_in;
  a.m = (int)m;
  a.n = (int)n;
  a.b = pl.b;
  a.slots = pl.slots;
  a.rows_total = rows_total;
  a.rows_per_batch = rows_per_batch;
  a.V = V;
  a.taus = reinterpret_cast<R*>(V + batch * m * n);
  a.out = out;
  a.out_bstride = out_bstride;
  a.ldr = ldr;
  a.out_rh = out_rh;
  a.perm = perm;
  a.Q = Qout;
  a.q_bstride = q_bstride;
  a.ldq = ldq;
  switch (qr_slices((int)m)) {
    case 1: return launch<R, 1>(a, pl, batch, s);
    case 2: return launch<R, 2>(a, pl, batch, s);
    case 3: return launch<R, 3>(a, pl, batch, s);
    case 4: return launch<R, 4>(a, pl, batch, s);
    case 5: return launch<R, 5>(a, pl, batch, s);
    case 6: return launch<R, 6>(a, pl, batch, s);
    case 8: return launch<R, 8>(a, pl, batch, s);
    case 9: return launch<R, 9>(a, pl, batch, s);
    case 12: return launch<R, 12>(a, pl, batch, s);
    default: return launch<R, 16>(a, pl, batch, s);
  }
}
template int qtt_qr_cluster<float>(const cc*, MIdx, MIdx, MIdx, int, int64_t, int64_t, int64_t, int64_t, int64_t, cc*,
                                   cc*, int64_t, int64_t, int, int*, cc*, int64_t, int64_t, cudaStream_t);
template int qtt_qr_cluster<double>(const zc*, MIdx, MIdx, MIdx, int, int64_t, int64_t, int64_t, int64_t, int64_t, zc*,
                                    zc*, int64_t, int64_t, int, int*, zc*, int64_t, int64_t, cudaStream_t);
