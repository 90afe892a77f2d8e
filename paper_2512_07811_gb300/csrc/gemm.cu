// Batched complex GEMM over two-level multi-indices (CUDA cores, FP64 / FP32).
//
// Every core contraction of the tensor-train path (absorbing R or U*S into a
// neighbouring core, transfer matrices of inner products, the structured
// sketch contractions of operator-times-train products) is one call of this
// kernel with suitable index strides, so no contraction needs an explicit
// permutation pass.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace {

// With splits > 1 every CTA sums only its share of K and stores the raw
// partial tile to P[split][batch][m][n] (dense); a second kernel reduces the
// partials in split order and applies alpha, beta and the output strides.
//
// Index arithmetic: the element offsets of the tile's BM rows of A and BN
// columns of B are computed once per CTA, those of each K-tile's BK values
// once per tile (two tiles ahead, in a ring of three), so the loads do no
// division.  Threads walk a tile along whichever index is contiguous in
// memory (k or m for A, k or n for B) so that neighbouring threads read
// neighbouring elements.  The main loop is software-pipelined: the next
// tile is loaded into registers while the current one is multiplied from
// shared memory.
//
// Sums: every 8 values of k are summed on their own and then added to the
// accumulator.  In one FP32 chain over k the rounding errors of the long
// running sum add up (K u at worst where all terms have one sign, as in the
// mean fields of a solve): these sums were the largest part of a complex64
// solve's error.  With runs of 8 it is (8 + K / 8) u.  C_eff of a 16^3 sphere with
// exact operators, rms over 24 solves 1.7e-6 / 1.2e-6 / 1.3e-6 with runs of 16 / 8 / 4
// (one chain 2.9e-6 / runs of 8 1.8e-6 before the QR and the SVD set their vectors'
// norms right); roundings 1.1 to 2.1 times more exact; the sums cost 3 % of a
// contrast step at rank 128 (11.34 / 11.70 ms), compensated ones 8-20 % for 0.9e-6.
QTT_HD bool midx_unit_inner(const MIdx& m) { return (m.n2 == 1 ? m.s1 : m.s2) == 1; }

template <class R, int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
gemm_midx_kernel(GemmDesc g, cplx<R> alpha, cplx<R> beta,
                 const cplx<R>* __restrict__ A, const cplx<R>* __restrict__ B,
                 cplx<R>* __restrict__ C, int splits, int64_t kchunk, cplx<R>* __restrict__ P) {
  constexpr int NT = (BM / TM) * (BN / TN);
  constexpr int TX = BN / TN;
  constexpr int LA = BM * BK / NT, LB = BN * BK / NT;  // tile elements each thread loads
  static_assert(2 * BK <= NT && LA * NT == BM * BK && LB * NT == BN * BK, "tile shape");
  __shared__ cplx<R> As[BK][BM + 1];
  __shared__ cplx<R> Bs[BK][BN + 1];
  __shared__ int64_t rowA[BM], colB[BN], kOffA[3][BK], kOffB[3][BK];

  const int64_t b = blockIdx.z / splits;
  const int split = blockIdx.z - (int)(b * splits);
  const int64_t kbeg = (int64_t)split * kchunk;
  const int64_t kend = min(g.K, kbeg + kchunk);
  const int64_t m0 = (int64_t)blockIdx.y * BM;
  const int64_t n0 = (int64_t)blockIdx.x * BN;
  const int tid = threadIdx.x;
  const int tx = tid % TX, ty = tid / TX;
  const int ntiles = kend > kbeg ? (int)((kend - kbeg + BK - 1) / BK) : 0;

  const int64_t offA = midx_off(g.bA, b), offB = midx_off(g.bB, b), offC = midx_off(g.bC, b);
  for (int i = tid; i < BM; i += NT) rowA[i] = (m0 + i < g.M) ? offA + midx_off(g.mA, m0 + i) : -1;
  for (int i = tid; i < BN; i += NT) colB[i] = (n0 + i < g.N) ? offB + midx_off(g.nB, n0 + i) : -1;
  // K offsets of tile t live in slot t mod 3, computed two tiles ahead
  auto koffs = [&](int t) {
    const int sl = t % 3;
    if (tid < BK) {
      const int64_t k = kbeg + (int64_t)t * BK + tid;
      kOffA[sl][tid] = k < kend ? midx_off(g.kA, k) : -1;
    } else if (tid < 2 * BK) {
      const int64_t k = kbeg + (int64_t)t * BK + tid - BK;
      kOffB[sl][tid - BK] = k < kend ? midx_off(g.kB, k) : -1;
    }
  };
  koffs(0);
  koffs(1);
  const bool a_kfast = midx_unit_inner(g.kA) && !midx_unit_inner(g.mA);
  const bool b_kfast = midx_unit_inner(g.kB) && !midx_unit_inner(g.nB);
  __syncthreads();

  // global -> registers for tile t (this thread's LA + LB elements)
  cplx<R> ra[LA], rb[LB];
  auto fetch = [&](int t) {
    const int sl = t % 3;
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = tid + l * NT;
      const int mm = a_kfast ? e / BK : e % BM;
      const int kk = a_kfast ? e % BK : e / BM;
      const int64_t r = rowA[mm], k = kOffA[sl][kk];
      cplx<R> v(0, 0);
      if (r >= 0 && k >= 0) {
        v = A[r + k];
        if (g.conjA) v.im = -v.im;
      }
      ra[l] = v;
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = tid + l * NT;
      const int nn = b_kfast ? e / BK : e % BN;
      const int kk = b_kfast ? e % BK : e / BN;
      const int64_t c = colB[nn], k = kOffB[sl][kk];
      cplx<R> v(0, 0);
      if (c >= 0 && k >= 0) {
        v = B[c + k];
        if (g.conjB) v.im = -v.im;
      }
      rb[l] = v;
    }
  };

  constexpr int RUN = 8;  // values of k summed before they join the accumulator
  static_assert(BK % RUN == 0, "runs end with a tile");
  cplx<R> acc[TM][TN], part[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = part[i][j] = cplx<R>(0, 0);

  if (ntiles > 0) fetch(0);
  for (int t = 0; t < ntiles; ++t) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = tid + l * NT;
      As[a_kfast ? e % BK : e / BM][a_kfast ? e / BK : e % BM] = ra[l];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = tid + l * NT;
      Bs[b_kfast ? e % BK : e / BN][b_kfast ? e / BK : e % BN] = rb[l];
    }
    __syncthreads();
    // the next tile's loads are in flight while this one is multiplied
    if (t + 1 < ntiles) fetch(t + 1);
    koffs(t + 2);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      cplx<R> a[TM], bb[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + i * (BM / TM)];
#pragma unroll
      for (int j = 0; j < TN; ++j) bb[j] = Bs[kk][tx + j * TX];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) cfma(part[i][j], a[i], bb[j]);
      if ((kk + 1) % RUN == 0) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) {
            acc[i][j] = acc[i][j] + part[i][j];
            part[i][j] = cplx<R>(0, 0);
          }
      }
    }
    __syncthreads();
  }
  const bool use_beta = (beta.re != R(0) || beta.im != R(0));
  if (splits > 1) {
    cplx<R>* Pt = P + ((int64_t)split * g.batch + b) * g.M * g.N;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      int64_t m = m0 + ty + i * (BM / TM);
      if (m >= g.M) continue;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        int64_t n = n0 + tx + j * TX;
        if (n < g.N) Pt[m * g.N + n] = acc[i][j];
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    int64_t m = m0 + ty + i * (BM / TM);
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      int64_t n = n0 + tx + j * TX;
      if (n >= g.N) continue;
      int64_t o = offC + midx_off(g.mC, m) + midx_off(g.nC, n);
      cplx<R> v = alpha * acc[i][j];
      if (use_beta) v = v + beta * C[o];
      C[o] = v;
    }
  }
}

// FP64 kernel: BM x BN outputs per CTA of 256 threads, KG threads per output that
// take KD of every BK = KG KD values of k each.  An SM issues two FP64 FMAs a
// clock, and each of its quarters holds its FP64 unit for 64 cycles per warp
// instruction, so a warp's complex multiply-add takes 256 cycles whatever else
// happens (the shared-memory traffic of one output per thread is hidden
// under it): what counts is that every quarter of every SM has its share of
// the work, and how much of a tile is padding.  Hence tiles from 16 x 16 down to
// 4 x 4, always with eight warps; see f64_tile() for the choice.  The KG partial
// sums are added pairwise in a fixed order.
template <int BM, int BN, int KG, int BK>
__global__ void __launch_bounds__(256)
gemm_f64_kernel(GemmDesc g, zc alpha, zc beta, const zc* __restrict__ A, const zc* __restrict__ B, zc* __restrict__ C,
                int splits, int64_t kchunk, zc* __restrict__ P) {
  constexpr int NT = 256, NO = BM * BN, KD = BK / KG;
  static_assert(NO * KG == NT && KD * KG == BK, "tile shape");
  __shared__ zc As[BK][BM + 1], Bs[BK][BN + 1], red[KG > 1 ? NT / 2 : 1];
  const int64_t b = blockIdx.z / splits;
  const int split = blockIdx.z - (int)(b * splits);
  const int64_t kbeg = (int64_t)split * kchunk, kend = min(g.K, kbeg + kchunk);
  const unsigned ntn = (unsigned)((g.N + BN - 1) / BN), row = blockIdx.x / ntn;
  const int64_t m0 = (int64_t)row * BM, n0 = (int64_t)(blockIdx.x - row * ntn) * BN;
  const int tid = threadIdx.x, o = tid % NO, kg = tid / NO, tn = o % BN, tm = o / BN;
  const int64_t m = m0 + tm, n = n0 + tn;
  const bool in = m < g.M && n < g.N;
  const zc* Ab = A + midx_off(g.bA, b);
  const zc* Bb = B + midx_off(g.bB, b);
  const bool a_kfast = midx_unit_inner(g.kA) && !midx_unit_inner(g.mA);
  const bool b_kfast = midx_unit_inner(g.kB) && !midx_unit_inner(g.nB);
  constexpr int LA = (BM * BK + NT - 1) / NT, LB = (BN * BK + NT - 1) / NT;
  zc ra[LA], rb[LB];
  int64_t oa[LA], ob[LB];  // offsets of the rows and columns this thread loads, -1 beyond the matrix
#pragma unroll
  for (int l = 0; l < LA; ++l) {
    const int e = tid + l * NT, mm = a_kfast ? e / BK : e % BM;
    oa[l] = e < BM * BK && m0 + mm < g.M ? midx_off(g.mA, m0 + mm) : -1;
  }
#pragma unroll
  for (int l = 0; l < LB; ++l) {
    const int e = tid + l * NT, nn = b_kfast ? e / BK : e % BN;
    ob[l] = e < BN * BK && n0 + nn < g.N ? midx_off(g.nB, n0 + nn) : -1;
  }
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = tid + l * NT, kk = a_kfast ? e % BK : e / BM;
      zc v(0, 0);
      if (oa[l] >= 0 && k0 + kk < kend) {
        v = Ab[oa[l] + midx_off(g.kA, k0 + kk)];
        if (g.conjA) v.im = -v.im;
      }
      ra[l] = v;
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = tid + l * NT, kk = b_kfast ? e % BK : e / BN;
      zc v(0, 0);
      if (ob[l] >= 0 && k0 + kk < kend) {
        v = Bb[ob[l] + midx_off(g.kB, k0 + kk)];
        if (g.conjB) v.im = -v.im;
      }
      rb[l] = v;
    }
  };
  zc acc(0, 0);
  if (kbeg < kend) fetch(kbeg);
  for (int64_t k0 = kbeg; k0 < kend; k0 += BK) {
#pragma unroll
    for (int l = 0; l < LA; ++l) {
      const int e = tid + l * NT;
      if (e < BM * BK) As[a_kfast ? e % BK : e / BM][a_kfast ? e / BK : e % BM] = ra[l];
    }
#pragma unroll
    for (int l = 0; l < LB; ++l) {
      const int e = tid + l * NT;
      if (e < BN * BK) Bs[b_kfast ? e % BK : e / BN][b_kfast ? e / BK : e % BN] = rb[l];
    }
    __syncthreads();
    if (k0 + BK < kend) fetch(k0 + BK);
    if (in) {  // (a warp of padding alone costs no FP64 time)
      const int kb = kg * KD, kn = (int)min((int64_t)KD, kend - k0 - kb);
      if (kn == KD) {
#pragma unroll
        for (int kk = 0; kk < KD; ++kk) cfma(acc, As[kb + kk][tm], Bs[kb + kk][tn]);
      } else {
        for (int kk = 0; kk < kn; ++kk) cfma(acc, As[kb + kk][tm], Bs[kb + kk][tn]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int s = KG / 2; s > 0; s /= 2) {
    if (kg >= s && kg < 2 * s) red[(kg - s) * NO + o] = acc;
    __syncthreads();
    if (kg < s) acc = acc + red[kg * NO + o];
    __syncthreads();
  }
  if (kg > 0 || !in) return;
  if (splits > 1) {
    P[(((int64_t)split * g.batch + b) * g.M + m) * g.N + n] = acc;
    return;
  }
  const int64_t oc = midx_off(g.bC, b) + midx_off(g.mC, m) + midx_off(g.nC, n);
  zc v = alpha * acc;
  if (beta.re != 0.0 || beta.im != 0.0) v = v + beta * C[oc];
  C[oc] = v;
}

// C[b][m][n] = alpha sum_s P[s][b][m][n] + beta C[b][m][n], summed in split order
template <class R>
__global__ void splitk_reduce_kernel(GemmDesc g, cplx<R> alpha, cplx<R> beta, const cplx<R>* __restrict__ P,
                                     int splits, cplx<R>* __restrict__ C) {
  const int64_t mn = g.M * g.N, total = g.batch * mn;
  const bool use_beta = (beta.re != R(0) || beta.im != R(0));
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t b = e / mn, r = e - b * mn;
    int64_t m = r / g.N, n = r - m * g.N;
    cplx<R> acc(0, 0);
    for (int s = 0; s < splits; ++s) acc = acc + P[(int64_t)s * total + e];
    int64_t o = midx_off(g.bC, b) + midx_off(g.mC, m) + midx_off(g.nC, n);
    cplx<R> v = alpha * acc;
    if (use_beta) v = v + beta * C[o];
    C[o] = v;
  }
}

}  // namespace

// FP32 tile edge: 64, or 32 for thin shapes and for grids of
// 64 x 64 tiles that would not fill a quarter of the SMs.
static int64_t gemm_tile(const GemmDesc& g) {
  if (g.M <= 32 || g.N <= 32) return 32;
  const int64_t t64 = ((g.M + 63) / 64) * ((g.N + 63) / 64) * g.batch;
  return t64 < 38 ? 32 : 64;
}

// FP64 tile of a contraction: the one with the least time on the busiest SM, in
// cycles: two FP64 FMAs a clock for the tile's 4 K BM BN (a few per cent less in the
// 64-wide ones), and 350 per level of the KG sums for each CTA beyond the three
// that hide one another's start.  us of one tile against another: 128 x 124 x 124
// 16 x 16 41, 8 x 8 23, 4 x 4 27; 512 x 64 x 64 23, 25, 31; 74 x 68 x 74 27, 12, 10; 1024 x
// 1024 x 1024 7220, 7550 (64 x 64, no longer there, 8330); 256 x 4 x 310, batch 144, 16 x 4
// 367, 64 x 4 395, 4 x 4 410; 70000 x 3 x 2 64 x 4 20, 16 x 4 35.  Before this rule (8 x 8 by
// two warps, 16 x 16 or 64 x 64 by the number of outputs) and with it: 144 x 4 x 72
// 20.6 / 8.3, 74 x 68 x 74 22.6 / 12.3, 96 x 48 x 520 70 / 29, 144 x 72 x 1240 287 / 131, 310 x
// 72 x 256, batch 8, 428 / 358 (floor 316).
struct F64Tile {
  int bm, bn, levels;
  double work;
};
static const F64Tile kF64Tiles[] = {{16, 16, 0, 2.0}, {8, 8, 2, 2.0},  {4, 4, 4, 2.0}, {16, 4, 2, 2.0},
                                    {4, 16, 2, 2.0},  {64, 4, 0, 2.1}, {4, 64, 0, 2.1}};

static int64_t f64_tiles(const GemmDesc& g, int bm, int bn) {
  return ((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn) * g.batch;
}

static const F64Tile& f64_tile(const GemmDesc& g) {
  const F64Tile* best = kF64Tiles;
  double cost = 1e300;
  for (const F64Tile& t : kF64Tiles) {
    const double ctas = (double)((f64_tiles(g, t.bm, t.bn) + 151) / 152);  // on the busiest SM
    const double c = ctas * t.work * t.bm * t.bn * g.K + t.levels * (200.0 + 350.0 * std::max(0.0, ctas - 3));
    if (c < cost) {
      cost = c;
      best = &t;
    }
  }
  return *best;
}

// K splits of an FP64 contraction: about one CTA per SM, at least 64 of K each
int qtt_gemm_splits_f64(const GemmDesc& g) {
  const F64Tile& t = f64_tile(g);
  const int64_t tiles = f64_tiles(g, t.bm, t.bn);
  if (tiles >= 76 || g.K < 128) return 1;
  return (int)std::min<int64_t>(32, std::min<int64_t>((g.K + 63) / 64, std::max<int64_t>(1, 152 / tiles)));
}

static int launch_f64(const GemmDesc& g, zc alpha, zc beta, const zc* A, const zc* B, zc* C, int splits,
                      int64_t kchunk, zc* P, cudaStream_t s) {
  const F64Tile& t = f64_tile(g);
  const int64_t edge = gemm_tile(g);
  if ((g.M + edge - 1) / edge > 65535 || g.batch * splits > 65535) return QTT_ERR_ARG;  // the sizes that FP32 takes
  const dim3 grid((unsigned)(f64_tiles(g, t.bm, t.bn) / g.batch), 1, (unsigned)(g.batch * splits));
#define QTT_F64(X, Y, KG, BK)    \
  if (t.bm == X && t.bn == Y) \
    gemm_f64_kernel<X, Y, KG, BK><<<grid, 256, 0, s>>>(g, alpha, beta, A, B, C, splits, kchunk, P)
  QTT_F64(16, 16, 1, 16);
  QTT_F64(8, 8, 4, 32);
  QTT_F64(4, 4, 16, 64);
  QTT_F64(16, 4, 4, 32);
  QTT_F64(4, 16, 4, 32);
  QTT_F64(64, 4, 1, 16);
  QTT_F64(4, 64, 1, 16);
#undef QTT_F64
  return QTT_OK;
}

// Number of K splits worth using for this shape (1 = no split): GEMMs whose
// output tiles cannot occupy half the SMs and whose K is at least 128 get
// their K range cut into chunks of 64 or more, about one CTA per SM.
int qtt_gemm_splits(const GemmDesc& g) {
  const int64_t tile = gemm_tile(g);
  const int64_t tiles = ((g.M + tile - 1) / tile) * ((g.N + tile - 1) / tile) * g.batch;
  if (tiles >= 76 || g.K < 128) return 1;
  int64_t s = std::min<int64_t>((g.K + 63) / 64, std::max<int64_t>(1, 152 / tiles));
  return (int)std::min<int64_t>(s, 32);
}

template <class R>
int qtt_gemm_ex(const GemmDesc& g, cplx<R> alpha, cplx<R> beta, const cplx<R>* A, const cplx<R>* B, cplx<R>* C,
                int splits, cplx<R>* P, cudaStream_t s, int tile) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return QTT_OK;
  if (splits < 1 || (splits > 1 && !P)) return QTT_ERR_ARG;
  const int64_t kchunk = splits > 1 ? (g.K + splits - 1) / splits : std::max<int64_t>(g.K, 1);
  [[maybe_unused]] const bool thin = (tile ? tile : gemm_tile(g)) == 32;  // (FP64 chooses its own tiles)
  constexpr int BK = 16;
  const int64_t zdim = g.batch * splits;
  if (zdim > 65535) return QTT_ERR_ARG;
  if constexpr (sizeof(R) == 8) {
    const int st = launch_f64(g, alpha, beta, A, B, C, splits, kchunk, P, s);
    if (st != QTT_OK) return st;
  } else if (thin) {
    dim3 grid((unsigned)((g.N + 31) / 32), (unsigned)((g.M + 31) / 32), (unsigned)zdim);
    if (grid.y > 65535) return QTT_ERR_ARG;
    gemm_midx_kernel<R, 32, 32, BK, 2, 2><<<grid, 256, 0, s>>>(g, alpha, beta, A, B, C, splits, kchunk, P);
  } else {
    dim3 grid((unsigned)((g.N + 63) / 64), (unsigned)((g.M + 63) / 64), (unsigned)zdim);
    if (grid.y > 65535) return QTT_ERR_ARG;
    gemm_midx_kernel<R, 64, 64, BK, 4, 4><<<grid, 256, 0, s>>>(g, alpha, beta, A, B, C, splits, kchunk, P);
  }
  if (splits > 1) {
    const int64_t total = g.batch * g.M * g.N;
    splitk_reduce_kernel<R><<<(unsigned)std::min<int64_t>((total + 255) / 256, 65535), 256, 0, s>>>(g, alpha, beta, P,
                                                                                                     splits, C);
  }
  return cudaGetLastError() == cudaSuccess ? QTT_OK : QTT_ERR_CUDA;
}

template int qtt_gemm_ex<double>(const GemmDesc&, zc, zc, const zc*, const zc*, zc*, int, zc*, cudaStream_t, int);
template int qtt_gemm_ex<float>(const GemmDesc&, cc, cc, const cc*, const cc*, cc*, int, cc*, cudaStream_t, int);

// the rule's tile edge and the split count the rule would take with a given tile
int qtt_gemm_tile_rule(const GemmDesc& g) { return (int)gemm_tile(g); }
int qtt_gemm_splits_for(const GemmDesc& g, int tile) {
  const int64_t tiles = ((g.M + tile - 1) / tile) * ((g.N + tile - 1) / tile) * g.batch;
  if (tiles >= 76 || g.K < 128) return 1;
  int64_t s = std::min<int64_t>((g.K + 63) / 64, std::max<int64_t>(1, 152 / tiles));
  return (int)std::min<int64_t>(s, 32);
}

template <class R>
int qtt_gemm(const GemmDesc& g, cplx<R> alpha, cplx<R> beta, const cplx<R>* A,
             const cplx<R>* B, cplx<R>* C, cudaStream_t s) {
  return qtt_gemm_ex<R>(g, alpha, beta, A, B, C, 1, nullptr, s, 64);
}

template int qtt_gemm<double>(const GemmDesc&, zc, zc, const zc*, const zc*, zc*, cudaStream_t);
template int qtt_gemm<float>(const GemmDesc&, cc, cc, const cc*, const cc*, cc*, cudaStream_t);
