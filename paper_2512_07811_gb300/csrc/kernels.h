// Internal kernel launchers (C++ linkage; not part of the C-ABI).
#pragma once

#include "common.cuh"

// raise a kernel's dynamic shared-memory limit to the maximum once per device (linalg.cu)
int qtt_allow_max_smem(const void* func);

template <class R>
int qtt_gemm(const GemmDesc& g, cplx<R> alpha, cplx<R> beta, const cplx<R>* A, const cplx<R>* B,
             cplx<R>* C, cudaStream_t s);

// split-K aware variant: `splits` K ranges, partials in P (splits x batch x M x N), see qtt_gemm_splits
int qtt_gemm_splits(const GemmDesc& g);
int qtt_gemm_splits_f64(const GemmDesc& g);  // the same for FP64 contractions (tile chosen by shape, never tuned)
// tile: 0 = the rule (gemm_tile), else 32 or 64
template <class R>
int qtt_gemm_ex(const GemmDesc& g, cplx<R> alpha, cplx<R> beta, const cplx<R>* A, const cplx<R>* B, cplx<R>* C,
                int splits, cplx<R>* P, cudaStream_t s, int tile = 0);
int qtt_gemm_tile_rule(const GemmDesc& g);
int qtt_gemm_splits_for(const GemmDesc& g, int tile);

template <class R>
int qtt_qr_r(const cplx<R>* in, MIdx inB, MIdx rowI, MIdx colI, int conj_in, int64_t m, int64_t n,
             int64_t rows_total, int64_t rows_per_batch, int64_t batch, cplx<R>* W, cplx<R>* out,
             int64_t out_bstride, int64_t ldr, cudaStream_t s, cplx<R>* tauws = nullptr,
             cplx<R>* Qout = nullptr, int64_t q_bstride = 0, int64_t ldq = 0, cplx<R>* Qws = nullptr,
             bool one_cta = false);

// Householder QR by one cluster per matrix (qr.cu): V (batch * (m + 1) * n elements) receives the reflectors and
// their scalars, out R or (out_rh) R^H, perm (n ints per matrix, or null) the column order by decreasing norm, Qout Q or null.
// QTT_ERR_UNSUPPORTED for shapes it does not take (m > 512, or columns beyond its shared memory).
template <class R>
int qtt_qr_cluster(const cplx<R>* in, MIdx inB, MIdx rowI, MIdx colI, int conj_in, int64_t m, int64_t n,
                   int64_t rows_total, int64_t rows_per_batch, int64_t batch, cplx<R>* V, cplx<R>* out,
                   int64_t out_bstride, int64_t ldr, int out_rh, int* perm, cplx<R>* Qout, int64_t q_bstride,
                   int64_t ldq, cudaStream_t s);

// One-sided Jacobi SVD by one cluster per matrix (jacobi.cu): left singular vectors of G (p x q row-major, matrices
// p*q apart), conjugated, one per row of Vh (q x p) by decreasing singular value, component i of G's rows at perm[i]
// (p per matrix; null: i).  sigma (q, or null); trunc (4 ints per matrix, or null): the rank that the tail threshold
// delta (deltas[b] if not null) and max_rank (0: no cap) keep, 1 if the cap cut it, the discarded tail as a double;
// mask: rows of Vh from that rank on are zeroed.  Where delta is not negative the caller truncates at that tail, and
// trailing columns of rounding noise may be left out: their rows of Vh are zero, and sigma holds their norm as one value
// and zeros.  QTT_ERR_UNSUPPORTED where qtt_svd_fits is false.
template <class R>
bool qtt_svd_fits(int p, int q, int batch);
template <class R>
int qtt_svd(const cplx<R>* G, const int* perm, cplx<R>* Vh, R* sigma, int* trunc, double delta, const double* deltas,
            int max_rank, int mask, int p, int q, int batch, int max_sweeps, int* sweeps, cudaStream_t s);
// Column rotations of an FP64 matrix computed in FP32: V with the columns of G V orthogonal to about 1e-6, V itself
// unitary to FP32 rounding.  Vt (3 batch q^2 elements): V transposed, then two identity matrices per matrix.
bool qtt_svd_pre_fits(int p, int q, int batch);  // where that and the FP64 products are cheaper than the sweeps saved
// (delta, deltas as in qtt_svd)
int qtt_svd_pre(const zc* G, zc* Vt, double delta, const double* deltas, int p, int q, int batch,
                int* sweeps, cudaStream_t s);
// whether qtt_qr_cluster takes the shape with sorted columns
template <class R>
bool qtt_qr_cluster_fits(int64_t m, int64_t n, int64_t batch);

template <class R>
size_t qtt_jacobi_smem_bytes(int p, int q);
template <class R>
int qtt_jacobi_smem(const cplx<R>* G, cplx<R>* Vws, R* sigma, cplx<R>* Vsorted, cplx<R>* Usorted, int p, int q,
                    int max_sweeps, int* sweeps, cudaStream_t s);

template <class R>
int qtt_jacobi(cplx<R>* G, cplx<R>* Vwork, R* sigma, cplx<R>* Vsorted, int p, int q, int batch,
               int max_sweeps, int* sweeps, cudaStream_t s, cplx<R>* Usorted = nullptr);

template <class R>
int qtt_jacobi_wide(const cplx<R>* G, cplx<R>* Gwork, cplx<R>* Vwork, R* sigma, cplx<R>* Vsorted, cplx<R>* Usorted,
                    int p, int q, int max_sweeps, int* dflag, int* sweeps_done, int64_t* launches, cudaStream_t s);

template <class R>
int qtt_trunc_rank(const R* sigma, int q, double delta, int max_rank, int* out, double* tail,
                   cudaStream_t s);

// ---- elementwise / placement kernels (elem.cu)
template <class R>
int qtt_place_block(const cplx<R>* src, int64_t s0, int64_t n, int64_t s1, cplx<R>* dst, int64_t d1,
                    int64_t off0, int64_t off1, cplx<R> scale, cudaStream_t s);
template <class R>
int qtt_hadamard_core(const cplx<R>* x, int64_t a0, int64_t a1, const cplx<R>* y, int64_t b0,
                      int64_t b1, int64_t n, cplx<R>* out, cudaStream_t s);
template <class R>
int qtt_mpo_core(const cplx<R>* D, int64_t g0, int64_t no, int64_t ni, int64_t g1, const cplx<R>* X,
                 int64_t a0, int64_t a1, cplx<R>* out, cudaStream_t s);
template <class R>
int qtt_scale(cplx<R>* x, int64_t count, cplx<R> scale, cudaStream_t s);
template <class R>
int qtt_sumsq(const cplx<R>* x, int64_t count, double* out, cudaStream_t s);
template <class R>
int qtt_copy_strided(const cplx<R>* in, MIdx rows, MIdx cols, int64_t nrows, int64_t ncols, int conj_in,
                     cplx<R>* out, int64_t ldo, cudaStream_t s);
// U += D diag(1 / sv) (row-major, leading dimensions ldu, ldd)
template <class R>
int qtt_add_scaled_cols(cplx<R>* U, int64_t ldu, const cplx<R>* D, int64_t ldd, int64_t rows, int64_t cols, const R* sv,
                        cudaStream_t s);
template <class R>
int qtt_scale_rows(cplx<R>* x, int64_t rows, int64_t cols, int64_t ld, const R* sv, int invert,
                   cudaStream_t s);
template <class R>
int qtt_isfinite(const cplx<R>* x, int64_t count, int* flag, cudaStream_t s);

// ---- one launch over the cores of a train (elem.cu): up to QTT_TABLE cores each
#define QTT_TABLE 48
struct CoreTable {
  int n;
  const void* src[QTT_TABLE];
  void* dst[QTT_TABLE];
  int64_t cnt[QTT_TABLE];
};
// what: 0 copy (elem bytes each, 8 or 16), 1 complex128 -> complex64, 2 complex64 -> complex128
int qtt_cores_move(const CoreTable& t, int what, int elem, cudaStream_t s);
// Products of a train's first cores (p x r row-major to P) and of its last ones (r x q to S), each partial product at
// most QTT_ENDS / sizeof(R) elements: one CTA each
#define QTT_ENDS 4096
struct EndsTable {
  int n[2];                 // cores of either end, at most 16
  const void* core[2][16];  // in train order
  int r0[2][16], m[2][16], r1[2][16];
};
template <class R>
int qtt_train_ends(const EndsTable& t, cplx<R>* P, cplx<R>* S, cudaStream_t s);
// *flag = 1 if an element of the src cores is not finite
template <class R>
int qtt_cores_isfinite(const CoreTable& t, int* flag, cudaStream_t s);
// sketch cores: the M x M identity where M > 0, else real Gaussian N(0, scale^2) from (seed, stream + core)
struct SketchTable {
  int n;
  void* dst[QTT_TABLE];
  int64_t cnt[QTT_TABLE], M[QTT_TABLE];
  double scale[QTT_TABLE];
  uint64_t seed, stream;
};
template <class R>
int qtt_fill_sketch(const SketchTable& t, cudaStream_t s);
// cores of a x + b y: blocks [x | y] on the bonds, zero elsewhere; xa, xb, ya, yb the bond sizes, first / last: the
// train's end cores (bond 0 not stacked; scale on the first)
template <class R>
struct AddTable {
  int n;
  const cplx<R>* x[QTT_TABLE];
  const cplx<R>* y[QTT_TABLE];
  cplx<R>* z[QTT_TABLE];
  int xa[QTT_TABLE], xb[QTT_TABLE], ya[QTT_TABLE], yb[QTT_TABLE], nk[QTT_TABLE];
  int first, last;  // index of the first / last core in this table, or -1
  cplx<R> a, b;
  int ua, ub;  // a / b is exactly 1: the block is copied
};
template <class R>
int qtt_add_cores(const AddTable<R>& t, int64_t max_count, cudaStream_t s);

// ---- operator construction on the device (elem.cu)
template <class R>
int qtt_fill_qft_dense(cplx<R>* out, int n, double sign, cudaStream_t s);
template <class R>
int qtt_fill_green_dense(cplx<R>* out, const SiteMap& m, int ncomp, double k0, double lam0, double mu0,
                         cudaStream_t s);
template <class R>
int qtt_fill_indicator_sites(const double* ind, const SiteMap& m, cplx<R>* out, cudaStream_t s);
template <class R>
int qtt_fill_gaussian(cplx<R>* out, int64_t count, uint64_t seed, uint64_t stream, double scale, cudaStream_t s);
template <class R>
int qtt_diag_mpo_core(const cplx<R>* X, int64_t r0, int64_t n, int64_t r1, cplx<R>* D, cudaStream_t s);
template <class R>
int qtt_identity_core(int64_t g, int64_t n, cplx<R>* D, cudaStream_t s);
template <class R>
int qtt_adjoint_core(const cplx<R>* D, int64_t g0, int64_t no, int64_t ni, int64_t g1, cplx<R>* out,
                     cudaStream_t s);

// tensor-core complex64 GEMM (tc_gemm.cu), batch 1
size_t qtt_tc_gemm_workspace(int64_t M, int64_t N, int64_t K);
size_t qtt_tc_gemm_workspace_ex(int64_t M, int64_t N, int64_t K, int64_t batch, int passes);
int qtt_tc_gemm_ex(const GemmDesc& g, cc alpha, cc beta, const cc* A, const cc* B, cc* C, void* ws, int* err,
                   cudaStream_t s, int passes);
int qtt_tc_gemm(const GemmDesc& g, cc alpha, cc beta, const cc* A, const cc* B, cc* C, void* ws, int* err,
                cudaStream_t s);

// one-sided Jacobi over a thread-block cluster of nc CTAs (4 or 8), rows split over the CTAs (linalg.cu)
template <class R>
size_t qtt_jacobi_cluster_bytes(int p, int q, int nc);
template <class R>
int qtt_jacobi_cluster(const cplx<R>* G, R* sigma, cplx<R>* Vsorted, cplx<R>* Usorted, int p, int q, int nc,
                       int max_sweeps, int* sweeps, cudaStream_t s);

// block-cyclic one-sided Jacobi over a cluster (columns split into blocks, linalg.cu); no rotations output
template <class R>
int qtt_jacobi_block_plan(int p, int q, int* bs_out);
// batch: that many p x q matrices back to back (sigma q apart, Usorted p*q apart), one cluster each
template <class R>
int qtt_jacobi_block(const cplx<R>* G, R* sigma, cplx<R>* Usorted, int p, int q, int max_sweeps, int* sweeps,
                     cudaStream_t s, int batch = 1);
// truncation rule for a batch of sorted singular-value vectors (q apart), delta per vector;
// out[4b] = t, out[4b+1] = capped, out[4b+2..3] = discarded tail (double)
template <class R>
int qtt_trunc_rank_batch(const R* sigma, int q, const double* delta, int max_rank, int* out, int batch,
                         cudaStream_t s);
// ---- batched copies (elem.cu)
// out[b*ob + i*ldo + j] = op(in[b*ib + rows(i) + cols(j)]), op = conj if conj_in
template <class R>
int qtt_copy_batch(const cplx<R>* in, int64_t ib, MIdx rows, MIdx cols, int64_t nrows, int64_t ncols, int conj_in,
                   cplx<R>* out, int64_t ldo, int64_t ob, int batch, cudaStream_t s);
// zero columns j >= t[b * tstride] of each rows x cols matrix (leading dimension ld, matrices bs apart)
template <class R>
int qtt_mask_cols_batch(cplx<R>* X, int64_t bs, int64_t rows, int64_t cols, int64_t ld, const int* t, int tstride,
                        int batch, cudaStream_t s);
// dst[b] (t0[b] x n x t1[b]) = src[b][:t0[b], :, :t1[b]] of the padded r0 x n x r1 cores (src cores sb apart)
template <class R>
int qtt_crop_batch(const cplx<R>* src, int64_t sb, int64_t r0, int64_t n, int64_t r1, cplx<R>* const* dst,
                   const int* t0, const int* t1, int batch, cudaStream_t s);
// polar compression helpers (elem.cu): out = (H + H^H)/2 - shift I; S <- (I + S)/2 with Re tr into *tr
template <class R>
int qtt_herm_shift(const cplx<R>* H, int64_t q, double shift, cplx<R>* out, cudaStream_t s);
template <class R>
int qtt_half_identity_plus(cplx<R>* S, int64_t q, double* tr, cudaStream_t s);

// TT-cross (cross.cu): superblock sampler, maximum-volume rows, index sets
template <class R>
int qtt_cross_eval(const CrossFn& f, int d, int k, const uint8_t* Il, int rl, const uint8_t* Jr, int rr, int n0,
                   int n1, int herm, cplx<R>* out, cudaStream_t s);
template <class R>
size_t qtt_maxvol_smem(int m, int r);
template <class R>
int qtt_maxvol(cplx<R>* A, int m, int r, int* piv, double tol, int max_iters, int* status, cudaStream_t s);
int qtt_cross_left_index(const uint8_t* Iprev, int k, int n0, const int* piv, int t, uint8_t* Inew, cudaStream_t s);
int qtt_cross_right_index(const uint8_t* Jnext, int nr, int rr, const int* piv, int t, uint8_t* Jnew, cudaStream_t s);
template <class R>
int qtt_cross_gather(const cplx<R>* S, int64_t ld, const int* piv, int t, int64_t len, int trans, cplx<R>* out,
                     cudaStream_t s);

// full tensor in site order (control first) -> voxel field (elem.cu)
template <class R>
int qtt_sites_to_voxels(const cplx<R>* in, const SiteMap& m, int ncomp, cplx<R>* out, cudaStream_t s);
