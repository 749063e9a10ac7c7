// Vector and block kernels of the eigensolver and the CG (internal).
#pragma once
#include "qs_internal.cuh"

#define QS_RED_BLOCKS 608      // most partial sums per vector (4 x 152 SMs)

// v has k vectors of nr reals each ([k][nr]); out[r] = sum over vector r of v^2 (FP64)
template <typename R>
cudaError_t qs_norm2(const R *v, int k, int64_t nr, double *part, double *out, cudaStream_t st);
// out[r] = || a_r - theta[r] b_r ||^2 (FP64 or FP32 vectors, FP64 sum, theta on device)
template <typename R>
cudaError_t qs_resid2(const R *a, const R *b, const double *theta, int k, int64_t nr,
                      double *part, double *out, cudaStream_t st);
// G[i][j] = <A_i, B_j>, i < ka, j < kb, complex row-major [ka][kb] (FP64 vectors);
// lowp: products and per-chunk sums in FP32, chunk sums accumulated in FP64
// A == B: half of the Hermitian G is computed
cudaError_t qs_gram(const double *A, int ka, const double *B, int kb, int64_t nr, double *part,
                    double2 *G, cudaStream_t st, int lowp = 0);
// V_j = sum_i W_i C[i][j], j < kc (C complex row-major [ka][kc]); V must not alias W;
// lowp: the k-term sums in FP32; upper: C[i][j] = 0 for i > j
cudaError_t qs_rotate(const double *W, int ka, const double2 *C, int kc, int64_t nr, double *V,
                      cudaStream_t st, int lowp = 0, int upper = 0);
// the Gram matrix and the rotation on FP32 blocks (FP32 products, FP64 Gram totals)
cudaError_t qs_gram32(const float *A, int ka, const float *B, int kb, int64_t nr, double *part, double2 *G,
                      cudaStream_t st);
cudaError_t qs_rotate32(const float *W, int ka, const double2 *C, int kc, int64_t nr, float *V, cudaStream_t st,
                        int upper = 0);
// y_r = (float)(x_r * scale[r])  (scale on device, may be NULL for 1)
cudaError_t qs_d2f(const double *x, float *y, const double *scale, int k, int64_t nr, cudaStream_t st);
// y_r = (double) x_r
cudaError_t qs_f2d(const float *x, double *y, int k, int64_t nr, cudaStream_t st);
// x_r += coef[r] * (double) e_r  (coef on device)
cudaError_t qs_axpy_f2d(double *x, const float *e, const double *coef, int k, int64_t nr, cudaStream_t st);
// ynew = s1 * (ay - c * y) - s2 * x   (all vectors of the block)
template <typename R>
cudaError_t qs_cheb_step(R *ynew, const R *ay, const R *y, const R *x, double c, double s1, double s2,
                         int64_t n, cudaStream_t st);
// y = a * x + b * y over n reals
template <typename R>
cudaError_t qs_axpby(double a, const R *x, double b, R *y, int64_t n, cudaStream_t st);
// x_r *= scale[r] (device)
template <typename R>
cudaError_t qs_scale_cols(R *x, const double *scale, int k, int64_t nr, cudaStream_t st);
// Gaussian entries from a counter-based hash of (seed, index)
cudaError_t qs_fill_gauss(double *x, int64_t n, uint64_t seed, cudaStream_t st);
// x_r = b_r * coef[r] (coef on device)
cudaError_t qs_scaled_copy(double *x, const double *b, const double *coef, int k, int64_t nr, cudaStream_t st);
// out[r] = 1 / sqrt(in[r]) (0 stays 0), or theta^-2 style maps, on device
cudaError_t qs_map_scalars(const double *in, double *out, int k, int mode, cudaStream_t st);
// C* partner map P v = C T gamma_5 v^* of k FP64 or FP32 vectors (partner.cu); in != out
cudaError_t qs_partner(const double *in, double *out, const Geom &g, int k, int tiled, cudaStream_t st);
cudaError_t qs_partner32(const float *in, float *out, const Geom &g, int k, cudaStream_t st);
// dense kernels (k <= 64), one block per matrix
cudaError_t qs_chol_rinv(const double2 *G, int k, double2 *Rinv, int *info, cudaStream_t st);
// eigenvalues of H0 and eigenpairs H = Y diag(evals) Y^H, both ordered by |eigenvalue|, k even;
// scratch: QS_EIG_SCRATCH(k) doubles, 16-byte aligned (the rotations of at most 40 sweeps)
#define QS_EIG_SCRATCH(k) (64 + (size_t)40 * ((k) - 1) * ((k) / 2) * 4)
cudaError_t qs_herm_eig2(const double2 *H0, double *ev0, int *info0, const double2 *H, double *evals, double2 *Y, int *info,
                         int k, double *scratch, cudaStream_t st);

// CG helpers (FP32 vectors, per-rhs scalars on device)
struct CgScalars {
    double *rr, *rr0;
    float *alpha, *beta;
    int *live, *iters;   // still iterating; iterations done
};
// part: [k][nb] shares of |Q p|^2 (alpha), of |r|^2 (beta)
cudaError_t qs_cg_alpha(const CgScalars &s, int k, const double *part, int nb, cudaStream_t st);
cudaError_t qs_cg_beta_xp(float *x, float *p, const float *r, const CgScalars &s, double tol2, int k, int64_t nr,
                          const double *part, int nb, cudaStream_t st);
cudaError_t qs_cg_init(CgScalars s, const double *rr, int k, cudaStream_t st);

// Ritz values (sorted by |theta|) and residual norms of the current block
// Ritz pairs ordered by <v, Q^2 v> = theta^2 + r^2; col[i] is the device column of
// pair i; theta_dev / res_dev are in device column order.
struct Ritz {
    double theta[64], res[64];
    double theta_dev[64], res_dev[64];
    int col[64];
    double mu_max;   // largest Q^2 Ritz value of the block
};
int qs_lowmodes_impl(qs_lattice *lat, double m0, const qs_eig_opts *o, Ritz *rz, int *conv, qs_eig_stats *stats);
