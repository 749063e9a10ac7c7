// Small dense FP64 kernels (k <= 64), one thread block each: Cholesky factor
// and its inverse for the Cholesky-QR orthogonalisation, and a cyclic Jacobi
// eigensolver for the Rayleigh-Ritz matrix.  Complex matrices are row-major
// double2 [k][k].
#include "blas.cuh"
#include "rank.h"

#include <mutex>

namespace {

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(fma(-a.y, b.y, a.x * b.x), fma(a.y, b.x, a.x * b.y));
}
__device__ __forceinline__ double2 cconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 cscale(double s, double2 a) { return make_double2(s * a.x, s * a.y); }

// G = R^H R with R upper triangular; Rinv = R^-1 (upper).  info = 1 if G is not
// numerically positive definite.  256 threads on one SM, whose FP64 pipe (1.6 lanes a clock) and
// the k dependent steps bound it: the factor is right-looking (each step's rank-1 update is spread
// over all threads), and column j of the inverse is -X R_j / r_jj with 8 threads per row of
// the finished part X.  k = 32: 95 us (312 us with one thread per column and the inverse in
// global memory).
__global__ void __launch_bounds__(256) chol_rinv_kernel(const double2 *G, int k, double2 *Rinv, int *info)
{
    extern __shared__ double2 sm[];
    double2 *R = sm;            // [k][k], upper: the working copy of G, row by row the factor
    double2 *X = sm + k * k;    // [k][k]: the inverse
    __shared__ int bad;
    const int t = threadIdx.x;
    if (t == 0) bad = 0;
    for (int i = t; i < k * k; i += 256) {
        R[i] = i / k <= i % k ? G[i] : make_double2(0, 0);
        X[i] = make_double2(0, 0);
    }
    __syncthreads();
    for (int j = 0; j < k; ++j) {
        double d = R[j * k + j].x;   // the same in every thread
        const bool ok = d > 0 && isfinite(d);
        if (!ok) d = 1.0;
        const double r = sqrt(d), ir = 1.0 / r;
        __syncthreads();
        if (t == 0) {
            if (!ok) bad = 1;
            R[j * k + j] = make_double2(r, 0);
            X[j * k + j] = make_double2(ir, 0);
        }
        for (int l = j + 1 + t; l < k; l += 256) R[j * k + l] = cscale(ir, R[j * k + l]);
        __syncthreads();
        const int n = k - j - 1;
        for (int e = t; e < n * n; e += 256) {
            const int i = j + 1 + e / n, l = j + 1 + e % n;
            if (l < i) continue;
            const double2 a = R[j * k + i], b = R[j * k + l];
            double2 c = R[i * k + l];   // c -= conj(a) b
            c.x = fma(-a.y, b.y, fma(-a.x, b.x, c.x));
            c.y = fma(a.y, b.x, fma(-a.x, b.y, c.y));
            R[i * k + l] = c;
        }
        __syncthreads();
    }
    for (int j = 1; j < k; ++j) {   // X[i][j] = -(sum_{i <= l < j} X[i][l] R[l][j]) / r_jj
        for (int i0 = 0; i0 < j; i0 += 32) {
            const int i = i0 + (t >> 3);
            double2 acc = make_double2(0, 0);
            if (i < j)
                for (int l = i + (t & 7); l < j; l += 8) {
                    const double2 a = X[i * k + l], b = R[l * k + j];
                    acc.x = fma(-a.y, b.y, fma(a.x, b.x, acc.x));
                    acc.y = fma(a.y, b.x, fma(a.x, b.y, acc.y));
                }
            for (int o = 4; o > 0; o >>= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            }
            if (i < j && (t & 7) == 0) X[i * k + j] = cscale(-X[j * k + j].x, acc);
        }
        __syncthreads();
    }
    for (int i = t; i < k * k; i += 256) Rinv[i] = X[i];
    if (t == 0) *info = bad;
}

// Jacobi eigensolver for a Hermitian H: H = Y diag(ev) Y^H; eigenpairs returned in
// order of increasing |ev|.  Parallel ordering (Brent and Luk's round-robin): a sweep
// is k - 1 rounds, each round rotates k / 2 disjoint pivot pairs at once (a tournament
// schedule in which every pair (p, q) meets exactly once per sweep).  Rotation for
// pivot (p, q), h_pq = c u (|u| = 1): with D = diag(1, conj u) the 2x2 block becomes real
// symmetric [[a, c], [c, b]], diagonalised by [[cs, sn], [-sn, cs]], t = sn / cs the
// smaller root of t^2 + 2 tau t - 1 = 0, tau = (b - a) / (2 c).  J = D [[cs, sn], [-sn, cs]].
// Disjoint rotations commute, so a round is one pass over the 2 x 2 blocks (pair i, pair j),
// i <= j, of the upper triangle: J_i^H B J_j, and on the diagonal the two new eigenvalue estimates
// in closed form.  The rotations are logged, and a second kernel applies them to the rows of
// the identity, one warp per row on its own SM, which gives the eigenvectors.  k must be even.
//
// What bounds it: the FP64 pipe of the one SM a matrix lives on, and the chain of square roots and
// divisions of a rotation.  Full-matrix column and row passes and the eigenvectors in the same
// block cost 36 k^2 / 2 lane instructions a round (k = 32: 1.5 ms a matrix); this costs
// 48 (k / 2)^2 / 2 (0.95 ms for both matrices of a Rayleigh-Ritz, which share a launch, and 0.12 ms
// for the vectors).
__device__ __forceinline__ int rr_player(int j, int r, int k)
{
    return j == 0 ? 0 : ((j - 1 + r) % (k - 1)) + 1;
}

#define JAC_SWEEPS 40
struct __align__(16) Rot {
    double cs, sn, ux, uy;
};
struct JacobiJob {
    const double2 *H;
    double *ev;
    int *info;
    Rot *log;       // NULL (eigenvalues only), or [round][k / 2] rotations (cs, sn, u); cs = 0: none
    int *nround;    // rounds logged, then the order of the eigenvalues (k columns)
};

__global__ void __launch_bounds__(256) jacobi_kernel(JacobiJob j0, JacobiJob j1, int k)
{
    extern __shared__ double2 sm[];
    double2 *H = sm;              // [k][k], upper triangle
    __shared__ double s_cs[32], s_sn[32];
    __shared__ double2 s_u[32];
    __shared__ int s_p[32], s_q[32];
    __shared__ double red[2][16];
    const JacobiJob job = blockIdx.x ? j1 : j0;
    const int t = threadIdx.x, nt = blockDim.x, half = k / 2;
    for (int i = t; i < k * k; i += nt) {   // Hermitian up to rounding: the mean of both halves
        const int r = i / k, c = i % k;
        if (r > c) continue;
        const double2 a = job.H[r * k + c], b = job.H[c * k + r];
        H[i] = make_double2(0.5 * (a.x + b.x), r == c ? 0.0 : 0.5 * (a.y - b.y));
    }
    __syncthreads();
    // upper-triangle access: element (r, c) for any order
    auto get = [&](int r, int c) { return r < c ? H[r * k + c] : cconj(H[c * k + r]); };
    auto put = [&](int r, int c, double2 v) {
        if (r < c) H[r * k + c] = v;
        else H[c * k + r] = cconj(v);
    };
    const int nblk = half * (half - 1) / 2;
    int sweep, rounds = 0;
    for (sweep = 0; sweep < JAC_SWEEPS; ++sweep) {
        double o = 0, s = 0;
        for (int i = t; i < k * k; i += nt) {
            const int r = i / k, c = i % k;
            if (r > c) continue;
            const double m2 = H[i].x * H[i].x + H[i].y * H[i].y;
            s += r == c ? m2 : 2 * m2;
            if (r != c) o += 2 * m2;
        }
        for (int d = 16; d > 0; d >>= 1) {
            o += __shfl_xor_sync(0xffffffffu, o, d);
            s += __shfl_xor_sync(0xffffffffu, s, d);
        }
        if ((t & 31) == 0) { red[0][t >> 5] = o; red[1][t >> 5] = s; }
        __syncthreads();
        double off = 0, tot = 0;
        for (int w = 0; w < (nt >> 5); ++w) { off += red[0][w]; tot += red[1][w]; }
        __syncthreads();
        if (off <= 1e-30 * tot || off == 0.0) break;
        if (isnan(off) || isnan(tot)) { sweep = JAC_SWEEPS; break; }   // no sweep can help
        for (int r = 0; r < k - 1; ++r, ++rounds) {
            if (t < half) {
                int p = rr_player(t, r, k), q = rr_player(k - 1 - t, r, k);
                if (p > q) { int x = p; p = q; q = x; }
                s_p[t] = p;
                s_q[t] = q;
                const double2 h = H[p * k + q];
                const double h2 = fma(h.x, h.x, h.y * h.y), ic = rsqrt(h2), c = h2 > 0 ? h2 * ic : 0.0;
                const double a = H[p * k + p].x, b = H[q * k + q].x;
                double cs = 0.0, sn = 0.0;
                double2 u = make_double2(1, 0);
                if (!(c <= 1e-150 || c <= 1e-18 * (fabs(a) + fabs(b)))) {
                    u = make_double2(h.x * ic, h.y * ic);
                    const double tau = 0.5 * (b - a) * ic;
                    const double tt = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(fma(tau, tau, 1.0)));
                    cs = rsqrt(fma(tt, tt, 1.0));
                    sn = tt * cs;
                    H[p * k + p] = make_double2(a - tt * c, 0.0);
                    H[q * k + q] = make_double2(b + tt * c, 0.0);
                    H[p * k + q] = make_double2(0.0, 0.0);
                }
                s_cs[t] = cs;
                s_sn[t] = sn;
                s_u[t] = u;
                if (job.log) job.log[(int64_t)rounds * half + t] = Rot{cs, sn, u.x, u.y};
            }
            __syncthreads();
            for (int e = t; e < nblk; e += nt) {
                // pair numbers i < j of block e (row by row of the strict upper triangle)
                int i = 0, f = e;
                while (f >= half - 1 - i) { f -= half - 1 - i; ++i; }
                const int j = i + 1 + f;
                const int pi = s_p[i], qi = s_q[i], pj = s_p[j], qj = s_q[j];
                double ci = s_cs[i], cj = s_cs[j];
                const double si = s_sn[i], sj = s_sn[j];
                if (ci == 0.0 && cj == 0.0) continue;
                if (ci == 0.0) ci = 1.0;   // no rotation: sn = 0, u = 1
                if (cj == 0.0) cj = 1.0;
                const double2 ui = s_u[i], uj = cconj(s_u[j]);
                double2 b00 = get(pi, pj), b01 = get(pi, qj), b10 = get(qi, pj), b11 = get(qi, qj);
                // right: columns (p, q) of J = [[cs, sn], [-ub sn, ub cs]]
                double2 w = cmul(uj, b01);
                b01 = make_double2(fma(cj, w.x, sj * b00.x), fma(cj, w.y, sj * b00.y));
                b00 = make_double2(fma(-sj, w.x, cj * b00.x), fma(-sj, w.y, cj * b00.y));
                w = cmul(uj, b11);
                b11 = make_double2(fma(cj, w.x, sj * b10.x), fma(cj, w.y, sj * b10.y));
                b10 = make_double2(fma(-sj, w.x, cj * b10.x), fma(-sj, w.y, cj * b10.y));
                // left: rows p' = cs p - u sn q, q' = sn p + u cs q
                w = cmul(ui, b10);
                b10 = make_double2(fma(ci, w.x, si * b00.x), fma(ci, w.y, si * b00.y));
                b00 = make_double2(fma(-si, w.x, ci * b00.x), fma(-si, w.y, ci * b00.y));
                w = cmul(ui, b11);
                b11 = make_double2(fma(ci, w.x, si * b01.x), fma(ci, w.y, si * b01.y));
                b01 = make_double2(fma(-si, w.x, ci * b01.x), fma(-si, w.y, ci * b01.y));
                put(pi, pj, b00);
                put(pi, qj, b01);
                put(qi, pj, b10);
                put(qi, qj, b11);
            }
            __syncthreads();
        }
    }
    for (int i = t; i < k; i += nt) {   // stable order by |ev|; a permutation for any values
        const double e = fabs(H[i * k + i].x);
        int rank = 0;
        for (int j = 0; j < k; ++j) rank += qs_abs_before(fabs(H[j * k + j].x), j, e, i);
        job.ev[rank] = H[i * k + i].x;
        if (job.nround) job.nround[1 + rank] = i;
    }
    if (t == 0) {
        *job.info = sweep >= JAC_SWEEPS ? 1 : 0;
        if (job.nround) job.nround[0] = rounds;
    }
}

// row blockIdx.x of Y = J_1 J_2 ..., columns in the eigenvalues' order; one warp
__global__ void __launch_bounds__(32) jacobi_vectors_kernel(const Rot *__restrict__ log, const int *__restrict__ nround, int k,
                                                            double2 *Y)
{
    __shared__ double2 y[64];
    const int t = threadIdx.x, half = k / 2, n = nround[0];
    for (int i = t; i < k; i += 32) y[i] = make_double2(i == (int)blockIdx.x ? 1.0 : 0.0, 0.0);
    __syncwarp();
    Rot next = t < half && n > 0 ? log[t] : Rot{0, 0, 0, 0};
    for (int m = 0, r = 0; m < n; ++m) {
        const Rot g = next;
        if (t < half && m + 1 < n) next = log[(int64_t)(m + 1) * half + t];
        if (t < half && g.cs != 0.0) {
            int p = rr_player(t, r, k), q = rr_player(k - 1 - t, r, k);
            if (p > q) { int x = p; p = q; q = x; }
            const double2 a = y[p], w = cmul(make_double2(g.ux, -g.uy), y[q]);
            y[p] = make_double2(fma(-g.sn, w.x, g.cs * a.x), fma(-g.sn, w.y, g.cs * a.y));
            y[q] = make_double2(fma(g.cs, w.x, g.sn * a.x), fma(g.cs, w.y, g.sn * a.y));
        }
        __syncwarp();
        if (++r == k - 1) r = 0;
    }
    for (int c = t; c < k; c += 32) Y[blockIdx.x * k + c] = y[nround[1 + c]];
}

}  // namespace

cudaError_t qs_chol_rinv(const double2 *G, int k, double2 *Rinv, int *info, cudaStream_t st)
{
    if (k > 64) return cudaErrorInvalidValue;
    static std::once_flag attr;
    std::call_once(attr, [] {
        cudaFuncSetAttribute(chol_rinv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 64 * 64 * 16);
    });
    chol_rinv_kernel<<<1, 256, 2 * k * k * sizeof(double2), st>>>(G, k, Rinv, info);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_herm_eig2(const double2 *H0, double *ev0, int *info0, const double2 *H, double *evals, double2 *Y, int *info,
                         int k, double *scratch, cudaStream_t st)
{
    if (k > 64 || (k & 1)) return cudaErrorInvalidValue;   // the round-robin ordering pairs all indices
    static std::once_flag attr;
    std::call_once(attr, [] {
        cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 64 * 16);
    });
    JacobiJob a, b;
    a.H = H; a.ev = evals; a.info = info;
    a.nround = (int *)scratch;
    a.log = (Rot *)(scratch + 64);
    b.H = H0; b.ev = ev0; b.info = info0;
    b.nround = nullptr;
    b.log = nullptr;
    jacobi_kernel<<<2, 256, k * k * sizeof(double2), st>>>(a, b, k);
    jacobi_vectors_kernel<<<k, 32, 0, st>>>(a.log, a.nround, k, Y);
    qs_note_launches(2);
    return cudaGetLastError();
}
