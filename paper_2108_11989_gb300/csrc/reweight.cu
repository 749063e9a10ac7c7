// Mass reweighting and the even-odd preconditioned solve (Sec. 4).
//
// qs_ratapprox: the (n, n) rational function R(y) = A prod_i (y + nu_i^2) / (y + mu_i^2) of
// least uniform relative error |R(y) y^(1/4) - 1| on y in [r_a^2, r_b^2] (eq. ratapprox; R
// stands for (Q_hat^2)^(-1/4) in eq. detQ2).  Host code: a Remez exchange in which the
// 2n + 2 equioscillation equations at the reference points are solved by damped Newton in
// the logarithms of A, nu_i^2 and mu_i^2 (all positive), then the reference moves to the
// extrema of the error (located on a grid, refined by golden-section search).  The first
// guess is a staircase: n factors with equal log-steps spread over the interval and a margin
// on both sides, each lowering log R by 1/4 of its share of log y.
//
// qs_w_mass: the stochastic estimate of W_mass = det[R(Q_hat_m^2) R^-1(Q_hat_m'^2)]
// (eq. Wmass): for every j and source eta, q = (eta, R_j eta), R_j = X^+ + X + X^+ X,
// X = delta D S_j, delta D = D_hat(m') - D_hat(m), with
//   S_j = b^-1 i gamma_5 (mu_j - nu_j) a^-1,  a = D_hat(m) + i gamma_5 nu_j,
//                                              b = D_hat(m') + i gamma_5 mu_j,
// which is the printed three-term S_j after b^-1 (b - a - delta D) a^-1 is multiplied out.
// a^-1 v = (Q_hat_m - i nu)(Q_hat_m^2 + nu^2)^-1 gamma_5 v (gamma_5 a = Q_hat_m + i nu), the
// inverse by FP64 conjugate gradients on the positive operator Q_hat^2 + nu^2.  The estimate
// is prod_j (1/N) sum_l exp(-q_jl) (E[exp(-(eta, R_j eta))] = 1/det(1 + R_j) for sources of
// density ~ exp(-(eta, eta))).
//
// qs_solve_D: x = D^-1 b through the Schur complement on the even sites, with the same FP64
// CG (on Q_hat^2) and the odd-site inverses; or, for comparison, CG on the full-lattice Q^2.
#include "evenodd.cuh"

#include <math.h>

#include <algorithm>
#include <vector>

namespace {

// ---- rational approximation (host) -------------------------------------------------------

const double kP = 0.25;   // R approximates y^-p

inline double log_add_exp(double a, double b)
{
    const double mx = a > b ? a : b;
    return mx + log1p(exp(-fabs(a - b)));
}

// log(R(y) y^p) at S = log y; u = (log A, log nu_i^2 (n), log mu_i^2 (n))
double log_ratio(const double *u, int n, double S)
{
    double g = u[0] + kP * S;
    for (int i = 0; i < n; ++i) g += log_add_exp(S, u[1 + i]) - log_add_exp(S, u[1 + n + i]);
    return g;
}

inline double rel_err(const double *u, int n, double S) { return expm1(log_ratio(u, n, S)); }

// solve M x = b (m x m, row-major) by Gaussian elimination with partial pivoting; b <- x
bool dense_solve(std::vector<double> &M, std::vector<double> &b, int m)
{
    for (int c = 0; c < m; ++c) {
        int piv = c;
        for (int r = c + 1; r < m; ++r)
            if (fabs(M[r * m + c]) > fabs(M[piv * m + c])) piv = r;
        if (!(fabs(M[piv * m + c]) > 0)) return false;
        if (piv != c) {
            for (int j = 0; j < m; ++j) std::swap(M[c * m + j], M[piv * m + j]);
            std::swap(b[c], b[piv]);
        }
        for (int r = c + 1; r < m; ++r) {
            const double f = M[r * m + c] / M[c * m + c];
            if (f == 0) continue;
            for (int j = c; j < m; ++j) M[r * m + j] -= f * M[c * m + j];
            b[r] -= f * b[c];
        }
    }
    for (int r = m - 1; r >= 0; --r) {
        double s = b[r];
        for (int j = r + 1; j < m; ++j) s -= M[r * m + j] * b[j];
        b[r] = s / M[r * m + r];
    }
    return true;
}

// residuals of the levelled equations g(S_k) = log(1 + sg_k delta); u[2n+1] = delta
double level_residual(const std::vector<double> &u, int n, const std::vector<double> &S,
                      const std::vector<double> &sg, std::vector<double> *F)
{
    const int m = 2 * n + 2;
    const double d = u[2 * n + 1];
    double nrm = 0;
    for (int k = 0; k < m; ++k) {
        const double a = 1 + sg[k] * d;
        const double f = a > 0 ? log_ratio(u.data(), n, S[k]) - log(a) : INFINITY;
        if (F) (*F)[k] = f;
        nrm += f * f;
    }
    return sqrt(nrm);
}

// damped Newton on the levelled equations at a fixed reference
void newton_level(std::vector<double> &u, int n, const std::vector<double> &S, const std::vector<double> &sg)
{
    const int m = 2 * n + 2;
    std::vector<double> F(m), J(m * m), du(m), un(m);
    for (int it = 0; it < 60; ++it) {
        const double nF = level_residual(u, n, S, sg, &F);
        if (!(nF > 1e-15)) return;
        const double d = u[2 * n + 1];
        for (int k = 0; k < m; ++k) {
            double *row = &J[k * m];
            row[0] = 1;
            for (int i = 0; i < n; ++i) {
                row[1 + i] = exp(u[1 + i] - log_add_exp(S[k], u[1 + i]));
                row[1 + n + i] = -exp(u[1 + n + i] - log_add_exp(S[k], u[1 + n + i]));
            }
            row[2 * n + 1] = -sg[k] / (1 + sg[k] * d);
            du[k] = -F[k];
        }
        if (!dense_solve(J, du, m)) return;
        double lam = 1;
        bool ok = false;
        while (lam > 1e-6) {
            for (int k = 0; k < m; ++k) un[k] = u[k] + lam * du[k];
            if (fabs(un[2 * n + 1]) < 0.9) {
                const double nn = level_residual(un, n, S, sg, nullptr);
                if (std::isfinite(nn) && nn < (1 - 1e-4 * lam) * nF) { ok = true; break; }
            }
            lam *= 0.5;
        }
        if (!ok) return;
        u = un;
    }
}

// refine an extremum of |e| inside [a, b] by golden-section search
double refine_extremum(const std::vector<double> &u, int n, double a, double b)
{
    const double gr = 0.5 * (sqrt(5.0) - 1);
    double c = b - gr * (b - a), d = a + gr * (b - a);
    double fc = fabs(rel_err(u.data(), n, c)), fd = fabs(rel_err(u.data(), n, d));
    for (int it = 0; it < 60 && b - a > 1e-12 * (1 + fabs(a)); ++it) {
        if (fc > fd) { b = d; d = c; fd = fc; c = b - gr * (b - a); fc = fabs(rel_err(u.data(), n, c)); }
        else { a = c; c = d; fc = fd; d = a + gr * (b - a); fd = fabs(rel_err(u.data(), n, d)); }
    }
    return 0.5 * (a + b);
}

// the alternating extrema of the error on the grid (largest |e| of each run of one sign),
// trimmed to m by dropping the weaker end; refined off the grid.  Returns how many were found.
int find_extrema(const std::vector<double> &u, int n, const std::vector<double> &grid, int m,
                 std::vector<double> *S, std::vector<double> *sg, double *emax)
{
    const int ng = (int)grid.size();
    std::vector<double> e(ng);
    *emax = 0;
    for (int i = 0; i < ng; ++i) {
        e[i] = rel_err(u.data(), n, grid[i]);
        *emax = std::max(*emax, fabs(e[i]));
    }
    std::vector<int> ext;
    int start = 0;
    for (int i = 1; i <= ng; ++i)
        if (i == ng || (e[i] >= 0) != (e[start] >= 0)) {
            int best = start;
            for (int j = start; j < i; ++j)
                if (fabs(e[j]) > fabs(e[best])) best = j;
            ext.push_back(best);
            start = i;
        }
    while ((int)ext.size() > m) {
        if (fabs(e[ext.front()]) < fabs(e[ext.back()])) ext.erase(ext.begin());
        else ext.pop_back();
    }
    const int ne = (int)ext.size();
    if (ne < m) return ne;
    S->assign(m, 0);
    sg->assign(m, 0);
    for (int k = 0; k < m; ++k) {
        const int i = ext[k];
        double x = grid[i];
        if (i > 0 && i < ng - 1) x = refine_extremum(u, n, grid[i - 1], grid[i + 1]);
        const double ex = rel_err(u.data(), n, x);
        (*S)[k] = x;
        (*sg)[k] = ex >= 0 ? 1.0 : -1.0;
        *emax = std::max(*emax, fabs(ex));
    }
    return m;
}

}  // namespace

extern "C" int qs_ratapprox(int n, double ra, double rb, double *A, double *nu, double *mu, double *delta)
{
    if (n < 0 || n > 32 || !(ra > 0) || !(rb > ra) || !A || !delta || (n > 0 && (!nu || !mu)))
        return QS_EINVAL;
    const double la = 2 * log(ra), lb = 2 * log(rb), L = lb - la;
    if (n == 0) {   // best constant: A y^p - 1 = -delta at y_a, +delta at y_b
        const double a = exp(kP * la), b = exp(kP * lb);
        *A = 2 / (a + b);
        *delta = (b - a) / (b + a);
        return QS_OK;
    }
    const int m = 2 * n + 2;
    std::vector<double> u(m, 0.0);
    const double margin = 2.5;
    const double w = kP * (L + 2 * margin) / n;
    for (int i = 0; i < n; ++i) {
        const double c = la - margin + (L + 2 * margin) * (i + 0.5) / n;
        u[1 + i] = c + 0.5 * w;
        u[1 + n + i] = c - 0.5 * w;
    }
    const int ng = 4000 + 2000 * n;
    std::vector<double> grid(ng);
    for (int i = 0; i < ng; ++i) grid[i] = la + L * i / (ng - 1);
    {   // centre the error of the staircase
        double gmin = INFINITY, gmax = -INFINITY;
        for (int i = 0; i < ng; i += 7) {
            const double g = log_ratio(u.data(), n, grid[i]);
            gmin = std::min(gmin, g);
            gmax = std::max(gmax, g);
        }
        u[0] = -0.5 * (gmin + gmax);
    }
    std::vector<double> S, sg;
    double emax = 0;
    if (find_extrema(u, n, grid, m, &S, &sg, &emax) < m) {
        S.resize(m);
        sg.resize(m);
        for (int k = 0; k < m; ++k) {
            S[k] = 0.5 * (la + lb) - 0.5 * L * cos(M_PI * k / (m - 1));
            sg[k] = (k % 2) ? -1.0 : 1.0;
        }
    }
    bool done = false;
    for (int outer = 0; outer < 100 && !done; ++outer) {
        const std::vector<double> u0 = u;
        u[2 * n + 1] = 0;
        newton_level(u, n, S, sg);
        std::vector<double> S2, sg2;
        // a Newton solution that loses the alternation went too far: move only part of the way
        int found = find_extrema(u, n, grid, m, &S2, &sg2, &emax);
        const std::vector<double> u1 = u;
        for (int h = 1; h <= 12 && found < m; ++h) {
            const double f = ldexp(1.0, -h);
            for (int k = 0; k < m; ++k) u[k] = u0[k] + f * (u1[k] - u0[k]);
            found = find_extrema(u, n, grid, m, &S2, &sg2, &emax);
        }
        if (found < m) return QS_ENOCONV;
        double emin = INFINITY;
        for (int k = 0; k < m; ++k) emin = std::min(emin, fabs(rel_err(u.data(), n, S2[k])));
        S = S2;
        sg = sg2;
        done = emax - emin <= std::max(1e-9 * emax, 2e-13);   // the rounding floor of log_ratio
    }
    if (!done) return QS_ENOCONV;
    *A = exp(u[0]);
    std::vector<double> a(u.begin() + 1, u.begin() + 1 + n), b(u.begin() + 1 + n, u.begin() + 1 + 2 * n);
    std::sort(a.begin(), a.end());
    std::sort(b.begin(), b.end());
    for (int i = 0; i < n; ++i) {
        nu[i] = exp(0.5 * a[i]);
        mu[i] = exp(0.5 * b[i]);
    }
    *delta = emax;
    return QS_OK;
}

// ---- W_mass (GPU) -------------------------------------------------------------------------
namespace {

#define RW_PARTS 304   // blocks per right-hand side in the reductions (2 x 152 SMs)
#define RW_LAG 2       // iterations the host may be ahead of the convergence flags it has seen

// y += c x over n doubles
__global__ void rw_axpy(double *__restrict__ y, const double *__restrict__ x, double c, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] += c * x[i];
}

// out = in + c i x (complex, c real); in may equal out
__global__ void rw_add_ix(double2 *out, const double2 *in, const double2 *__restrict__ x, double c, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 a = in[i], b = x[i];
        out[i] = make_double2(a.x - c * b.y, a.y + c * b.x);
    }
}

// component of element i of a vector: [site][12], or [site / 16][12][site % 16]
__device__ __forceinline__ int rw_comp(int64_t i, int tiled) { return (int)((tiled ? i >> 4 : i) % 12); }

// out = c i gamma_5 x (c real; chiral basis: spins 2, 3 negated); out may equal x
__global__ void rw_ig5(double2 *out, const double2 *x, double c, int64_t n, int tiled)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double s = rw_comp(i, tiled) >= 6 ? -c : c;
        const double2 b = x[i];
        out[i] = make_double2(-s * b.y, s * b.x);
    }
}

// out = gamma_5 x; out may equal x
__global__ void rw_g5(double2 *out, const double2 *x, int64_t n, int tiled)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 b = x[i];
        out[i] = rw_comp(i, tiled) >= 6 ? make_double2(-b.x, -b.y) : b;
    }
}

// sum over the block (256 threads), fixed order; valid in thread 0
__device__ double rw_block_sum(double v)
{
    __shared__ double sh[8];
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    v = threadIdx.x < 8 ? sh[threadIdx.x] : 0.0;
    for (int d = 4; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}

// part[r][blk] = the block's share of Re (x_r, y_r)
__global__ void __launch_bounds__(256) rw_dot_part(const double2 *__restrict__ x, const double2 *__restrict__ y, int64_t n,
                                                   double *__restrict__ part)
{
    const int r = blockIdx.y;
    double re = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 a = x[r * n + i], b = y[r * n + i];
        re = fma(a.y, b.y, fma(a.x, b.x, re));
    }
    re = rw_block_sum(re);
    if (threadIdx.x == 0) part[r * gridDim.x + blockIdx.x] = re;
}

__device__ double rw_sum_parts(const double *part, int nparts)
{
    double s = 0;
    for (int i = threadIdx.x; i < nparts; i += 256) s += part[i];
    return rw_block_sum(s);
}

__global__ void __launch_bounds__(256) rw_dot_sum(const double *__restrict__ part, int nparts, double *__restrict__ out)
{
    const double s = rw_sum_parts(part + (int64_t)blockIdx.x * nparts, nparts);
    if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// ---- conjugate gradients with the scalars on the device --------------------------------------
// Per right-hand side: |r|^2, its stopping value and whether it still iterates (live), in two
// slots: an iteration reads slot `o` and writes slot 1 - o.  Every block sums the partial sums
// it needs itself (a few hundred words from L2, in a fixed order), so an iteration is the
// operator's launches and two more; with separate launches for the scalars the launch gaps
// were a tenth of an iteration on 8^3 x 16.  A right-hand side that has converged is skipped by
// every kernel that follows.
struct RwScal {
    double *rr[2], *stop;
    int *live[2];
};

// x = 0, r = p = b, part = shares of |b|^2
__global__ void __launch_bounds__(256) rw_cg_start(const double2 *__restrict__ b, double2 *__restrict__ x,
                                                   double2 *__restrict__ r, double2 *__restrict__ p, int64_t n, double *part)
{
    const int64_t o = blockIdx.y * n;
    double acc = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 v = b[o + i];
        x[o + i] = make_double2(0.0, 0.0);
        r[o + i] = v;
        p[o + i] = v;
        acc = fma(v.y, v.y, fma(v.x, v.x, acc));
    }
    acc = rw_block_sum(acc);
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = acc;
}

__global__ void __launch_bounds__(256) rw_cg_first(RwScal s, const double *part, int nparts, double tol2)
{
    const int r = blockIdx.x;
    const double d = rw_sum_parts(part + (int64_t)r * nparts, nparts);
    if (threadIdx.x != 0) return;
    s.rr[0][r] = d;
    s.stop[r] = tol2 * d;
    s.live[0][r] = d > 0;
}

// the sum of the partials, known to every thread of the block
__device__ double rw_all_parts(const double *part, int nparts)
{
    __shared__ double d;
    const double v = rw_sum_parts(part, nparts);
    if (threadIdx.x == 0) d = v;
    __syncthreads();
    return d;
}

// r -= alpha A p, alpha = |r|^2 / (p, A p); rpart = shares of |r|^2
__global__ void __launch_bounds__(256) rw_cg_r(double2 *__restrict__ r, const double2 *__restrict__ ap, RwScal s, int o,
                                               int64_t n, const double *__restrict__ ppart, int nparts,
                                               double *__restrict__ rpart)
{
    const int k = blockIdx.y;
    if (!s.live[o][k]) return;
    const double pap = rw_all_parts(ppart + (int64_t)k * nparts, nparts);
    const double c = pap > 0 ? -s.rr[o][k] / pap : 0.0;
    double2 *rk = r + k * n;
    const double2 *ak = ap + k * n;
    double acc = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 a = ak[i];
        double2 v = rk[i];
        v = make_double2(fma(c, a.x, v.x), fma(c, a.y, v.y));
        rk[i] = v;
        acc = fma(v.y, v.y, fma(v.x, v.x, acc));
    }
    acc = rw_block_sum(acc);
    if (threadIdx.x == 0) rpart[k * gridDim.x + blockIdx.x] = acc;
}

// x += alpha p, p = r + beta p, beta = |r|^2 / |r_old|^2; the right-hand side lives on unless |r|^2
// has reached its stopping value
__global__ void __launch_bounds__(256) rw_cg_xp(double2 *__restrict__ x, double2 *__restrict__ p,
                                                const double2 *__restrict__ r, RwScal s, int o, int64_t n,
                                                const double *__restrict__ ppart, int nparts,
                                                const double *__restrict__ rpart)
{
    const int k = blockIdx.y;
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    if (!s.live[o][k]) {
        if (first) s.live[1 - o][k] = 0;
        return;
    }
    const double rr = s.rr[o][k];
    const double pap = rw_all_parts(ppart + (int64_t)k * nparts, nparts);
    __syncthreads();
    const double rn = rw_all_parts(rpart + (int64_t)k * gridDim.x, (int)gridDim.x);
    const double a = pap > 0 ? rr / pap : 0.0, b = rr > 0 ? rn / rr : 0.0;
    if (first) {
        s.rr[1 - o][k] = rn;
        s.live[1 - o][k] = !(rn <= s.stop[k]);
    }
    double2 *xk = x + k * n, *pk = p + k * n;
    const double2 *rk = r + k * n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 q = pk[i], v = rk[i];
        double2 y = xk[i];
        y = make_double2(fma(a, q.x, y.x), fma(a, q.y, y.y));
        xk[i] = y;
        pk[i] = make_double2(fma(b, q.x, v.x), fma(b, q.y, v.y));
    }
}

struct RwWork {
    qs_lattice *lat;
    int nrhs;
    int64_t len;          // doubles per vector
    double *eta, *t, *x, *r, *p, *ap, *tmp, *dwork;
    double *part, *rpart, *dots;
    RwScal sc;
    int *hflag;           // pinned, RW_LAG + 1 copies of the live flags
    double *hnorm;        // pinned, |b|^2 of the last rw_cg
    bool nan_rhs;         // a right-hand side of a rw_cg was not a number (it was not iterated)
    cudaEvent_t ev[RW_LAG + 1];
    int full;             // 1: Q^2 of the full-lattice operator instead of Q_hat^2
    // odd-site block inverses at the two masses of the estimate
    double mass[2];
    const double2 *inv[2];
    const double2 *inv_for(double m) const { return m == mass[0] ? inv[0] : inv[1]; }
};

int64_t rw_parts(const Geom &g) { return std::max<int64_t>(RW_PARTS, qs_hat_tiles(g)); }
// doubles of scalar and reduction storage
int64_t rw_small(const Geom &g, int nrhs) { return nrhs * (rw_parts(g) + RW_PARTS + 8); }

// lays out the small arrays at `buf` (rw_small doubles) and makes the pinned flags and events
int rw_begin(RwWork &w, double *buf)
{
    w.part = buf;
    w.rpart = buf + w.nrhs * rw_parts(w.lat->g);
    double *d = w.rpart + w.nrhs * RW_PARTS;
    w.dots = d;
    w.sc.stop = d + w.nrhs;
    for (int o = 0; o < 2; ++o) {
        w.sc.rr[o] = d + (2 + o) * w.nrhs;
        w.sc.live[o] = (int *)(d + (4 + o) * w.nrhs);
    }
    w.hflag = nullptr;
    w.nan_rhs = false;
    for (auto &e : w.ev) e = nullptr;
    QS_CUDA(cudaMallocHost(&w.hflag, (RW_LAG + 1) * 64 * sizeof(int) + 64 * sizeof(double)));
    w.hnorm = (double *)(w.hflag + (RW_LAG + 1) * 64);
    for (auto &e : w.ev) QS_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    return QS_OK;
}

void rw_end(RwWork &w)
{
    cudaStreamSynchronize(w.lat->stream);   // no flag copy may be in flight when its buffer goes
    for (auto e : w.ev)
        if (e) cudaEventDestroy(e);
    if (w.hflag) cudaFreeHost(w.hflag);
}

int rw_check(const char *where)
{
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { qs_record_cuda_error(e, where); return QS_ECUDA; }
    return QS_OK;
}

unsigned rw_blocks(int64_t n) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 511) / 512, RW_PARTS)); }

// out[r] = Re (x_r, y_r) on the host
int rw_dot(RwWork &w, const double *x, const double *y, double *out)
{
    cudaStream_t st = w.lat->stream;
    const unsigned nb = rw_blocks(w.len / 2);
    rw_dot_part<<<dim3(nb, w.nrhs), 256, 0, st>>>((const double2 *)x, (const double2 *)y, w.len / 2, w.part);
    rw_dot_sum<<<w.nrhs, 256, 0, st>>>(w.part, (int)nb, w.dots);
    qs_note_launches(2);
    QS_TRY(rw_check("rw_dot"));
    QS_CUDA(cudaMemcpyAsync(out, w.dots, w.nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
    QS_CUDA(cudaStreamSynchronize(st));
    return QS_OK;
}

unsigned rw_grid(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 4 * 152); }

// ap = (Q_hat(m)^2 + sigma) p for the live right-hand sides, and the shares of (p, ap) in
// w.part; *nparts of them per right-hand side
int rw_q2(RwWork &w, double m, double sigma, const int *live, int *nparts)
{
    if (w.full) {
        double mm[64];
        for (int r = 0; r < w.nrhs; ++r) mm[r] = m;
        QS_TRY(qs_dslash_run(w.lat, QS_F64, mm, w.p, w.tmp, w.nrhs, 1, 0));
        QS_TRY(qs_dslash_run(w.lat, QS_F64, mm, w.tmp, w.ap, w.nrhs, 1, 0));
        if (sigma != 0.0) {
            const int64_t n = w.nrhs * w.len;
            rw_axpy<<<rw_grid(n), 256, 0, w.lat->stream>>>(w.ap, w.p, sigma, n);
            qs_note_launches(1);
        }
        *nparts = (int)rw_blocks(w.len / 2);
        rw_dot_part<<<dim3(*nparts, w.nrhs), 256, 0, w.lat->stream>>>((const double2 *)w.p, (const double2 *)w.ap, w.len / 2,
                                                                     w.part);
        qs_note_launches(1);
        return rw_check("rw_q2");
    }
    const double2 *inv = w.inv_for(m);
    QS_TRY(qs_dhat_run(w.lat, m, w.p, w.tmp, w.nrhs, 1, w.dwork, inv, live));
    *nparts = (int)qs_hat_tiles(w.lat->g);
    return qs_dhat_run(w.lat, m, w.tmp, w.ap, w.nrhs, 1, w.dwork, inv, live, w.p, sigma, w.part);
}

// x = (Q_hat(m)^2 + sigma)^-1 b by conjugate gradients (x0 = 0), every right-hand side to
// ||r|| <= tol ||b||; *iters: iterations taken.  No iteration waits for the host: it reads the
// convergence flags RW_LAG iterations late, and the iterations it has launched by then find
// every right-hand side converged and return at once.
int rw_cg(RwWork &w, double m, double sigma, const double *b, double *x, double tol, int max_iter, int *iters)
{
    cudaStream_t st = w.lat->stream;
    const int64_t n = w.len / 2;
    const unsigned nb = rw_blocks(n);
    const dim3 grid(nb, w.nrhs);
    rw_cg_start<<<grid, 256, 0, st>>>((const double2 *)b, (double2 *)x, (double2 *)w.r, (double2 *)w.p, n, w.part);
    rw_cg_first<<<w.nrhs, 256, 0, st>>>(w.sc, w.part, (int)nb, tol * tol);
    qs_note_launches(2);
    QS_TRY(rw_check("rw_cg"));
    QS_CUDA(cudaMemcpyAsync(w.hflag, w.sc.live[0], w.nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
    QS_CUDA(cudaMemcpyAsync(w.hnorm, w.sc.rr[0], w.nrhs * sizeof(double), cudaMemcpyDeviceToHost, st));
    QS_CUDA(cudaStreamSynchronize(st));
    for (int r = 0; r < w.nrhs; ++r) w.nan_rhs = w.nan_rhs || std::isnan(w.hnorm[r]);
    auto any = [&](const int *f) {
        for (int r = 0; r < w.nrhs; ++r)
            if (f[r]) return true;
        return false;
    };
    if (!any(w.hflag)) { *iters = 0; return QS_OK; }
    int it = 0, seen = 0;   // iterations launched, and those whose flags have been read
    while (seen < max_iter) {
        if (it < max_iter && it <= seen + RW_LAG) {
            const int o = it & 1;
            int np = 0;
            QS_TRY(rw_q2(w, m, sigma, w.sc.live[o], &np));
            rw_cg_r<<<grid, 256, 0, st>>>((double2 *)w.r, (const double2 *)w.ap, w.sc, o, n, w.part, np, w.rpart);
            rw_cg_xp<<<grid, 256, 0, st>>>((double2 *)x, (double2 *)w.p, (const double2 *)w.r, w.sc, o, n, w.part, np,
                                           w.rpart);
            qs_note_launches(2);
            QS_TRY(rw_check("rw_cg"));
            const int slot = it % (RW_LAG + 1);
            QS_CUDA(cudaMemcpyAsync(w.hflag + 64 * slot, w.sc.live[1 - o], w.nrhs * sizeof(int), cudaMemcpyDeviceToHost, st));
            QS_CUDA(cudaEventRecord(w.ev[slot], st));
            ++it;
            continue;
        }
        const int slot = seen % (RW_LAG + 1);
        QS_CUDA(cudaEventSynchronize(w.ev[slot]));
        ++seen;
        if (!any(w.hflag + 64 * slot)) { *iters = seen; return QS_OK; }
    }
    *iters = max_iter;
    return QS_ENOCONV;
}

// out = a^-1 in with a = D_hat(m) + i gamma_5 shift: (Q_hat(m) - i shift)(Q_hat^2 + shift^2)^-1 gamma_5 in
int rw_shifted_inverse(RwWork &w, double m, double shift, const double *in, double *out, double tol, int max_iter,
                       int *iters)
{
    const int64_t nc = (int64_t)w.nrhs * w.len / 2;
    cudaStream_t st = w.lat->stream;
    rw_g5<<<rw_grid(nc), 256, 0, st>>>((double2 *)w.t, (const double2 *)in, nc, 1);
    qs_note_launches(1);
    QS_TRY(rw_cg(w, m, shift * shift, w.t, w.x, tol, max_iter, iters));
    QS_TRY(qs_dhat_run(w.lat, m, w.x, out, w.nrhs, 1, w.dwork, w.inv_for(m)));
    rw_add_ix<<<rw_grid(nc), 256, 0, st>>>((double2 *)out, (const double2 *)out, (const double2 *)w.x, -shift, nc);
    qs_note_launches(1);
    return rw_check("rw_shifted_inverse");
}

}  // namespace

extern "C" int qs_w_mass(qs_lattice *lat, double m, double mp, int n, const double *nu, const double *mu,
                         const void *eta, int nsrc, double tol, int max_iter, double *q, double *log_w,
                         int *cg_iterations)
{
    if (!lat || !nu || !mu || !eta || !q || n < 1 || n > 32 || nsrc < 1 || nsrc > 64) return QS_EINVAL;
    if (!(tol > 0) || max_iter < 1 || ((uintptr_t)eta & 15)) return QS_EINVAL;
    for (int j = 0; j < n; ++j)
        if (!(nu[j] > 0) || !(mu[j] > 0)) return QS_EINVAL;
    if (!lat->gauge_loaded) return QS_EINVAL;
    const Geom &g = lat->g;
    if ((g.T | g.L) & 1) return QS_EINVAL;   // hopping must connect opposite parities only
    QS_CUDA(cudaSetDevice(lat->device));
    RwWork w;
    w.lat = lat;
    w.full = 0;
    w.nrhs = nsrc;
    w.len = g.Ns * 12;                      // half vectors
    const int64_t vl = (int64_t)nsrc * w.len;   // doubles per block of nsrc vectors
    double *buf = nullptr;
    const size_t inv_len = (size_t)36 * g.Vphys;   // complex entries of the inverses at one mass
    QS_CUDA(cudaMalloc(&buf, (10 * vl + rw_small(g, nsrc)) * sizeof(double) + 2 * inv_len * sizeof(double2)));
    w.eta = buf;
    w.t = buf + vl;
    w.x = buf + 2 * vl;
    w.r = buf + 3 * vl;
    w.p = buf + 4 * vl;
    w.ap = buf + 5 * vl;
    w.tmp = buf + 6 * vl;
    w.dwork = buf + 7 * vl;
    double *v1 = buf + 8 * vl, *v2 = buf + 9 * vl;
    double2 *inv = (double2 *)(buf + 10 * vl);
    w.mass[0] = m;
    w.mass[1] = mp;
    w.inv[0] = inv;
    w.inv[1] = inv + inv_len;
    cudaStream_t st = lat->stream;
    const int64_t nc = vl / 2;
    int total_it = 0;
    int s = rw_begin(w, (double *)(inv + 2 * inv_len));
    double lw = 0;
    if (s == QS_OK) do {
        if ((s = qs_parity_pack(lat, (const double *)eta, w.eta, nsrc, 0)) != QS_OK) break;
        if ((s = qs_clover_inverse_odd(lat, m, (double2 *)w.inv[0])) != QS_OK) break;
        if ((s = qs_clover_inverse_odd(lat, mp, (double2 *)w.inv[1])) != QS_OK) break;
        for (int j = 0; j < n && s == QS_OK; ++j) {
            int it = 0;
            // v1 = i gamma_5 (mu - nu) a^-1 eta, v2 = b^-1 v1 = S_j eta
            if ((s = rw_shifted_inverse(w, m, nu[j], w.eta, v1, tol, max_iter, &it)) != QS_OK) break;
            total_it += it;
            rw_ig5<<<rw_grid(nc), 256, 0, st>>>((double2 *)v1, (const double2 *)v1, mu[j] - nu[j], nc, 1);
            qs_note_launches(1);
            if ((s = rw_shifted_inverse(w, mp, mu[j], v1, v2, tol, max_iter, &it)) != QS_OK) break;
            total_it += it;
            // v1 = X eta = D_hat(m') S_j eta - D_hat(m) S_j eta
            if ((s = qs_dhat_run(lat, mp, v2, v1, nsrc, 0, w.dwork, w.inv_for(mp))) != QS_OK) break;
            if ((s = qs_dhat_run(lat, m, v2, w.tmp, nsrc, 0, w.dwork, w.inv_for(m))) != QS_OK) break;
            rw_axpy<<<rw_grid(vl), 256, 0, st>>>(v1, w.tmp, -1.0, vl);
            qs_note_launches(1);
            // q = (eta, R_j eta) = 2 Re (eta, X eta) + ||X eta||^2
            double ex[64], xx[64];
            if ((s = rw_dot(w, w.eta, v1, ex)) != QS_OK) break;
            if ((s = rw_dot(w, v1, v1, xx)) != QS_OK) break;
            double mx = -INFINITY;
            for (int l = 0; l < nsrc; ++l) {
                q[(size_t)j * nsrc + l] = 2 * ex[l] + xx[l];
                mx = std::max(mx, -q[(size_t)j * nsrc + l]);
            }
            double sum = 0;   // log of the mean of exp(-q), shifted by the largest exponent
            for (int l = 0; l < nsrc; ++l) sum += exp(-q[(size_t)j * nsrc + l] - mx);
            lw += mx + log(sum / nsrc);
        }
    } while (0);
    rw_end(w);
    cudaFree(buf);
    if (cg_iterations) *cg_iterations = total_it;
    if (s == QS_OK && log_w) *log_w = lw;
    return s;
}

// ---- the even-odd preconditioned solve of D x = b (Sec. 4) ---------------------------------
// even_odd = 1:  b'_e = b_e - D_eo (D_oo)^-1 b_o;  D_hat x_e = b'_e by CG on Q_hat^2
// (x_e = Q_hat (Q_hat^2)^-1 gamma_5 b'_e);  x_o = (D_oo)^-1 (b_o - D_oe x_e).
// even_odd = 0:  x = Q (Q^2)^-1 gamma_5 b by CG on the full-lattice Q^2 (the comparison).
extern "C" int qs_solve_D(qs_lattice *lat, double m0, const void *b, void *x, int nrhs, int even_odd, double tol,
                          int max_iter, int *iterations)
{
    if (!lat || !b || !x || nrhs < 1 || nrhs > 64 || !(tol > 0) || max_iter < 1) return QS_EINVAL;
    if (((uintptr_t)b | (uintptr_t)x) & 15) return QS_EINVAL;
    if (!lat->gauge_loaded) return QS_EINVAL;
    const Geom &g = lat->g;
    if (even_odd && ((g.T | g.L) & 1)) return QS_EINVAL;
    const size_t bytes = (size_t)nrhs * g.Ns * 24 * sizeof(double);
    const char *pa = (const char *)b, *pb = (const char *)x;
    if (pa < pb + bytes && pb < pa + bytes) return QS_EINVAL;
    QS_CUDA(cudaSetDevice(lat->device));
    RwWork w;
    w.lat = lat;
    w.full = even_odd ? 0 : 1;
    w.nrhs = nrhs;
    w.len = even_odd ? g.Ns * 12 : g.Ns * 24;
    const int64_t vl = (int64_t)nrhs * w.len;
    const size_t inv_len = even_odd ? (size_t)36 * g.Vphys : 0;
    double *buf = nullptr;
    QS_CUDA(cudaMalloc(&buf, (9 * vl + rw_small(g, nrhs)) * sizeof(double) + inv_len * sizeof(double2)));
    w.eta = nullptr;
    w.t = buf;
    w.x = buf + vl;
    w.r = buf + 2 * vl;
    w.p = buf + 3 * vl;
    w.ap = buf + 4 * vl;
    w.tmp = buf + 5 * vl;
    w.dwork = buf + 6 * vl;
    double *a1 = buf + 7 * vl, *a2 = buf + 8 * vl;
    double2 *inv = (double2 *)(buf + 9 * vl);
    w.mass[0] = w.mass[1] = m0;
    w.inv[0] = w.inv[1] = inv;
    cudaStream_t st = lat->stream;
    const int64_t nc = vl / 2;
    int s = rw_begin(w, (double *)(inv + inv_len)), it = 0;
    if (s == QS_OK) do {
        if (even_odd) {
            if ((s = qs_clover_inverse_odd(lat, m0, inv)) != QS_OK) break;
            if ((s = qs_parity_pack(lat, (const double *)b, w.tmp, nrhs, 1)) != QS_OK) break;
            if ((s = qs_hat_odd(lat, inv, w.tmp, a2, nrhs, 0, -1.0)) != QS_OK) break;       // -D_oo^-1 b_o
            if ((s = qs_parity_pack(lat, (const double *)b, w.tmp, nrhs, 0)) != QS_OK) break;
            if ((s = qs_hat_hop_even(lat, a2, w.tmp, 1.0, w.t, nrhs)) != QS_OK) break;      // b'_e
            rw_g5<<<rw_grid(nc), 256, 0, st>>>((double2 *)w.t, (const double2 *)w.t, nc, 1);
            qs_note_launches(1);
            if ((s = rw_cg(w, m0, 0.0, w.t, w.x, tol, max_iter, &it)) != QS_OK) break;
            if ((s = qs_dhat_run(lat, m0, w.x, a1, nrhs, 1, w.dwork, inv)) != QS_OK) break; // x_e
            if ((s = qs_hat_odd(lat, inv, a1, w.t, nrhs, 1, -1.0)) != QS_OK) break;         // -D_oo^-1 D_oe x_e
            if ((s = qs_parity_unpack(lat, a1, nullptr, (double *)x, nrhs, 0)) != QS_OK) break;
            if ((s = qs_parity_unpack(lat, w.t, a2, (double *)x, nrhs, 1)) != QS_OK) break; // x_o
        } else {
            rw_g5<<<rw_grid(nc), 256, 0, st>>>((double2 *)w.t, (const double2 *)b, nc, 0);
            qs_note_launches(1);
            if ((s = rw_cg(w, m0, 0.0, w.t, w.x, tol, max_iter, &it)) != QS_OK) break;
            double mm[64];
            for (int r = 0; r < nrhs; ++r) mm[r] = m0;
            if ((s = qs_dslash_run(lat, QS_F64, mm, w.x, x, nrhs, 1, 0)) != QS_OK) break;    // x = Q y
        }
        if ((s = rw_check("qs_solve_D")) != QS_OK) break;
        const cudaError_t e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) { qs_record_cuda_error(e, "qs_solve_D"); s = QS_ECUDA; }
        else if (w.nan_rhs) s = QS_ENUMERIC;   // the others are solved
    } while (0);
    rw_end(w);
    cudaFree(buf);
    if (iterations) *iterations = it;
    return s;
}
