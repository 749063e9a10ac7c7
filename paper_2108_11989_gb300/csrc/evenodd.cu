// Exact even-odd factor of the mass reweighting (Sec. 4):
//   W_eo(m -> m') = |det[D^oo_m' (D^oo_m)^-1]|^(1/2),
// D^oo = D restricted to the odd sites of the doubled lattice.  Hopping connects
// opposite parities only, so D^oo is site-diagonal: 4 + m0 + A(x), two 6 x 6 chiral
// blocks per site, and log|det D^oo| = sum over odd sites and blocks of log|det|.
// A physical site and its mirror have the same parity (L is even) and the mirror
// block S conj(A) S has the same (real) determinant, so the sum runs over odd physical
// sites and counts each twice.  One thread per physical site, a complex LU with
// partial pivoting per block in FP64, then a fixed-order two-stage sum.
#include "blas.cuh"
#include "dslash64.cuh"
#include "evenodd.cuh"

#include <math.h>
#include <stdlib.h>

namespace {

#define EO_MAX_MASS 16
#define EO_BLOCKS 304

__device__ double block_logdet(const double *__restrict__ clov, int64_t V, int64_t p, int b, double dm)
{
    double re[6][6], im[6][6];
    const double *cb = clov + (int64_t)b * 36 * V + p;
    for (int i = 0; i < 6; ++i) {
        re[i][i] = dm + cb[(int64_t)i * V];
        im[i][i] = 0.0;
        for (int j = 0; j < i; ++j) {
            const int k = 6 + 2 * qs_tri(i, j);
            re[i][j] = cb[(int64_t)k * V];
            im[i][j] = cb[(int64_t)(k + 1) * V];
            re[j][i] = re[i][j];          // Hermitian: upper = conj(lower)
            im[j][i] = -im[i][j];
        }
    }
    double acc = 0.0;
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        double best = re[c][c] * re[c][c] + im[c][c] * im[c][c];
        for (int r = c + 1; r < 6; ++r) {
            const double a = re[r][c] * re[r][c] + im[r][c] * im[r][c];
            if (a > best) { best = a; piv = r; }
        }
        if (piv != c)
            for (int j = 0; j < 6; ++j) {
                double t = re[c][j]; re[c][j] = re[piv][j]; re[piv][j] = t;
                t = im[c][j]; im[c][j] = im[piv][j]; im[piv][j] = t;
            }
        acc += 0.5 * log(best);           // log|u_cc|; a zero pivot gives -inf
        if (!(best > 0.0)) continue;
        const double ir = re[c][c] / best, ii = -im[c][c] / best;   // 1 / u_cc
        for (int r = c + 1; r < 6; ++r) {
            const double lr = re[r][c] * ir - im[r][c] * ii, li = re[r][c] * ii + im[r][c] * ir;
            for (int j = c + 1; j < 6; ++j) {
                re[r][j] -= lr * re[c][j] - li * im[c][j];
                im[r][j] -= lr * im[c][j] + li * re[c][j];
            }
        }
    }
    return acc;
}

__global__ void logdet_oo_kernel(Geom g, const double *__restrict__ clov, int nmass, const double *__restrict__ m0,
                                 double *part)
{
    __shared__ double sh[EO_MAX_MASS][8];
    double acc[EO_MAX_MASS];
    for (int q = 0; q < nmass; ++q) acc[q] = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < g.Vphys; p += (int64_t)gridDim.x * blockDim.x) {
        const int x = (int)(p % g.L);
        int64_t row = p / g.L;
        const int y = (int)(row % g.L);
        row /= g.L;
        const int z = (int)(row % g.L);
        const int t = (int)(row / g.L);
        if (((t + z + y + x) & 1) == 0) continue;
        for (int q = 0; q < nmass; ++q)
            for (int b = 0; b < 2; ++b) acc[q] += 2.0 * block_logdet(clov, g.Vphys, p, b, 4.0 + m0[q]);
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    for (int q = 0; q < nmass; ++q) {
        double v = acc[q];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (l == 0) sh[q][w] = v;
    }
    __syncthreads();
    if (threadIdx.x < nmass) {
        double s = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += sh[threadIdx.x][i];
        part[threadIdx.x * gridDim.x + blockIdx.x] = s;
    }
}

__global__ void sum_parts_kernel(const double *part, int nb, int nmass, double *out)
{
    const int q = threadIdx.x;
    if (q >= nmass) return;
    double s = 0.0;
    for (int i = 0; i < nb; ++i) s += part[q * nb + i];
    out[q] = s;
}

}  // namespace

extern "C" int qs_log_det_oo(qs_lattice *lat, int nmass, const double *m0, double *logdet)
{
    if (!lat || !m0 || !logdet || nmass < 1 || nmass > EO_MAX_MASS) return QS_EINVAL;
    if (!lat->gauge_loaded) return QS_EINVAL;
    QS_CUDA(cudaSetDevice(lat->device));
    double *d = nullptr;
    const size_t n = (size_t)EO_MAX_MASS + (size_t)EO_MAX_MASS * EO_BLOCKS + EO_MAX_MASS;
    QS_CUDA(cudaMalloc(&d, n * sizeof(double)));
    double *dm = d, *part = d + EO_MAX_MASS, *out = part + (size_t)EO_MAX_MASS * EO_BLOCKS;
    cudaError_t e = cudaMemcpyAsync(dm, m0, nmass * sizeof(double), cudaMemcpyHostToDevice, lat->stream);
    if (e == cudaSuccess) {
        logdet_oo_kernel<<<EO_BLOCKS, 256, 0, lat->stream>>>(lat->g, lat->clov64, nmass, dm, part);
        sum_parts_kernel<<<1, 32, 0, lat->stream>>>(part, EO_BLOCKS, nmass, out);
        qs_note_launches(2);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(logdet, out, nmass * sizeof(double), cudaMemcpyDeviceToHost, lat->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(lat->stream);
    cudaFree(d);
    if (e != cudaSuccess) {
        qs_record_cuda_error(e, "qs_log_det_oo");
        return QS_ECUDA;
    }
    for (int q = 0; q < nmass; ++q)
        if (!isfinite(logdet[q])) return QS_ENUMERIC;
    return QS_OK;
}

extern "C" int qs_w_eo(qs_lattice *lat, double m, double mp, double *w_eo, double *log_w_eo)
{
    if (!w_eo && !log_w_eo) return QS_EINVAL;
    double ms[2] = {m, mp}, ld[2];
    QS_TRY(qs_log_det_oo(lat, 2, ms, ld));
    const double lw = 0.5 * (ld[1] - ld[0]);
    if (log_w_eo) *log_w_eo = lw;
    if (w_eo) *w_eo = exp(lw);
    return QS_OK;
}

// ---- the even-odd preconditioned operator (Sec. 4) --------------------------------
// D_hat = D_ee - D_eo (D_oo)^-1 D_oe on the even sites, Q_hat = gamma_5 D_hat, in two passes:
//   v_o = -(D_oo)^-1 (D_oe x_e)  (hops, then the stored 6 x 6 inverses of the odd sites),
//   D_hat x_e = D_ee x_e + D_eo v_o.
// Vectors of one parity are stored alone, N_s / 2 sites in the site-tiled layout (site j of a
// parity is site s / 2 of the doubled lattice: a row of 2L sites holds L of each), so nothing
// is moved or computed for the other parity and the first pass has no SW term.  Bound by the
// FP64 pipe: 840 + 288 instructions per odd site and 1164 per even one, against 2 x 1650 + 430
// for two full-lattice site computations and a separate inverse.
// 8^3 x 16, 2 vectors: 40 + 42 us a D_hat against 2 x 75 + 26 + 4; qs_apply_Dhat on 12^3 x 24,
// 4 vectors: 2.87 -> 1.12 ms; the solve of 2 vectors there, to 1e-12: 203 -> 132 ms.
namespace {

struct Hat64 {
    Geom g;
    const double2 *links;
    const double *clov;
    const double2 *inv;
    int nrhs, gamma5;
    double dm;
    const int *live;      // NULL, or right-hand sides with live[r] = 0 are skipped
    // even pass: out += sigma add, part[r][tile] = Re (add, out)
    const double2 *add;
    double sigma;
    double *part;
};

// doubled site of the j-th site of a parity
__device__ __forceinline__ int parity_site(const Geom &g, int j, int parity)
{
    const int row = j / g.L, jx = j - row * g.L;
    const int y = row % g.L, z = (row / g.L) % g.L, t = row / (g.L * g.L);
    return row * g.L2 + 2 * jx + ((parity + t + z + y) & 1);
}

// rows of spin q of f (4 + m0 + A)^-1 v for chiral block b (stored inverse M; the mirror site's is
// S conj(M) S), v = own (spin q) and oth
__device__ __forceinline__ void inv_rows(const double2 *__restrict__ inv, int64_t V2, int64_t q, int b, double f,
                                         const Lane64 &ln, const double2 own[3], const double2 oth[3], double2 out[3])
{
    const int hq = ln.q ^ (ln.mir ? 1 : 0);
    const double2 *m = inv + ((int64_t)b * 36 + 18 * hq) * V2 + q;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        double2 o;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double2 e = __ldg(m + (int64_t)(6 * r + 3 * hq + c) * V2);
            e.y = qs_flip(e.y, ln.mir);
            o = c == 0 ? qs_cmul(e, own[c]) : qs_cfma(e, own[c], o);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double2 e = __ldg(m + (int64_t)(6 * r + 3 - 3 * hq + c) * V2);
            e.x = qs_flip(e.x, ln.mir);
            o = qs_cfma(e, oth[c], o);
        }
        out[r] = make_double2(f * o.x, f * o.y);
    }
}

__device__ __forceinline__ double2 partner_spin(double2 v)
{
    return make_double2(__shfl_xor_sync(0xffffffffu, v.x, 16), __shfl_xor_sync(0xffffffffu, v.y, 16));
}

// out_o = f (D_oo)^-1 (D_oe in_e) (HOP) or f (D_oo)^-1 in_o; in by AT, out tiled by parity
template <class AT, bool HOP>
__global__ void __launch_bounds__(128, 4) hat_odd_kernel(const __grid_constant__ Hat64 a, const double2 *__restrict__ in,
                                                         int64_t in_len, double2 *__restrict__ out, double f)
{
    const int r = (int)(blockIdx.x % (unsigned)a.nrhs);
    if (a.live && !a.live[r]) return;
    const int nh = (int)(a.g.Ns / 2);
    const int j0 = (int)(blockIdx.x / (unsigned)a.nrhs) * 64 + (int)(threadIdx.x >> 5) * 16 + (int)(threadIdx.x & 15);
    const int j = j0 < nh ? j0 : nh - 1;
    const Lane64 ln = qs_lane64(a.g, parity_site(a.g, j, 1));
    const double2 *v = in + r * in_len;
    double2 w[2][3];
    if constexpr (HOP) {
        qs_hops64<AT>(a.g, a.links, v, ln, w[0], w[1]);
    } else {
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            w[0][i] = __ldg(v + AT::at(ln.c.s, 3 * ln.q + i));
            w[1][i] = __ldg(v + AT::at(ln.c.s, 6 + 3 * ln.q + i));
        }
    }
    double2 *o = out + (int64_t)r * nh * 12;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        double2 oth[3], u[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) oth[i] = partner_spin(w[b][i]);
        inv_rows(a.inv, a.g.Vphys / 2, ln.c.p >> 1, b, f, ln, w[b], oth, u);
        if (j0 < nh) {
#pragma unroll
            for (int i = 0; i < 3; ++i) o[At64Tiled::at(j, 6 * b + 3 * ln.q + i)] = u[i];
        }
    }
}

// out_e = [gamma_5] (DIAG: (4 + m0 + A) x_e +) D_eo v_o (+ sigma add); v tiled by parity; x and out
// by AT, which for the full lattice also zeroes the odd site next to each even one.  part != NULL:
// the block's share of Re (add, out).
template <class AT, bool DIAG>
__global__ void __launch_bounds__(128, 4) hat_even_kernel(const __grid_constant__ Hat64 a, const double2 *__restrict__ v,
                                                          const double2 *__restrict__ x, double2 *__restrict__ out,
                                                          int64_t len, bool full)
{
    const int r = (int)(blockIdx.x % (unsigned)a.nrhs);
    if (a.live && !a.live[r]) return;
    const int nh = (int)(a.g.Ns / 2);
    const unsigned tile = blockIdx.x / (unsigned)a.nrhs;
    const int j0 = (int)tile * 64 + (int)(threadIdx.x >> 5) * 16 + (int)(threadIdx.x & 15);
    const int j = j0 < nh ? j0 : nh - 1;
    const Lane64 ln = qs_lane64(a.g, parity_site(a.g, j, 0));
    double2 w[2][3];
    qs_hops64<At64Half>(a.g, a.links, v + (int64_t)r * nh * 12, ln, w[0], w[1]);
    if constexpr (DIAG) qs_diag64<AT>(a.g, a.clov, x + r * len, ln, a.dm, w[0], w[1]);
    const unsigned g5 = a.gamma5 ? 0x80000000u : 0u;
    double acc = 0.0;
    double2 *o = out + r * len;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            double2 y = w[b][i];
            if (b) y = make_double2(qs_flip(y.x, g5), qs_flip(y.y, g5));
            const int64_t at = AT::at(ln.c.s, 6 * b + 3 * ln.q + i);
            if (a.add) {
                const double2 p = __ldg(a.add + r * len + at);
                y = make_double2(fma(a.sigma, p.x, y.x), fma(a.sigma, p.y, y.y));
                if (a.part) acc = fma(p.y, y.y, fma(p.x, y.x, acc));
            }
            if (j0 < nh) {
                o[at] = y;
                if (full) o[AT::at(ln.c.s ^ 1, 6 * b + 3 * ln.q + i)] = make_double2(0.0, 0.0);
            }
        }
    if (a.part) {
        __shared__ double sh[4];
        if (j0 >= nh) acc = 0.0;
        for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
        if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) a.part[(int64_t)r * (gridDim.x / a.nrhs) + tile] = (sh[0] + sh[1]) + (sh[2] + sh[3]);
    }
}

// canonical full-lattice vectors <-> tiled vectors of one parity; thread = (vector, site, component)
__global__ void parity_pack_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, Geom g, int k, int parity)
{
    const int64_t n = g.Ns / 2 * 12 * k;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t r = i / (g.Ns / 2 * 12), e = i - r * (g.Ns / 2 * 12);
    const int j = (int)(e / 12), c = (int)(e - 12 * (int64_t)j);
    const int s = parity_site(g, j, parity);
    out[r * (g.Ns / 2) * 12 + At64Tiled::at(j, c)] = in[(r * g.Ns + s) * 12 + c];
}

// x on the sites of `parity` of the full lattice = a (- b)
__global__ void parity_unpack_kernel(const double2 *__restrict__ a, const double2 *__restrict__ b,
                                     double2 *__restrict__ x, Geom g, int k, int parity)
{
    const int64_t n = g.Ns / 2 * 12 * k;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t r = i / (g.Ns / 2 * 12), e = i - r * (g.Ns / 2 * 12);
    const int j = (int)(e / 12), c = (int)(e - 12 * (int64_t)j);
    const int64_t at = r * (g.Ns / 2) * 12 + At64Tiled::at(j, c);
    double2 v = a[at];
    if (b) v = make_double2(v.x - b[at].x, v.y - b[at].y);
    x[(r * g.Ns + parity_site(g, j, parity)) * 12 + c] = v;
}

// inv = (4 + m0 + A(x))^-1 for every odd physical site x and chiral block (one thread each), by
// Gauss-Jordan elimination with partial pivoting in FP64; layout [block][6][6][V_phys / 2]
// complex, the odd physical site p at index p / 2 (L is even, so the odd sites of a row of L
// alternate).  The mirror site's block S conj(M) S has the inverse S conj(M^-1) S, formed on
// the fly when it is applied.
__global__ void clover_inverse_kernel(const double *__restrict__ clov, Geom g, double dm, double2 *__restrict__ inv)
{
    const int64_t V = g.Vphys, V2 = V / 2;
    const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i0 >= 2 * V2) return;
    const int b = i0 >= V2;
    const int64_t q = i0 - b * V2;
    int64_t p = 2 * q;   // the odd one of the sites 2q, 2q + 1 of a row
    {
        const int64_t row = p / g.L;
        const int x = (int)(p - row * g.L);
        const int y = (int)(row % g.L), z = (int)((row / g.L) % g.L), t = (int)(row / ((int64_t)g.L * g.L));
        p += ((t + z + y + x) & 1) ? 0 : 1;
    }
    const double *cb = clov + (int64_t)b * 36 * V + p;
    double ar[6][6], ai[6][6], br[6][6], bi[6][6];
    for (int i = 0; i < 6; ++i) {
        ar[i][i] = dm + cb[(int64_t)i * V];
        ai[i][i] = 0.0;
        for (int j = 0; j < i; ++j) {
            const int k = 6 + 2 * qs_tri(i, j);
            ar[i][j] = cb[(int64_t)k * V];
            ai[i][j] = cb[(int64_t)(k + 1) * V];
            ar[j][i] = ar[i][j];      // Hermitian: upper = conj(lower)
            ai[j][i] = -ai[i][j];
        }
        for (int j = 0; j < 6; ++j) { br[i][j] = i == j ? 1.0 : 0.0; bi[i][j] = 0.0; }
    }
    for (int c = 0; c < 6; ++c) {
        int piv = c;
        double best = ar[c][c] * ar[c][c] + ai[c][c] * ai[c][c];
        for (int r = c + 1; r < 6; ++r) {
            const double a2 = ar[r][c] * ar[r][c] + ai[r][c] * ai[r][c];
            if (a2 > best) { best = a2; piv = r; }
        }
        if (piv != c)
            for (int j = 0; j < 6; ++j) {
                double w = ar[c][j]; ar[c][j] = ar[piv][j]; ar[piv][j] = w;
                w = ai[c][j]; ai[c][j] = ai[piv][j]; ai[piv][j] = w;
                w = br[c][j]; br[c][j] = br[piv][j]; br[piv][j] = w;
                w = bi[c][j]; bi[c][j] = bi[piv][j]; bi[piv][j] = w;
            }
        const double pr = ar[c][c] / best, pim = -ai[c][c] / best;   // 1 / pivot
        for (int j = 0; j < 6; ++j) {
            double w = ar[c][j] * pr - ai[c][j] * pim;
            ai[c][j] = ar[c][j] * pim + ai[c][j] * pr;
            ar[c][j] = w;
            w = br[c][j] * pr - bi[c][j] * pim;
            bi[c][j] = br[c][j] * pim + bi[c][j] * pr;
            br[c][j] = w;
        }
        for (int r = 0; r < 6; ++r) {
            if (r == c) continue;
            const double fr = ar[r][c], fi = ai[r][c];
            for (int j = 0; j < 6; ++j) {
                ar[r][j] -= fr * ar[c][j] - fi * ai[c][j];
                ai[r][j] -= fr * ai[c][j] + fi * ar[c][j];
                br[r][j] -= fr * br[c][j] - fi * bi[c][j];
                bi[r][j] -= fr * bi[c][j] + fi * br[c][j];
            }
        }
    }
    for (int i = 0; i < 6; ++i)
        for (int j = 0; j < 6; ++j) inv[((int64_t)b * 36 + i * 6 + j) * V2 + q] = make_double2(br[i][j], bi[i][j]);
}

Hat64 hat_args(qs_lattice *lat, double m0, int nrhs, int gamma5, const double2 *inv, const int *live)
{
    Hat64 a;
    a.g = lat->g;
    a.links = lat->links64;
    a.clov = lat->clov64;
    a.inv = inv;
    a.nrhs = nrhs;
    a.gamma5 = gamma5;
    a.dm = 4.0 + m0;
    a.live = live;
    a.add = nullptr;
    a.sigma = 0.0;
    a.part = nullptr;
    return a;
}

unsigned hat_grid(const Geom &g, int nrhs) { return (unsigned)(((g.Ns / 2 + 63) / 64) * nrhs); }

int launched(int n, const char *where)
{
    qs_note_launches(n);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { qs_record_cuda_error(e, where); return QS_ECUDA; }
    return QS_OK;
}

}  // namespace

int64_t qs_hat_tiles(const Geom &g) { return (g.Ns / 2 + 63) / 64; }

int qs_clover_inverse_odd(qs_lattice *lat, double m0, double2 *inv)
{
    const int64_t n = lat->g.Vphys;
    clover_inverse_kernel<<<(unsigned)((n + 63) / 64), 64, 0, lat->stream>>>(lat->clov64, lat->g, 4.0 + m0, inv);
    return launched(1, "qs_clover_inverse_odd");
}

int qs_parity_pack(qs_lattice *lat, const double *in, double *out, int nrhs, int parity)
{
    const int64_t n = lat->g.Ns / 2 * 12 * nrhs;
    parity_pack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, lat->stream>>>((const double2 *)in, (double2 *)out, lat->g,
                                                                             nrhs, parity);
    return launched(1, "qs_parity_pack");
}

int qs_parity_unpack(qs_lattice *lat, const double *a, const double *b, double *x, int nrhs, int parity)
{
    const int64_t n = lat->g.Ns / 2 * 12 * nrhs;
    parity_unpack_kernel<<<(unsigned)((n + 255) / 256), 256, 0, lat->stream>>>(
        (const double2 *)a, (const double2 *)b, (double2 *)x, lat->g, nrhs, parity);
    return launched(1, "qs_parity_unpack");
}

int qs_hat_odd(qs_lattice *lat, const double2 *inv, const double *in, double *out, int nrhs, int hop, double f,
               const int *live)
{
    const Hat64 a = hat_args(lat, 0.0, nrhs, 0, inv, live);
    const int64_t len = lat->g.Ns / 2 * 12;
    if (hop)
        hat_odd_kernel<At64Half, true><<<hat_grid(a.g, nrhs), 128, 0, lat->stream>>>(a, (const double2 *)in, len,
                                                                                     (double2 *)out, f);
    else
        hat_odd_kernel<At64Half, false><<<hat_grid(a.g, nrhs), 128, 0, lat->stream>>>(a, (const double2 *)in, len,
                                                                                      (double2 *)out, f);
    return launched(1, "qs_hat_odd");
}

int qs_hat_hop_even(qs_lattice *lat, const double *v, const double *add, double sigma, double *out, int nrhs)
{
    Hat64 a = hat_args(lat, 0.0, nrhs, 0, nullptr, nullptr);
    a.add = (const double2 *)add;
    a.sigma = sigma;
    hat_even_kernel<At64Half, false><<<hat_grid(a.g, nrhs), 128, 0, lat->stream>>>(
        a, (const double2 *)v, nullptr, (double2 *)out, a.g.Ns / 2 * 12, false);
    return launched(1, "qs_hat_hop_even");
}

int qs_dhat_run(qs_lattice *lat, double m0, const double *in, double *out, int nrhs, int gamma5, double *work,
                const double2 *inv, const int *live, const double *add, double sigma, double *part)
{
    QS_TRY(qs_hat_odd(lat, inv, in, work, nrhs, 1, -1.0, live));
    Hat64 a = hat_args(lat, m0, nrhs, gamma5, inv, live);
    a.add = (const double2 *)add;
    a.sigma = sigma;
    a.part = part;
    hat_even_kernel<At64Half, true><<<hat_grid(a.g, nrhs), 128, 0, lat->stream>>>(
        a, (const double2 *)work, (const double2 *)in, (double2 *)out, a.g.Ns / 2 * 12, false);
    return launched(1, "qs_dhat_run");
}

extern "C" int qs_apply_Dhat(qs_lattice *lat, double m0, const void *in, void *out, int nrhs, int gamma5)
{
    if (!lat || !in || !out || nrhs < 1 || nrhs > 64) return QS_EINVAL;
    if (!lat->gauge_loaded) return QS_EINVAL;
    const Geom &g = lat->g;
    if ((g.T | g.L) & 1) return QS_EINVAL;   // hopping must connect opposite parities only
    const size_t bytes = (size_t)nrhs * g.Ns * 24 * sizeof(double);
    const char *pa = (const char *)in, *pb = (const char *)out;
    if (pa < pb + bytes && pb < pa + bytes) return QS_EINVAL;
    if (((uintptr_t)in | (uintptr_t)out) & 15) return QS_EINVAL;
    QS_CUDA(cudaSetDevice(lat->device));
    double *buf = nullptr;
    const size_t inv_len = (size_t)36 * g.Vphys;
    QS_CUDA(cudaMalloc(&buf, bytes / 2 + inv_len * sizeof(double2)));
    double2 *inv = (double2 *)(buf + bytes / 2 / sizeof(double));
    int s = qs_clover_inverse_odd(lat, m0, inv);
    if (s == QS_OK) {
        const Hat64 a = hat_args(lat, m0, nrhs, gamma5, inv, nullptr);
        hat_odd_kernel<At64Canon, true><<<hat_grid(g, nrhs), 128, 0, lat->stream>>>(a, (const double2 *)in, g.Ns * 12,
                                                                                    (double2 *)buf, -1.0);
        hat_even_kernel<At64Canon, true><<<hat_grid(g, nrhs), 128, 0, lat->stream>>>(
            a, (const double2 *)buf, (const double2 *)in, (double2 *)out, g.Ns * 12, true);
        s = launched(2, "qs_apply_Dhat");
    }
    if (s == QS_OK) {
        const cudaError_t e = cudaStreamSynchronize(lat->stream);
        if (e != cudaSuccess) { qs_record_cuda_error(e, "qs_apply_Dhat"); s = QS_ECUDA; }
    }
    cudaFree(buf);
    return s;
}
