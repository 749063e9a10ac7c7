// Vector, block and reduction kernels of the eigensolver and the CG.
// Reductions are two-stage: partial sums of a grid that depends on the vector's length alone
// (red_blocks), then one fixed-order pass.  So results are bit-reproducible, and a vector's sum
// does not depend on how many others it is summed with.
#include "blas.cuh"

#include <mutex>
#include <type_traits>

namespace {

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// block-wide sum (blockDim.x a multiple of 32, <= 1024); result valid in thread 0
__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double sh[32];
    v = warp_sum(v);
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    int nw = blockDim.x >> 5;
    v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
    if (w == 0) v = warp_sum(v);
    return v;
}

// (hi, lo) += x, with hi + lo exact to the rounding of the final add (Knuth's two-sum)
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x)
{
    const float s = hi + x;
    const float bp = s - hi;
    const float err = (hi - (s - bp)) + (x - bp);
    hi = s;
    lo += err;
}
__device__ __forceinline__ void two_sum_acc(double &hi, double &, double x) { hi += x; }
// the pair's value; a sum that has left the range is infinite (its error term is then NaN)
__device__ __forceinline__ double pair_value(float hi, float lo) { return isinf(hi) ? (double)hi : (double)hi + (double)lo; }
__device__ __forceinline__ double pair_value(double hi, double) { return hi; }

template <typename R> struct Vec16;   // 16 bytes of reals
template <> struct Vec16<float> { typedef float4 T; };
template <> struct Vec16<double> { typedef double2 T; };
// (hi, lo) += the squares of a word's reals.  FP32: exact squares by fused multiply-adds and two-sum
// (hi + a a = s + e with s rounded, b = s - hi, e = (a a - b) + (hi - (s - b))); a plain chain of the
// word's four is about twice as far from the 64-bit sum on 4^4 to 6^3 x 8 as one or two squares per
// thread are
__device__ __forceinline__ void add_sq(float &hi, float &lo, float a)
{
    const float s = fmaf(a, a, hi), nb = hi - s;
    lo += fmaf(a, a, nb) + (hi - (s + nb));
    hi = s;
}
__device__ __forceinline__ void add_sq(float &hi, float &lo, float4 a)
{
    add_sq(hi, lo, a.x);
    add_sq(hi, lo, a.y);
    add_sq(hi, lo, a.z);
    add_sq(hi, lo, a.w);
}
__device__ __forceinline__ void add_sq(double &hi, double &, double2 a) { hi += fma(a.y, a.y, a.x * a.x); }
__device__ __forceinline__ float4 diff(float4 a, float t, float4 b)
{
    return make_float4(fmaf(-t, b.x, a.x), fmaf(-t, b.y, a.y), fmaf(-t, b.z, a.z), fmaf(-t, b.w, a.w));
}
__device__ __forceinline__ double2 diff(double2 a, double t, double2 b) { return make_double2(fma(-t, b.x, a.x), fma(-t, b.y, a.y)); }

// Streaming kernels over [k][nr]: 16-byte words (nr is a multiple of 24 x 16), red_blocks(nr) blocks
// per vector, so that a block has some two thousand reals to itself; with 608 blocks per vector
// whatever its length a thread of an 8^3 x 12 problem has two.  FP32 sums are kept as a two-sum pair.
template <typename R>
__global__ void __launch_bounds__(256) norm2_part(const R *__restrict__ v, int64_t nr, double *part)
{
    typedef typename Vec16<R>::T T;
    const int64_t n = nr * (int64_t)sizeof(R) / 16;
    const T *x = reinterpret_cast<const T *>(v) + (int64_t)blockIdx.y * n;
    R acc = 0, lo = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        add_sq(acc, lo, x[i]);
    double s = block_sum(pair_value(acc, lo));
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// sum of nb partials per output (one block per output), fixed order
__global__ void finalize_sum(const double *part, int nb, int stride_out, double *out)
{
    const double *p = part + (int64_t)blockIdx.x * nb;
    double acc = 0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) acc += p[i];
    double s = block_sum(acc);
    if (threadIdx.x == 0) out[(int64_t)blockIdx.x * stride_out] = s;
}

template <typename R>
__global__ void __launch_bounds__(256) resid_part(const R *__restrict__ a, const R *__restrict__ b, const double *theta,
                                                  int64_t nr, double *part)
{
    typedef typename Vec16<R>::T T;
    const int64_t n = nr * (int64_t)sizeof(R) / 16;
    const T *x = reinterpret_cast<const T *>(a) + (int64_t)blockIdx.y * n;
    const T *y = reinterpret_cast<const T *>(b) + (int64_t)blockIdx.y * n;
    const R t = (R)theta[blockIdx.y];
    R acc = 0, lo = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        add_sq(acc, lo, diff(x[i], t, y[i]));
    double s = block_sum(pair_value(acc, lo));
    if (threadIdx.x == 0) part[blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// Gram partials G[i][j] = sum_e conj(A_i[e]) B_j[e] (i < ka, j < kb <= 64).  A block
// stages a chunk of GE elements of all vectors in shared memory, element-major
// ([e][vector], row padded by one complex to spread the banks); each thread owns a 4 x 4
// tile of (i, j) and a residue class of the chunk's elements, so every staged value it
// reads feeds four complex multiply-adds.  The element classes of a tile are summed in
// shared memory at the end, in a fixed order.  LOWP: values rounded to FP32, products
// and the sum over one chunk in FP32 (packed, two per instruction), chunk sums in FP64.
// herm (A = B): G is Hermitian, only the tiles of the upper triangle are computed and the vectors are
// staged once.  FP64 products are bound by the FP64 pipe (12^3 x 24, 16 vectors: 1.85 -> 1.38 ms with
// 10 of 16 tiles), FP32 ones by issue and by the block's own reduction (8^3 x 12, 32 vectors:
// 134 -> 87 us with 36 of 64 tiles, two blocks per SM instead of four and one conversion per total).
// V^H (Q V) is Hermitian only up to rounding, and its reader takes the mean of both triangles, which
// halves the error's variance: it is computed whole.
#define GE 64
__device__ __forceinline__ float2 pk_fma(float a, float2 b, float2 c) { return __ffma2_rn(make_float2(a, a), b, c); }

template <bool LOWP, typename TIn = double2>
__global__ void __launch_bounds__(256, LOWP ? 2 : 1) gram_tile_kernel(const TIn *__restrict__ A_, int ka,
                                                           const TIn *__restrict__ B_, int kb, int64_t nc,
                                                           double *part, int herm)
{
    typedef typename std::conditional<LOWP, float2, double2>::type V2;
    typedef typename std::conditional<LOWP, float, double>::type T;
    extern __shared__ __align__(16) unsigned char gsm_raw[];
    V2 *sv = reinterpret_cast<V2 *>(gsm_raw);
    const int kk = herm ? ka : ka + kb, row = kk + 1;   // padded row of one element
    const int boff = herm ? 0 : ka;
    const int ti_n = (ka + 3) / 4, tj_n = (kb + 3) / 4;
    const int ntile = herm ? ti_n * (ti_n + 1) / 2 : ti_n * tj_n;
    const int eg_n = 256 / ntile;                     // element classes (>= 1)
    const int t = threadIdx.x;
    const int tile = t % ntile, eg = t / ntile;
    const bool active = eg < eg_n;
    int ti, tj;   // herm: tiles row by row of the upper triangle
    auto place = [&](int q, int &i, int &j) {
        if (!herm) { i = q / tj_n; j = q % tj_n; return; }
        i = 0;
        while (q >= ti_n - i) { q -= ti_n - i; ++i; }
        j = i + q;
    };
    place(tile, ti, tj);
    const int i0 = 4 * ti, j0 = 4 * tj;
    // running totals: FP64 (FP64 products), or an FP32 (hi, lo) pair per real sum kept
    // exact to ~2^-48 by Knuth's two-sum (FP32 products: GB300's FP64 pipe is too slow
    // for a per-chunk FP64 add)
    typedef typename std::conditional<LOWP, float, double>::type A;
    A acc[4][4][2], accl[4][4][2];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b][0] = acc[a][b][1] = accl[a][b][0] = accl[a][b][1] = (A)0;
    const int64_t nch = (nc + GE - 1) / GE;
    const int nq = kk * GE;
    for (int64_t ch = blockIdx.x; ch < nch; ch += gridDim.x) {
        const int64_t e0 = ch * GE;
        __syncthreads();
        // staging: SU independent loads in flight per thread before their stores
        constexpr int SU = LOWP ? 4 : 8;
        for (int q0 = t; q0 < nq; q0 += 256 * SU) {
            TIn val[SU];
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                const int q = q0 + 256 * u;
                val[u].x = 0;
                val[u].y = 0;
                if (q < nq) {
                    const int v = q / GE, e = q % GE;
                    const int64_t idx = e0 + e;
                    if (idx < nc) val[u] = v < ka ? __ldg(A_ + (int64_t)v * nc + idx) : __ldg(B_ + (int64_t)(v - ka) * nc + idx);
                }
            }
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                const int q = q0 + 256 * u;
                if (q < nq) {
                    V2 x;
                    x.x = (T)val[u].x;
                    x.y = (T)val[u].y;
                    sv[(q % GE) * row + q / GE] = x;
                }
            }
        }
        __syncthreads();
        if (!active) continue;
        if constexpr (LOWP) {
            // FP32 sums over the chunk, added to the (hi, lo) totals once per chunk:
            // conj(x) y = x.re (y.re, y.im) + x.im (y.im, -y.re)
            float2 c[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) c[a][b] = make_float2(0.f, 0.f);
            for (int e = eg; e < GE; e += eg_n) {
                const V2 *r = sv + e * row;
                V2 x[4], y[4], z[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) x[a] = (i0 + a < ka) ? r[i0 + a] : V2{0.f, 0.f};
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    y[b] = (j0 + b < kb) ? r[boff + j0 + b] : V2{0.f, 0.f};
                    z[b] = make_float2(y[b].y, -y[b].x);
                }
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) c[a][b] = pk_fma(x[a].y, z[b], pk_fma(x[a].x, y[b], c[a][b]));
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    two_sum_acc(acc[a][b][0], accl[a][b][0], c[a][b].x);
                    two_sum_acc(acc[a][b][1], accl[a][b][1], c[a][b].y);
                }
        } else {
            for (int e = eg; e < GE; e += eg_n) {
                const V2 *r = sv + e * row;
                V2 x[4], y[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) x[a] = (i0 + a < ka) ? r[i0 + a] : V2{0.0, 0.0};
#pragma unroll
                for (int b = 0; b < 4; ++b) y[b] = (j0 + b < kb) ? r[boff + j0 + b] : V2{0.0, 0.0};
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {   // conj(x) y
                        acc[a][b][0] = fma(x[a].x, y[b].x, fma(x[a].y, y[b].y, acc[a][b][0]));
                        acc[a][b][1] = fma(x[a].x, y[b].y, fma(-x[a].y, y[b].x, acc[a][b][1]));
                    }
            }
        }
    }
    // sum the element classes of each tile (fixed order), reusing the staging buffer; FP32 sums
    // stay two-sum pairs until the block's total, since each conversion to FP64 costs what an
    // FP64 addition does
    typedef typename std::conditional<LOWP, float2, double>::type S;
    __syncthreads();
    S *red = reinterpret_cast<S *>(gsm_raw);   // [ntile][32]
    for (int c = 0; c < eg_n; ++c) {
        if (active && eg == c) {
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        S &d = red[tile * 32 + (a * 4 + b) * 2 + h];
                        if constexpr (LOWP) {
                            if (c == 0) {
                                d = make_float2(acc[a][b][h], accl[a][b][h]);
                            } else {
                                two_sum_acc(d.x, d.y, acc[a][b][h]);
                                d.y += accl[a][b][h];
                            }
                        } else {
                            d = c == 0 ? acc[a][b][h] : d + acc[a][b][h];
                        }
                    }
        }
        __syncthreads();
    }
    double *out = part + (int64_t)blockIdx.x * 2 * ka * kb;
    for (int q = t; q < ntile * 32; q += 256) {
        const int tl = q / 32, ab = (q % 32) / 2, a = ab / 4, b = ab % 4;
        int pi, pj;
        place(tl, pi, pj);
        const int i = 4 * pi + a, j = 4 * pj + b;
        if (i < ka && j < kb) {
            if constexpr (LOWP) out[2 * (i * kb + j) + (q & 1)] = (double)red[q].x + (double)red[q].y;
            else out[2 * (i * kb + j) + (q & 1)] = red[q];
        }
    }
}

// G from the partials [nb][2 ka kb]: 32 consecutive reals per block, 8 warps over the partials
// (fixed order); herm: entries below the computed tiles are the conjugates of those above
__global__ void __launch_bounds__(256) gram_sum_kernel(const double *__restrict__ part, int nb, int n, int kb, int herm, double *G)
{
    __shared__ double sh[8][32];
    const int l = threadIdx.x & 31, w = threadIdx.x >> 5, q = blockIdx.x * 32 + l;
    const int i = q / 2 / kb, j = q / 2 % kb;
    const bool on = q < n && !(herm && i / 4 > j / 4);
    double s = 0;
    if (on) {
#pragma unroll 4
        for (int b = w; b < nb; b += 8) s += part[(int64_t)b * n + q];
    }
    sh[w][l] = s;
    __syncthreads();
    if (w != 0 || !on) return;
    for (int v = 1; v < 8; ++v) s += sh[v][l];
    G[q] = s;
    if (herm && i / 4 < j / 4) G[2 * (j * kb + i) + (q & 1)] = (q & 1) ? -s : s;
}

// V_j = sum_i W_i C[i][j] (j < kc): each thread computes RE elements for a block of
// up to RJ output vectors, the coefficients read from shared memory (the same word for
// all threads of a warp); each W value it loads feeds RJ multiply-adds.  LOWP: values and
// coefficients rounded to FP32, the sums in FP32.  upper: C is upper triangular (the inverse
// Cholesky factor), so a pass of RJ columns needs the first j0 + RJ vectors only; FP64 rotations
// are bound by the FP64 pipe (8^3 x 12, 32 vectors: 1.02 ms whole, 0.64 ms upper).
#define RE 2
template <bool LOWP, typename TIn = double2, typename TOut = double2>
__global__ void __launch_bounds__(256, 2) rotate_tile_kernel(const TIn *__restrict__ W, int ka,
                                                             const double2 *__restrict__ C, int kc, int64_t nc,
                                                             TOut *__restrict__ V, int upper)
{
    typedef typename std::conditional<LOWP, float2, double2>::type V2;
    typedef typename std::conditional<LOWP, float, double>::type T;
    constexpr int RJ = LOWP ? 16 : 8;   // output columns per pass (register budget)
    extern __shared__ __align__(16) unsigned char rsm_raw[];
    V2 *cs = reinterpret_cast<V2 *>(rsm_raw);         // [ka][kc]
    for (int q = threadIdx.x; q < ka * kc; q += blockDim.x) {
        V2 x;
        x.x = (T)C[q].x;
        x.y = (T)C[q].y;
        cs[q] = x;
    }
    __syncthreads();
    const int64_t stride = (int64_t)gridDim.x * blockDim.x * RE;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x * RE + threadIdx.x; base < nc; base += stride) {
        for (int j0 = 0; j0 < kc; j0 += RJ) {
            T ar[RE][RJ], ai[RE][RJ];
#pragma unroll
            for (int u = 0; u < RE; ++u)
#pragma unroll
                for (int jj = 0; jj < RJ; ++jj) ar[u][jj] = ai[u][jj] = (T)0;
            const int itop = upper && j0 + RJ < ka ? j0 + RJ : ka;   // C[i][j] = 0 for i > j
            for (int i0 = 0; i0 < itop; i0 += 4) {
                // four input vectors' values loaded together (independent loads in flight)
                T wr[4][RE], wi[4][RE];
#pragma unroll
                for (int di = 0; di < 4; ++di)
#pragma unroll
                    for (int u = 0; u < RE; ++u) {
                        const int64_t e = base + (int64_t)u * blockDim.x;
                        TIn w;
                        w.x = 0;
                        w.y = 0;
                        if (e < nc && i0 + di < ka) w = __ldg(W + (int64_t)(i0 + di) * nc + e);
                        wr[di][u] = (T)w.x;
                        wi[di][u] = (T)w.y;
                    }
#pragma unroll
                for (int di = 0; di < 4; ++di) {
                    if (i0 + di >= ka) break;
                    const V2 *crow = cs + (i0 + di) * kc + j0;
#pragma unroll
                    for (int jj = 0; jj < RJ; ++jj) {
                        if (j0 + jj < kc) {
                            const V2 c = crow[jj];
#pragma unroll
                            for (int u = 0; u < RE; ++u) {
                                ar[u][jj] = fma(wr[di][u], c.x, fma(-wi[di][u], c.y, ar[u][jj]));
                                ai[u][jj] = fma(wr[di][u], c.y, fma(wi[di][u], c.x, ai[u][jj]));
                            }
                        }
                    }
                }
            }
#pragma unroll
            for (int jj = 0; jj < RJ; ++jj)
                if (j0 + jj < kc)
#pragma unroll
                    for (int u = 0; u < RE; ++u) {
                        const int64_t e = base + (int64_t)u * blockDim.x;
                        if (e < nc) {
                            TOut o;
                            o.x = ar[u][jj];
                            o.y = ai[u][jj];
                            V[(int64_t)(j0 + jj) * nc + e] = o;
                        }
                    }
        }
    }
}

__global__ void d2f_kernel(const double *__restrict__ x, float *__restrict__ y, const double *scale, int64_t nr)
{
    double s = scale ? scale[blockIdx.y] : 1.0;
    const double *a = x + (int64_t)blockIdx.y * nr;
    float *b = y + (int64_t)blockIdx.y * nr;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (float)(a[i] * s);
}

__global__ void f2d_kernel(const float *__restrict__ x, double *__restrict__ y, int64_t nr)
{
    const float *a = x + (int64_t)blockIdx.y * nr;
    double *b = y + (int64_t)blockIdx.y * nr;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (double)a[i];
}

__global__ void axpy_f2d_kernel(double *__restrict__ x, const float *__restrict__ e, const double *coef, int64_t nr)
{
    double c = coef[blockIdx.y];
    double *a = x + (int64_t)blockIdx.y * nr;
    const float *b = e + (int64_t)blockIdx.y * nr;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x)
        a[i] += c * (double)b[i];
}

template <typename R>
__global__ void scale_cols_kernel(R *x, const double *scale, int64_t nr)
{
    const R c = (R)scale[blockIdx.y];
    R *a = x + (int64_t)blockIdx.y * nr;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x)
        a[i] *= c;
}

__global__ void scaled_copy_kernel(double *x, const double *b, const double *coef, int64_t nr)
{
    double c = coef[blockIdx.y];
    double *a = x + (int64_t)blockIdx.y * nr;
    const double *q = b + (int64_t)blockIdx.y * nr;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nr; i += (int64_t)gridDim.x * blockDim.x)
        a[i] = c * q[i];
}

template <typename R>
__global__ void cheb_kernel(R *__restrict__ ynew, const R *__restrict__ ay, const R *__restrict__ y,
                            const R *__restrict__ x, R c, R s1, R s2, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        ynew[i] = s1 * (ay[i] - c * y[i]) - s2 * x[i];
}

template <typename R>
__global__ void axpby_kernel(R a, const R *__restrict__ x, R b, R *__restrict__ y, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = a * x[i] + b * y[i];
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t z)
{
    z += 0x9e3779b97f4a7c15ULL;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
    return z ^ (z >> 31);
}

__global__ void gauss_kernel(double *x, int64_t n, uint64_t seed)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t h1 = splitmix64(seed ^ splitmix64(2 * (uint64_t)i));
        uint64_t h2 = splitmix64(seed ^ splitmix64(2 * (uint64_t)i + 1));
        double u1 = ((h1 >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        double u2 = ((h2 >> 11) + 0.5) * (1.0 / 9007199254740992.0);
        x[i] = sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
    }
}

__global__ void map_scalars_kernel(const double *in, double *out, int k, int mode)
{
    int r = threadIdx.x;
    if (r >= k) return;
    double v = in[r];
    if (mode == 0) out[r] = v > 0 ? 1.0 / sqrt(v) : 0.0;      // 1/sqrt
    else if (mode == 1) out[r] = sqrt(v > 0 ? v : 0.0);        // sqrt
    else if (mode == 2) out[r] = v != 0 ? 1.0 / (v * v) : 0.0; // theta^-2
    else out[r] = v;
}

// ---- CG (FP32 vectors, FP64 scalars) ----------------------------------------
// An iteration is t = Q p with the shares of |t|^2 (= <p, Q^2 p>), alpha, r -= alpha Q t with the
// shares of |r|^2, beta, and the update of x and p: five launches, of which only the last streams
// vectors of its own (Q^2 p is never written, and neither it nor Q p is read for a sum).  Vectors
// that have converged are skipped.  12^3 x 24, 8 vectors, per iteration: 159 us, 192 with separate
// passes for |Q p|^2 and r.
// alpha = |r|^2 / |Q p|^2, one block per vector; 0 for vectors that are done
__global__ void __launch_bounds__(256) cg_alpha_kernel(CgScalars s, const double *part, int nb)
{
    const int q = blockIdx.x;
    double acc = 0;
    if (s.live[q])
        for (int i = threadIdx.x; i < nb; i += 256) acc += part[(int64_t)q * nb + i];
    acc = block_sum(acc);
    if (threadIdx.x == 0) s.alpha[q] = s.live[q] && acc > 0 ? (float)(s.rr[q] / acc) : 0.f;
}

// beta = |r|^2 / |r_old|^2; the vector lives on while |r|^2 > tol2 |r_0|^2
__global__ void __launch_bounds__(256) cg_beta_kernel(CgScalars s, const double *part, int nb, double tol2)
{
    const int q = blockIdx.x;
    if (!s.live[q]) return;
    double acc = 0;
    for (int i = threadIdx.x; i < nb; i += 256) acc += part[(int64_t)q * nb + i];
    acc = block_sum(acc);
    if (threadIdx.x != 0) return;
    s.beta[q] = s.rr[q] > 0 ? (float)(acc / s.rr[q]) : 0.f;
    s.rr[q] = acc;
    ++s.iters[q];
    s.live[q] = acc > tol2 * s.rr0[q] && isfinite(acc);
}

// x += alpha p, p = r + beta p
__global__ void __launch_bounds__(256) cg_xp_kernel(float4 *__restrict__ x, float4 *__restrict__ p,
                                                    const float4 *__restrict__ r, CgScalars s, int64_t n)
{
    const int q = blockIdx.y;
    const float a = s.alpha[q], b = s.beta[q];
    if (a == 0.f) return;
    const bool live = s.live[q];
    float4 *xq = x + q * n, *pq = p + q * n;
    const float4 *rq = r + q * n;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 v = pq[i];
        xq[i] = diff(xq[i], -a, v);
        if (live) pq[i] = diff(rq[i], -b, v);
    }
}

__global__ void cg_init_kernel(CgScalars s, const double *rr, int k)
{
    int q = threadIdx.x;
    if (q >= k) return;
    s.rr[q] = rr[q];
    s.rr0[q] = rr[q];
    s.live[q] = rr[q] > 0;
    s.iters[q] = 0;
}

// blocks per vector of the reductions, from the length alone: a count that fell with k (two to eight
// blocks per SM over all k vectors) made a vector's sum depend on its neighbours, and at k = 64
// each thread added thousands of terms in sequence
inline int red_blocks(int64_t nr)
{
    const int64_t b = nr / 2048;
    return b < 1 ? 1 : b > QS_RED_BLOCKS ? QS_RED_BLOCKS : (int)b;
}

// blocks per vector of the streaming updates: two to eight per SM over the k vectors
inline int stream_blocks(int64_t nr, int k)
{
    const int64_t b = red_blocks(nr), top = 1216 / k;
    return (int)(b < top ? b : top);
}

inline int grid_for(int64_t n, int per = 256)
{
    int64_t b = (n + per - 1) / per;
    return (int)(b < 1216 ? (b < 1 ? 1 : b) : 1216);
}

}  // namespace

template <typename R>
cudaError_t qs_norm2(const R *v, int k, int64_t nr, double *part, double *out, cudaStream_t st)
{
    const int nb = red_blocks(nr);
    norm2_part<R><<<dim3(nb, k), 256, 0, st>>>(v, nr, part);
    finalize_sum<<<k, 256, 0, st>>>(part, nb, 1, out);
    qs_note_launches(2);
    return cudaGetLastError();
}
template cudaError_t qs_norm2<float>(const float *, int, int64_t, double *, double *, cudaStream_t);
template cudaError_t qs_norm2<double>(const double *, int, int64_t, double *, double *, cudaStream_t);

template <typename R>
cudaError_t qs_resid2(const R *a, const R *b, const double *theta, int k, int64_t nr,
                      double *part, double *out, cudaStream_t st)
{
    const int nb = red_blocks(nr);
    resid_part<R><<<dim3(nb, k), 256, 0, st>>>(a, b, theta, nr, part);
    finalize_sum<<<k, 256, 0, st>>>(part, nb, 1, out);
    qs_note_launches(2);
    return cudaGetLastError();
}
template cudaError_t qs_resid2<double>(const double *, const double *, const double *, int, int64_t, double *,
                                       double *, cudaStream_t);
template cudaError_t qs_resid2<float>(const float *, const float *, const double *, int, int64_t, double *, double *,
                                      cudaStream_t);

template <bool LOWP, typename TIn>
static cudaError_t gram_launch(const TIn *A, int ka, const TIn *B, int kb, int64_t nc, double *part, double2 *G,
                               cudaStream_t st)
{
    if (ka < 1 || kb < 1 || ka > 64 || kb > 64) return cudaErrorInvalidValue;
    const int herm = A == B && ka == kb;
    const int tn = (ka + 3) / 4, ntile = herm ? tn * (tn + 1) / 2 : tn * ((kb + 3) / 4);
    const size_t stage = (size_t)GE * ((herm ? ka : ka + kb) + 1) * (LOWP ? sizeof(float2) : sizeof(double2));
    const size_t red = (size_t)ntile * 32 * sizeof(double);
    const size_t sm = stage > red ? stage : red;
    static std::once_flag attr;
    std::call_once(attr, [] {
        cudaFuncSetAttribute(gram_tile_kernel<LOWP, TIn>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024);
    });
    const int64_t nch = (nc + GE - 1) / GE;
    const int nb = (int)(nch < QS_RED_BLOCKS / 2 ? nch : QS_RED_BLOCKS / 2), n = 2 * ka * kb;   // two blocks per SM
    gram_tile_kernel<LOWP, TIn><<<nb, 256, sm, st>>>(A, ka, B, kb, nc, part, herm);
    gram_sum_kernel<<<(n + 31) / 32, 256, 0, st>>>(part, nb, n, kb, herm, reinterpret_cast<double *>(G));
    qs_note_launches(2);
    return cudaGetLastError();
}

cudaError_t qs_gram(const double *A, int ka, const double *B, int kb, int64_t nr, double *part,
                    double2 *G, cudaStream_t st, int lowp)
{
    const double2 *a = (const double2 *)A, *b = (const double2 *)B;
    return lowp ? gram_launch<true, double2>(a, ka, b, kb, nr / 2, part, G, st)
                : gram_launch<false, double2>(a, ka, b, kb, nr / 2, part, G, st);
}

cudaError_t qs_rotate(const double *W, int ka, const double2 *C, int kc, int64_t nr, double *V, cudaStream_t st,
                      int lowp, int upper)
{
    if (ka < 1 || kc < 1 || ka > 64 || kc > 64) return cudaErrorInvalidValue;
    int64_t nc = nr / 2;
    size_t sm = (size_t)ka * kc * (lowp ? sizeof(float2) : sizeof(double2));
    static std::once_flag attr;
    std::call_once(attr, [] {
        cudaFuncSetAttribute(rotate_tile_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 64 * 16);
        cudaFuncSetAttribute(rotate_tile_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 64 * 64 * 16);
    });
    int64_t blocks = (nc + 256 * RE - 1) / (256 * RE);
    int nb = (int)(blocks < 4 * 152 ? blocks : 4 * 152);
    if (lowp) rotate_tile_kernel<true><<<nb, 256, sm, st>>>((const double2 *)W, ka, C, kc, nc, (double2 *)V, upper);
    else rotate_tile_kernel<false><<<nb, 256, sm, st>>>((const double2 *)W, ka, C, kc, nc, (double2 *)V, upper);
    qs_note_launches(1);
    return cudaGetLastError();
}

// the same contractions on FP32 blocks (products and per-chunk sums in FP32)
cudaError_t qs_gram32(const float *A, int ka, const float *B, int kb, int64_t nr, double *part, double2 *G,
                      cudaStream_t st)
{
    return gram_launch<true, float2>((const float2 *)A, ka, (const float2 *)B, kb, nr / 2, part, G, st);
}

cudaError_t qs_rotate32(const float *W, int ka, const double2 *C, int kc, int64_t nr, float *V, cudaStream_t st,
                        int upper)
{
    if (ka < 1 || kc < 1 || ka > 64 || kc > 64) return cudaErrorInvalidValue;
    int64_t nc = nr / 2;
    size_t sm = (size_t)ka * kc * sizeof(float2);
    static std::once_flag attr;
    std::call_once(attr, [] {
        cudaFuncSetAttribute(rotate_tile_kernel<true, float2, float2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             64 * 64 * 8);
    });
    int64_t blocks = (nc + 256 * RE - 1) / (256 * RE);
    int nb = (int)(blocks < 4 * 152 ? blocks : 4 * 152);
    rotate_tile_kernel<true, float2, float2><<<nb, 256, sm, st>>>((const float2 *)W, ka, C, kc, nc, (float2 *)V, upper);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_d2f(const double *x, float *y, const double *scale, int k, int64_t nr, cudaStream_t st)
{
    dim3 g(grid_for(nr) / k + 1, k);
    d2f_kernel<<<g, 256, 0, st>>>(x, y, scale, nr);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_f2d(const float *x, double *y, int k, int64_t nr, cudaStream_t st)
{
    dim3 g(grid_for(nr) / k + 1, k);
    f2d_kernel<<<g, 256, 0, st>>>(x, y, nr);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_axpy_f2d(double *x, const float *e, const double *coef, int k, int64_t nr, cudaStream_t st)
{
    dim3 g(grid_for(nr) / k + 1, k);
    axpy_f2d_kernel<<<g, 256, 0, st>>>(x, e, coef, nr);
    qs_note_launches(1);
    return cudaGetLastError();
}

template <typename R>
cudaError_t qs_scale_cols(R *x, const double *scale, int k, int64_t nr, cudaStream_t st)
{
    dim3 g(grid_for(nr) / k + 1, k);
    scale_cols_kernel<R><<<g, 256, 0, st>>>(x, scale, nr);
    qs_note_launches(1);
    return cudaGetLastError();
}
template cudaError_t qs_scale_cols<double>(double *, const double *, int, int64_t, cudaStream_t);
template cudaError_t qs_scale_cols<float>(float *, const double *, int, int64_t, cudaStream_t);

cudaError_t qs_scaled_copy(double *x, const double *b, const double *coef, int k, int64_t nr, cudaStream_t st)
{
    dim3 g(grid_for(nr) / k + 1, k);
    scaled_copy_kernel<<<g, 256, 0, st>>>(x, b, coef, nr);
    qs_note_launches(1);
    return cudaGetLastError();
}

template <typename R>
cudaError_t qs_cheb_step(R *ynew, const R *ay, const R *y, const R *x, double c, double s1, double s2,
                         int64_t n, cudaStream_t st)
{
    cheb_kernel<R><<<grid_for(n), 256, 0, st>>>(ynew, ay, y, x, (R)c, (R)s1, (R)s2, n);
    qs_note_launches(1);
    return cudaGetLastError();
}
template cudaError_t qs_cheb_step<float>(float *, const float *, const float *, const float *, double, double, double, int64_t, cudaStream_t);
template cudaError_t qs_cheb_step<double>(double *, const double *, const double *, const double *, double, double, double, int64_t, cudaStream_t);

template <typename R>
cudaError_t qs_axpby(double a, const R *x, double b, R *y, int64_t n, cudaStream_t st)
{
    axpby_kernel<R><<<grid_for(n), 256, 0, st>>>((R)a, x, (R)b, y, n);
    qs_note_launches(1);
    return cudaGetLastError();
}
template cudaError_t qs_axpby<float>(double, const float *, double, float *, int64_t, cudaStream_t);
template cudaError_t qs_axpby<double>(double, const double *, double, double *, int64_t, cudaStream_t);

cudaError_t qs_fill_gauss(double *x, int64_t n, uint64_t seed, cudaStream_t st)
{
    gauss_kernel<<<grid_for(n), 256, 0, st>>>(x, n, seed);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_map_scalars(const double *in, double *out, int k, int mode, cudaStream_t st)
{
    map_scalars_kernel<<<1, 64, 0, st>>>(in, out, k, mode);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_cg_alpha(const CgScalars &s, int k, const double *part, int nb, cudaStream_t st)
{
    cg_alpha_kernel<<<k, 256, 0, st>>>(s, part, nb);
    qs_note_launches(1);
    return cudaGetLastError();
}

cudaError_t qs_cg_beta_xp(float *x, float *p, const float *r, const CgScalars &s, double tol2, int k, int64_t nr,
                          const double *part, int nb, cudaStream_t st)
{
    cg_beta_kernel<<<k, 256, 0, st>>>(s, part, nb, tol2);
    cg_xp_kernel<<<dim3(stream_blocks(nr, k), k), 256, 0, st>>>((float4 *)x, (float4 *)p, (const float4 *)r, s, nr / 4);
    qs_note_launches(2);
    return cudaGetLastError();
}

cudaError_t qs_cg_init(CgScalars s, const double *rr, int k, cudaStream_t st)
{
    cg_init_kernel<<<1, 64, 0, st>>>(s, rr, k);
    qs_note_launches(1);
    return cudaGetLastError();
}
