// The operator D and Q = gamma_5 D with FP32 arithmetic (Sec. 2 operator on the
// C*-doubled lattice, Sec. 3 doublet and Q) for FP32 or 16-bit spinor storage.
//
//   out = (4 + m0) psi + A psi - 1/2 sum_mu [ V (1 - g_mu) psi(x+mu) + V^+ (1 + g_mu) psi(x-mu) ]
//
// Thread map.  One thread computes one right-hand side at a physical site p AND at its
// mirror site p + L e_x.  The mirror's links are the complex conjugates of the same
// words, its SW block is S conj(A) S of the same block, and its neighbours are the
// mirrors of p's neighbours, so every link and SW word that is loaded feeds two sites
// and all conjugations and spin swaps are compile-time (only the backward hops across a
// C* boundary need a sign, which costs nothing in the multiply-adds that use it).
//
// Arithmetic.  The matrix products use the packed FP32 instructions (two multiply-adds per
// instruction): with a link entry u and the pair h = (re, im) of a spinor component,
// a += (u.re, u.re) h and b += (u.im, u.im) h, and the product is a + i b (a - i b for the
// conjugate link), combined once per row.  The links are stored times -1/2.
//
// What bounds it.  16^3 x 32, 16 right-hand sides, FP32: 298 us (406 us with one thread per
// doubled site and unpacked arithmetic), 2.96 TB/s of algorithmic bytes; FP16 storage 308 us
// (409), so not the bytes.  1280 thread instructions per site and right-hand side (2200), of
// which 820 go to the FMA pipe, where a packed instruction with three distinct operands
// takes 3 cycles; the pipe alone needs about 180 us.  The rest is the latency of the neighbour loads at the
// 12 warps per SM that 168 registers allow, so the next spinor and link are requested before
// the current ones are multiplied (hops below: 308 -> 298 us).  Tried and slower: one site
// per thread at 20 to 24 warps per SM (382 us: the links and their broadcasts are no longer
// shared), unpacked multiply-adds (346 us).
//
// Storage.  FP32: the solver's site-tiled layout [site / 16][12][site % 16] float2 or
// the canonical [site][12] float2.  FP16 / BF16: tiles of 16 sites, 12 x 16 half2 (or
// bf162) components followed by 16 FP32 scales (832 B per tile); a site's 24 reals are
// stored divided by the largest of their magnitudes, which is its scale.  Arithmetic
// is FP32 throughout.
//
// Epilogue.  PLAIN: out = D in or Q in.  CHEB: one step of the scaled Chebyshev
// recurrence of the filter, out = s1 (Q in - c y) - s2 x, with y, x in the same
// storage (saves a separate pass over four vectors).  NORM: out = Q in and each warp's share of
// |out|^2.  RESID: out = y - alpha Q in (y may be out) and the shares of |out|^2; with these two a
// CG iteration never writes Q^2 p and reads neither it nor Q p for its sums.
#include "qs_internal.cuh"
#include "dslash.cuh"
#include "stencil.cuh"

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <mutex>

namespace {

typedef float2 cf;

__device__ __forceinline__ cf cadd(cf a, cf b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ cf csub(cf a, cf b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ cf cneg(cf a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ cf cmi(cf a) { return make_float2(-a.y, a.x); }   // i a
// packed FP32: both halves at once
__device__ __forceinline__ cf dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ cf add2(cf a, cf b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ cf mul2(cf a, cf b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ cf fma2(cf a, cf b, cf c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ cf sub2(cf a, cf b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// ---- storage formats ------------------------------------------------------
// loads that stay where they are written, so that the next neighbour's words are in flight
// while the current one is multiplied
__device__ __forceinline__ cf ldv(const cf *p)
{
    cf r;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}
__device__ __forceinline__ float4 ldv(const float4 *p)
{
    float4 r;
    asm volatile("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w) : "l"(p));
    return r;
}
__device__ __forceinline__ unsigned ldv(const unsigned *p)
{
    unsigned r;
    asm volatile("ld.global.nc.u32 %0, [%1];" : "=r"(r) : "l"(p));
    return r;
}
__device__ __forceinline__ float ldv(const float *p)
{
    float r;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(r) : "l"(p));
    return r;
}

struct StF32Tiled {
    static constexpr int64_t kBytesPerSite = 96;
    static constexpr bool kScaled = false;
    struct Raw { cf v[12]; };
    __device__ static void fetch(const char *__restrict__ base, int s, Raw &r)
    {
        const cf *b = reinterpret_cast<const cf *>(base) + ((int64_t)(s >> 4) * 12) * 16 + (s & 15);
#pragma unroll
        for (int c = 0; c < 12; ++c) r.v[c] = ldv(b + c * 16);
    }
    __device__ static void open(const Raw &r, cf v[12])
    {
#pragma unroll
        for (int c = 0; c < 12; ++c) v[c] = r.v[c];
    }
    __device__ static void ld(const char *__restrict__ base, int s, cf v[12])
    {
        const cf *b = reinterpret_cast<const cf *>(base) + ((int64_t)(s >> 4) * 12) * 16 + (s & 15);
#pragma unroll
        for (int c = 0; c < 12; ++c) v[c] = __ldg(b + c * 16);
    }
    // the 6 components of chiral block `blk` (spins 2 blk, 2 blk + 1)
    __device__ static void ld6(const char *__restrict__ base, int s, int blk, cf v[6])
    {
        const cf *b = reinterpret_cast<const cf *>(base) + ((int64_t)(s >> 4) * 12 + 6 * blk) * 16 + (s & 15);
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c] = __ldg(b + c * 16);
    }
    __device__ static void st(char *__restrict__ base, int s, const cf v[12])
    {
        cf *b = reinterpret_cast<cf *>(base) + ((int64_t)(s >> 4) * 12) * 16 + (s & 15);
#pragma unroll
        for (int c = 0; c < 12; ++c) b[c * 16] = v[c];
    }
};

struct StF32Canon {
    static constexpr int64_t kBytesPerSite = 96;
    static constexpr bool kScaled = false;
    struct Raw { float4 v[6]; };
    __device__ static void fetch(const char *__restrict__ base, int s, Raw &r)
    {
        const float4 *q = reinterpret_cast<const float4 *>(base) + (int64_t)s * 6;
#pragma unroll
        for (int i = 0; i < 6; ++i) r.v[i] = ldv(q + i);
    }
    __device__ static void open(const Raw &r, cf v[12])
    {
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            v[2 * i] = make_float2(r.v[i].x, r.v[i].y);
            v[2 * i + 1] = make_float2(r.v[i].z, r.v[i].w);
        }
    }
    __device__ static void ld(const char *__restrict__ base, int s, cf v[12])
    {
        const float4 *q = reinterpret_cast<const float4 *>(base) + (int64_t)s * 6;
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            float4 a = __ldg(q + i);
            v[2 * i] = make_float2(a.x, a.y);
            v[2 * i + 1] = make_float2(a.z, a.w);
        }
    }
    __device__ static void ld6(const char *__restrict__ base, int s, int blk, cf v[6])
    {
        const float4 *q = reinterpret_cast<const float4 *>(base) + (int64_t)s * 6 + 3 * blk;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float4 a = __ldg(q + i);
            v[2 * i] = make_float2(a.x, a.y);
            v[2 * i + 1] = make_float2(a.z, a.w);
        }
    }
    __device__ static void st(char *__restrict__ base, int s, const cf v[12])
    {
        float4 *q = reinterpret_cast<float4 *>(base) + (int64_t)s * 6;
#pragma unroll
        for (int i = 0; i < 6; ++i) q[i] = make_float4(v[2 * i].x, v[2 * i].y, v[2 * i + 1].x, v[2 * i + 1].y);
    }
};

// 16-bit storage with a per-site FP32 scale: tile = 12 x 16 words of two 16-bit
// reals, then 16 scales.
template <typename H2>
struct StScaled {
    static constexpr int64_t kBytesPerSite = 52;
    static constexpr bool kScaled = true;
    static constexpr int kTile = 832;
    __device__ static float2 cvt(H2 h);
    __device__ static H2 pack(float a, float b);
    // the stored (site-normalised) values and the site's scale
    struct Raw { unsigned w[12]; float sc; };
    __device__ static void fetch(const char *__restrict__ base, int s, Raw &r)
    {
        const char *t = base + (int64_t)(s >> 4) * kTile;
        const unsigned *w = reinterpret_cast<const unsigned *>(t) + (s & 15);
        r.sc = ldv(reinterpret_cast<const float *>(t + 768) + (s & 15));
#pragma unroll
        for (int c = 0; c < 12; ++c) r.w[c] = ldv(w + c * 16);
    }
    __device__ static void open(const Raw &r, cf v[12])
    {
#pragma unroll
        for (int c = 0; c < 12; ++c) v[c] = cvt(*reinterpret_cast<const H2 *>(&r.w[c]));
    }
    __device__ static void ld(const char *__restrict__ base, int s, cf v[12])
    {
        const char *t = base + (int64_t)(s >> 4) * kTile;
        const unsigned *w = reinterpret_cast<const unsigned *>(t) + (s & 15);
        const float sc = __ldg(reinterpret_cast<const float *>(t + 768) + (s & 15));
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            unsigned u = __ldg(w + c * 16);
            H2 h = *reinterpret_cast<H2 *>(&u);
            float2 f = cvt(h);
            v[c] = make_float2(f.x * sc, f.y * sc);
        }
    }
    __device__ static void ld6(const char *__restrict__ base, int s, int blk, cf v[6])
    {
        const char *t = base + (int64_t)(s >> 4) * kTile;
        const unsigned *w = reinterpret_cast<const unsigned *>(t) + 96 * blk + (s & 15);
        const float sc = __ldg(reinterpret_cast<const float *>(t + 768) + (s & 15));
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            unsigned u = __ldg(w + c * 16);
            H2 h = *reinterpret_cast<H2 *>(&u);
            v[c] = mul2(dup(sc), cvt(h));
        }
    }
    __device__ static void st(char *__restrict__ base, int s, const cf v[12])
    {
        char *t = base + (int64_t)(s >> 4) * kTile;
        float m = 0.f;
#pragma unroll
        for (int c = 0; c < 12; ++c) m = fmaxf(m, fmaxf(fabsf(v[c].x), fabsf(v[c].y)));
        const float inv = m > 0.f ? 1.0f / m : 0.f;
        unsigned *w = reinterpret_cast<unsigned *>(t) + (s & 15);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            H2 h = pack(v[c].x * inv, v[c].y * inv);
            w[c * 16] = *reinterpret_cast<unsigned *>(&h);
        }
        reinterpret_cast<float *>(t + 768)[s & 15] = m;
    }
};
template <> __device__ float2 StScaled<__half2>::cvt(__half2 h) { return __half22float2(h); }
template <> __device__ __half2 StScaled<__half2>::pack(float a, float b) { return __floats2half2_rn(a, b); }
template <> __device__ float2 StScaled<__nv_bfloat162>::cvt(__nv_bfloat162 h) { return __bfloat1622float2(h); }
template <> __device__ __nv_bfloat162 StScaled<__nv_bfloat162>::pack(float a, float b) { return __floats2bfloat162_rn(a, b); }

typedef StScaled<__half2> StF16;
typedef StScaled<__nv_bfloat162> StBF16;

// ---- spin projection / reconstruction (chiral basis, see dslash.cu) ---------
// half spinor h for direction MU, forward (FW: 1 - g_mu) or backward (1 + g_mu)
template <int MU, bool FW>
__device__ __forceinline__ void project(const cf v[12], cf h[2][3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const cf p0 = v[c], p1 = v[3 + c], p2 = v[6 + c], p3 = v[9 + c];
        if (MU == 0) {
            h[0][c] = FW ? add2(p0, p2) : sub2(p0, p2);
            h[1][c] = FW ? add2(p1, p3) : sub2(p1, p3);
        } else if (MU == 1) {
            h[0][c] = FW ? cadd(p0, cmi(p3)) : csub(p0, cmi(p3));
            h[1][c] = FW ? cadd(p1, cmi(p2)) : csub(p1, cmi(p2));
        } else if (MU == 2) {
            h[0][c] = FW ? add2(p0, p3) : sub2(p0, p3);
            h[1][c] = FW ? sub2(p1, p2) : add2(p1, p2);
        } else {
            h[0][c] = FW ? cadd(p0, cmi(p2)) : csub(p0, cmi(p2));
            h[1][c] = FW ? csub(p1, cmi(p3)) : cadd(p1, cmi(p3));
        }
    }
}

// acc += row (q, c) of (x, lower(x)), lower = -+ e_mu^+ x
template <int MU, bool FW, int Q>
__device__ __forceinline__ void reconstruct(cf acc[12], int c, cf x)
{
    acc[3 * Q + c] = add2(acc[3 * Q + c], x);
    constexpr int LO = (MU == 0 || MU == 3) ? 6 + 3 * Q : 9 - 3 * Q;   // lower spin fed by x
    cf &l = acc[LO + c];
    if (MU == 0) l = FW ? add2(l, x) : sub2(l, x);
    else if (MU == 2) l = (FW == (Q == 0)) ? add2(l, x) : sub2(l, x);
    else if (MU == 1) l = FW ? csub(l, cmi(x)) : cadd(l, cmi(x));
    else l = (FW == (Q == 0)) ? csub(l, cmi(x)) : cadd(l, cmi(x));
}

__host__ __device__ constexpr int tri(int i, int j) { return i * (i - 1) / 2 + j; }

// real diagonal I of a packed SW block (pairs: 3 of real diagonals, 15 of strict-lower
// complex entries)
__device__ __forceinline__ float sw_diag(const cf P[18], int i) { return (i & 1) ? P[i / 2].y : P[i / 2].x; }

// acc = (dm + A) v for one chiral block of the physical site (MIR = false), or with the mirror
// site's block S conj(A) S: element (i, j) of it is t_i t_j conj(A[i'][j']), i' = i +- 3 the
// other spin half and t = (+, -) on the two halves.
template <bool MIR>
__device__ __forceinline__ void sw_block(const cf P[18], float dm, const cf v[6], cf acc[6])
{
    cf w[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) w[j] = !MIR ? v[j] : (j < 3 ? cneg(v[j + 3]) : v[j - 3]);
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        cf a = mul2(dup(dm + sw_diag(P, i)), w[i]);
        cf lo = make_float2(0.f, 0.f), up = lo;   // sums of im(A_ij) w_j over j < i, im(A_ji) w_j over j > i
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j == i) continue;
            const cf e = j < i ? P[3 + tri(i, j)] : P[3 + tri(j, i)];
            a = fma2(dup(e.x), w[j], a);
            if (j < i) lo = j == 0 ? mul2(dup(e.y), w[j]) : fma2(dup(e.y), w[j], lo);
            else up = j == i + 1 ? mul2(dup(e.y), w[j]) : fma2(dup(e.y), w[j], up);
        }
        const cf d = i == 0 ? cneg(up) : i == 5 ? lo : sub2(lo, up);   // a + i d (physical), a - i d (mirror)
        if (!MIR) acc[i] = make_float2(a.x - d.y, a.y + d.x);
        else if (i < 3) acc[i + 3] = make_float2(-a.x - d.y, d.x - a.y);
        else acc[i - 3] = make_float2(a.x + d.y, a.y - d.x);
    }
}

struct D32 {
    Geom g;
    const cf *links;    // [mu][9][Vphys], times -1/2
    const cf *clov;     // [2][18][Vphys]
    const char *in;     // right-hand side r at in + r * vbytes
    char *out;
    const char *y, *x;  // CHEB epilogue operands
    int64_t vbytes;
    int nrhs, gamma5;
    float c, s1, s2;    // CHEB: out = s1 (Q in - c y) - s2 x
    float dm[QS_MAX_RHS];   // 4 + m0 per right-hand side
    // device-side overrides (for launches replayed from a CUDA graph): if set, (c, s1, s2)
    // are read from coef[0..2] and 4 + m0 of right-hand side r from dmdev[r]
    const float *coef, *dmdev;
    const int *live;    // NORM, RESID: NULL, or flags: right-hand sides with live[r] = 0 are skipped
    const float *alpha; // RESID: per right-hand side
    double *part;       // NORM, RESID: [nrhs][ntile] shares of |out|^2
    int ntile;
};

// acc += upper and lower parts of M h for a neighbour's spinor, M = U (FW, sigma = +1),
// conj(U) (FW, -1), U^+ (backward, -1) or U^T (backward, +1)
template <int MU, bool FW, class S>
__device__ __forceinline__ void hop_apply(const cf U[9], float sigma, float f, bool anti, const typename S::Raw &raw,
                                          cf acc[12])
{
    cf v[12], h[2][3];
    S::open(raw, v);
    project<MU, FW>(v, h);
    if constexpr (S::kScaled) {
        // the site's scale commutes with the projection: apply it to the 6 projected
        // components instead of the 12 loaded ones
        const float sc = MU == 0 ? raw.sc * f : raw.sc;
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < 3; ++i) h[q][i] = mul2(dup(sc), h[q][i]);
    } else if (MU == 0 && anti) {
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int i = 0; i < 3; ++i) h[q][i] = mul2(dup(f), h[q][i]);
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        cf a[2], b[2];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const cf u = FW ? U[i * 3 + j] : U[j * 3 + i];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                a[q] = j == 0 ? mul2(dup(u.x), h[q][j]) : fma2(dup(u.x), h[q][j], a[q]);
                b[q] = j == 0 ? mul2(dup(u.y), h[q][j]) : fma2(dup(u.y), h[q][j], b[q]);
            }
        }
        reconstruct<MU, FW, 0>(acc, i, make_float2(fmaf(-sigma, b[0].y, a[0].x), fmaf(sigma, b[0].x, a[0].y)));
        reconstruct<MU, FW, 1>(acc, i, make_float2(fmaf(-sigma, b[1].y, a[1].x), fmaf(sigma, b[1].x, a[1].y)));
    }
}

// one direction of a physical site and its mirror: the neighbour sites, the link in flight
struct Hop {
    cf U[9];
    int n, nm;      // the neighbours of the site and of its mirror
    float sigma, f;
};

// hop number D: direction D / 2, forward for even D
template <int D>
__device__ __forceinline__ void hop_begin(const D32 &a, const Site &c, Hop &h)
{
    constexpr int MU = D / 2, STEP = D % 2 ? -1 : 1;
    int sg;
    const Nb n = nbr_of<MU, STEP>(a.g, c, &sg);
    const int lp = STEP > 0 ? c.p : n.p;
    const int64_t V = a.g.Vphys;
#pragma unroll
    for (int k = 0; k < 9; ++k) h.U[k] = ldv(a.links + (int64_t)(MU * 9 + k) * V + lp);
    h.sigma = STEP > 0 ? 1.f : (n.mir ? 1.f : -1.f);
    h.f = (float)sg;
    h.n = n.s;
    h.nm = n.mir ? n.s - a.g.L : n.s + a.g.L;
}

// hops D .. 7; `h` and `v` hold hop D's link and the physical site's neighbour, already
// requested.  While one spinor is multiplied the next one is in flight.
template <int D, class S>
__device__ __forceinline__ void hops(const D32 &a, const Site &c, const char *in, Hop &h, typename S::Raw &v,
                                     cf acc[12], cf accm[12])
{
    typename S::Raw w;
    S::fetch(in, h.nm, w);
    hop_apply<D / 2, D % 2 == 0, S>(h.U, h.sigma, h.f, a.g.t_anti, v, acc);
    if constexpr (D < 7) {
        Hop h2;
        hop_begin<D + 1>(a, c, h2);
        S::fetch(in, h2.n, v);
        hop_apply<D / 2, D % 2 == 0, S>(h.U, -h.sigma, h.f, a.g.t_anti, w, accm);
        hops<D + 1, S>(a, c, in, h2, v, acc, accm);
    } else {
        hop_apply<D / 2, D % 2 == 0, S>(h.U, -h.sigma, h.f, a.g.t_anti, w, accm);
    }
}

// |v|^2 of 12 components as an unevaluated sum q + lo: exact squares by fused multiply-adds, their
// sums by two-sum (hi + v v = s + e with s rounded, b = s - hi, e = (v v - b) + (hi - (s - b))).
// A plain FP32 chain of the 24 squares is three to six times further from the 64-bit sum
// on 4^4 to 8^3 x 12 than reductions with one or two squares per thread.
__device__ __forceinline__ cf site_norm2(const cf v[12])
{
    cf q = mul2(v[0], v[0]), lo = fma2(v[0], v[0], cneg(q));
#pragma unroll
    for (int i = 1; i < 12; ++i) {
        const cf s = fma2(v[i], v[i], q), nb = sub2(q, s);   // -b
        lo = add2(lo, add2(fma2(v[i], v[i], nb), sub2(q, add2(s, nb))));
        q = s;
    }
    const float t = q.x + q.y, b = t - q.x;
    return make_float2(t, lo.x + lo.y + ((q.x - (t - b)) + (q.y - b)));
}

// hops D .. 7 of one site only (sg = 1: the physical one, -1: its mirror), the next neighbour's
// spinor and link in flight while the current one is multiplied
template <int D, class S>
__device__ __forceinline__ void hops_one(const D32 &a, const Site &c, const char *in, bool mir, float sg, const Hop &h,
                                         const typename S::Raw &v, cf acc[12])
{
    if constexpr (D < 7) {
        Hop h2;
        typename S::Raw w;
        hop_begin<D + 1>(a, c, h2);
        S::fetch(in, mir ? h2.nm : h2.n, w);
        hop_apply<D / 2, D % 2 == 0, S>(h.U, sg * h.sigma, h.f, a.g.t_anti, v, acc);
        hops_one<D + 1, S>(a, c, in, mir, sg, h2, w, acc);
    } else {
        hop_apply<D / 2, D % 2 == 0, S>(h.U, sg * h.sigma, h.f, a.g.t_anti, v, acc);
    }
}

// the warp's sum of x.x + x.y, kept as a two-sum pair, to *out by lane 0
__device__ __forceinline__ void warp_share(cf x, double *out)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, x.x, o), l2 = __shfl_xor_sync(0xffffffffu, x.y, o);
        const float t = x.x + h2, b = t - x.x;
        x.y += l2 + ((x.x - (t - b)) + (h2 - b));
        x.x = t;
    }
    if ((threadIdx.x & 31) == 0) *out = (double)x.x + (double)x.y;
}

// returns |out|^2 at the site for NORM and RESID (site_norm2)
template <class S, int EPI>
__device__ __forceinline__ cf finish_site(const D32 &a, int64_t off, int s, int r, bool on, cf acc[12])
{
    if (a.gamma5) {
#pragma unroll
        for (int i = 6; i < 12; ++i) acc[i] = cneg(acc[i]);
    }
    if (EPI == QS_EPI_CHEB) {
        cf yv[12], xv[12];
        S::ld(a.y + off, s, yv);
        S::ld(a.x + off, s, xv);
        const float cc = a.coef ? __ldg(a.coef) : a.c;
        const float s1 = a.coef ? __ldg(a.coef + 1) : a.s1;
        const float s2 = a.coef ? __ldg(a.coef + 2) : a.s2;
#pragma unroll
        for (int i = 0; i < 12; ++i)
            acc[i] = fma2(dup(s1), fma2(dup(-cc), yv[i], acc[i]), mul2(dup(-s2), xv[i]));
    }
    if (EPI == QS_EPI_RESID) {
        const float al = a.alpha[r];
        const cf *y = reinterpret_cast<const cf *>(a.y + off) + ((int64_t)(s >> 4) * 12) * 16 + (s & 15);   // tiled FP32
#pragma unroll
        for (int i = 0; i < 12; ++i) acc[i] = fma2(dup(-al), acc[i], y[i * 16]);   // no read-only load: y may be out
    }
    if (EPI < QS_EPI_NORM || on) S::st(a.out + off, s, acc);
    return EPI >= QS_EPI_NORM && on ? site_norm2(acc) : make_float2(0.f, 0.f);
}

// physical site p and its mirror, right-hand side r (one per warp); on = false: nothing is
// stored (NORM and RESID keep whole warps for their sums)
template <class S, int EPI>
__device__ __forceinline__ void site_kernel(const D32 &a, int p, int r, bool on = true)
{
    if (EPI >= QS_EPI_NORM && a.live && !a.live[r]) return;
    const int row = p / a.g.L;
    const Site c = site_of(a.g, p + row * a.g.L);   // x < L: s = row 2L + x, p = row L + x
    const int64_t off = (int64_t)r * a.vbytes;
    const char *in = a.in + off;

    cf acc[12], accm[12];
    {
        // diagonal part (4 + m0 + A) psi, one chiral block at a time
        const float dm = a.dmdev ? __ldg(a.dmdev + r) : a.dm[r];
        const int64_t V = a.g.Vphys;
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            cf P[18], v[6];
#pragma unroll
            for (int q = 0; q < 18; ++q) P[q] = __ldg(a.clov + (int64_t)(b * 18 + q) * V + p);
            S::ld6(in, c.s, b, v);
            sw_block<false>(P, dm, v, acc + 6 * b);
            S::ld6(in, c.s + a.g.L, b, v);
            sw_block<true>(P, dm, v, accm + 6 * b);
        }
    }
    Hop h;
    typename S::Raw v;
    hop_begin<0>(a, c, h);
    S::fetch(in, h.n, v);
    hops<0, S>(a, c, in, h, v, acc, accm);
    const cf n2 = finish_site<S, EPI>(a, off, c.s, r, on, acc);
    const cf m2 = finish_site<S, EPI>(a, off, c.s + a.g.L, r, on, accm);
    if (EPI >= QS_EPI_NORM) {   // two shares per 32 physical sites, the ones that one_kernel leaves
        double *sh = a.part + (int64_t)r * a.ntile + 2 * (p / 32);
        warp_share(n2, sh);
        warp_share(m2, sh + 1);
    }
}

// physical site p (mir = false) or its mirror alone: the same arithmetic as site_kernel's for that
// site, in half the chain of loads and products.  mir is the same in the whole warp.
template <class S, int EPI>
__device__ __forceinline__ void one_kernel(const D32 &a, int p, int r, bool mir, bool on)
{
    if (EPI >= QS_EPI_NORM && a.live && !a.live[r]) return;
    const Site c = site_of(a.g, p + (p / a.g.L) * a.g.L);
    const int s = mir ? c.s + a.g.L : c.s;
    const int64_t off = (int64_t)r * a.vbytes;
    const char *in = a.in + off;
    cf acc[12];
    const float dm = a.dmdev ? __ldg(a.dmdev + r) : a.dm[r];
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        cf P[18], v[6];
#pragma unroll
        for (int q = 0; q < 18; ++q) P[q] = __ldg(a.clov + (int64_t)(b * 18 + q) * a.g.Vphys + p);
        S::ld6(in, s, b, v);
        if (mir) sw_block<true>(P, dm, v, acc + 6 * b);
        else sw_block<false>(P, dm, v, acc + 6 * b);
    }
    Hop h;
    typename S::Raw v;
    hop_begin<0>(a, c, h);
    S::fetch(in, mir ? h.nm : h.n, v);
    hops_one<0, S>(a, c, in, mir, mir ? -1.f : 1.f, h, v, acc);
    const cf n2 = finish_site<S, EPI>(a, off, s, r, on, acc);
    if (EPI >= QS_EPI_NORM) warp_share(n2, a.part + (int64_t)r * a.ntile + 2 * (p / 32) + (mir ? 1 : 0));
}

// A block's NT / 32 warps are WR right-hand sides x (NT / 32 / WR) groups of 32 physical sites;
// it computes `gpb` groups of WR right-hand sides one after the other.
template <class S, int EPI, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) dslash32_kernel(const __grid_constant__ D32 a, unsigned nchunk, int lwr,
                                                            int gpb)
{
    const unsigned tile = blockIdx.x / nchunk, chunk = blockIdx.x % nchunk;
    const int w = threadIdx.x >> 5, wr = 1 << lwr;
    int p = (int)((tile * (NT / 32 >> lwr) + (w >> lwr)) * 32 + (threadIdx.x & 31));
    bool on = p < (int)a.g.Vphys;
    if (EPI >= QS_EPI_NORM) {
        if ((p & ~31) >= (int)a.g.Vphys) return;   // the whole warp
        if (!on) p = (int)a.g.Vphys - 1;           // same warp tile as lane 0
    } else if (!on) {
        return;
    }
    int r = (int)(chunk * gpb) * wr + (w & (wr - 1));
    for (int i = 0; i < gpb && r < a.nrhs; ++i, r += wr) site_kernel<S, EPI>(a, p, r, on);
}

// Problems that fill the SMs a few times at most: a block is 32 physical sites and one right-hand
// side, its first warp on the sites and its second on their mirrors.  A pair thread's chain is about
// 17 k cycles, all the time there is when few warps run: 4^3 x 8, 24 vectors, 8.2 -> 6.2 us back to
// back, even with the pairs at 100 k sites x vectors, slower beyond (12^3 x 24, 8 vectors: 71
// against 61 us).
template <class S, int EPI>
__global__ void __launch_bounds__(64, 8) dslash32_one_kernel(const __grid_constant__ D32 a)
{
    const int r = (int)(blockIdx.x % (unsigned)a.nrhs), p0 = (int)(blockIdx.x / (unsigned)a.nrhs) * 32;
    const int p = p0 + (int)(threadIdx.x & 31);
    const bool on = p < (int)a.g.Vphys;
    if (EPI < QS_EPI_NORM && !on) return;
    one_kernel<S, EPI>(a, on ? p : (int)a.g.Vphys - 1, r, threadIdx.x >= 32, on);
}

template <class S, int EPI>
cudaError_t launch_one(const D32 &a, cudaStream_t st)
{
    dslash32_one_kernel<S, EPI><<<(unsigned)((a.g.Vphys + 31) / 32) * (unsigned)a.nrhs, 64, 0, st>>>(a);
    return cudaGetLastError();
}

// Batched form: work items (lattice i, tile of physical sites, right-hand side) numbered lattice by
// lattice, right-hand sides fastest.  Large batches are persistent: each block takes items
// w = blockIdx.x, blockIdx.x + gridDim.x, ... of 128 sites.  Small ones launch a block per item of 32
// sites, as dslash32_one_kernel.
#define QS_BATCH_TILE 128     // physical sites per work item
#define QS_BATCH_ONE_TILE 32
// Physical sites x right-hand sides up to which a block per 32 sites and its mirrors is the faster
// form, of a batch and of a single launch whose variants are not timed: below it the pair threads do
// not fill the chip, and their chain is the time.  Batches: device time, in a graph: two 4^3 x 3 of one vector, FP32, 5.7 -> 4.1 us and FP16 6.0 -> 4.0; 4^3 x 4, 6^3 x 5
// and 8^3 x 8 of 3, 5 and 2 vectors 7.0 -> 5.2; even at 32 k (two 8^3 x 8 of 4 vectors: 8.1 and 7.9, FP16 7.9
// and 7.8), slower at 49 k (10.7 against 11.4 us).
#define QS_ONE_MAX 32768

struct D32B {
    int n;
    unsigned off[QS_BATCH_MAX + 1];   // first work item of lattice i; off[n] = all items
    D32 item[QS_BATCH_MAX];
};

static_assert(sizeof(D32B) <= 4096, "batched operator arguments exceed the kernel parameter space");

template <class S>
__global__ void __launch_bounds__(128, 3) dslash32_batch_kernel(const __grid_constant__ D32B b)
{
    for (unsigned w = blockIdx.x; w < b.off[b.n]; w += gridDim.x) {
        int i = 0;
#pragma unroll 1
        while (i + 1 < b.n && w >= b.off[i + 1]) ++i;
        const unsigned local = w - b.off[i];
        const int p = (int)(local / (unsigned)b.item[i].nrhs) * QS_BATCH_TILE + (int)threadIdx.x;
        if (p < (int)b.item[i].g.Vphys) site_kernel<S, QS_EPI_PLAIN>(b.item[i], p, (int)(local % (unsigned)b.item[i].nrhs));
    }
}

template <class S>
__global__ void __launch_bounds__(64, 8) dslash32_batch_one_kernel(const __grid_constant__ D32B b)
{
    int i = 0;
#pragma unroll 1
    while (i + 1 < b.n && blockIdx.x >= b.off[i + 1]) ++i;
    const D32 &a = b.item[i];
    const unsigned local = blockIdx.x - b.off[i], nrhs = (unsigned)a.nrhs;
    const int p = (int)(local / nrhs) * 32 + (int)(threadIdx.x & 31);
    if (p < (int)a.g.Vphys) one_kernel<S, QS_EPI_PLAIN>(a, p, (int)(local % nrhs), threadIdx.x >= 32, true);
}

// ---- conversions between tiled storages (per right-hand side and site) -----------
struct StF64Tiled {
    static constexpr int64_t kBytesPerSite = 192;
    __device__ static void ld(const char *__restrict__ base, int s, cf v[12])
    {
        const double2 *b = reinterpret_cast<const double2 *>(base) + ((int64_t)(s >> 4) * 12) * 16 + (s & 15);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            double2 d = b[c * 16];
            v[c] = make_float2((float)d.x, (float)d.y);
        }
    }
    __device__ static void st(char *__restrict__ base, int s, const cf v[12])
    {
        double2 *b = reinterpret_cast<double2 *>(base) + ((int64_t)(s >> 4) * 12) * 16 + (s & 15);
#pragma unroll
        for (int c = 0; c < 12; ++c) b[c * 16] = make_double2((double)v[c].x, (double)v[c].y);
    }
};

template <class SA, class SB>
__global__ void convert_kernel(const char *__restrict__ in, char *__restrict__ out, int64_t Ns, int k)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= Ns * k) return;
    const int r = (int)(i / Ns);
    const int s = (int)(i - (int64_t)r * Ns);
    cf v[12];
    SA::ld(in + (int64_t)r * Ns * SA::kBytesPerSite, s, v);
    SB::st(out + (int64_t)r * Ns * SB::kBytesPerSite, s, v);
}

template <class SA>
cudaError_t convert_from(int to, const void *in, void *out, int64_t Ns, int k, cudaStream_t st)
{
    const unsigned nb = (unsigned)((Ns * k + 255) / 256);
    const char *a = (const char *)in;
    char *b = (char *)out;
    switch (to) {
    case QS_D32_F32_TILED: convert_kernel<SA, StF32Tiled><<<nb, 256, 0, st>>>(a, b, Ns, k); break;
    case QS_D32_F16: convert_kernel<SA, StF16><<<nb, 256, 0, st>>>(a, b, Ns, k); break;
    case QS_D32_BF16: convert_kernel<SA, StBF16><<<nb, 256, 0, st>>>(a, b, Ns, k); break;
    case QS_D32_F64_TILED: convert_kernel<SA, StF64Tiled><<<nb, 256, 0, st>>>(a, b, Ns, k); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// ---- launch ------------------------------------------------------------------
template <class S, int EPI, int NT, int MINB>
cudaError_t launch(const D32 &a, int lwr, int gpb, cudaStream_t st)
{
    const int spb = NT >> lwr, ngroup = (a.nrhs + (1 << lwr) - 1) >> lwr;
    if (gpb > ngroup) gpb = ngroup;
    const unsigned ntile = (unsigned)((a.g.Vphys + spb - 1) / spb);
    const unsigned nchunk = (unsigned)((ngroup + gpb - 1) / gpb);
    dslash32_kernel<S, EPI, NT, MINB><<<ntile * nchunk, NT, 0, st>>>(a, nchunk, lwr, gpb);
    return cudaGetLastError();
}

// variant table: threads per block and blocks per SM (168 registers a thread in all), right-hand
// sides side by side in a block (1 << lwr), groups of them one after the other (gpb).  Right-hand
// sides side by side or in turn read a site's links and SW words from L1 instead of L2, which
// pays from about 16 vectors on a lattice that fills the chip (16^3 x 32, 16 vectors, FP32: 298
// against 308 us); small blocks of one vector spread small problems over the SMs and keep the
// neighbour rows of large ones close (12^3 x 24, 8 vectors: 61 against 63 us; 32^3 x 64, 24
// vectors, FP16: 7.4 against 7.8 ms); the smallest problems take a thread per site.  All variants
// compute a site in the same order, and NORM and RESID leave the same shares of |out|^2 (the 32
// sites of a warp, their mirrors apart), so the choice, which is made by timing, does not show in
// any result.
template <class S, int EPI>
cudaError_t launch_variant(int v, const D32 &a, cudaStream_t st)
{
    switch (v) {
    case 0: return launch<S, EPI, 64, 6>(a, 0, 1, st);
    case 1: return launch<S, EPI, 32, 12>(a, 0, 1, st);
    case 2: return launch<S, EPI, 128, 3>(a, 0, 1, st);
    case 3: return launch<S, EPI, 128, 3>(a, 1, 64, st);
    case 4: return launch<S, EPI, 128, 3>(a, 2, 64, st);
    case 5: return launch_one<S, EPI>(a, st);
    default: return launch<S, EPI, 384, 1>(a, 2, 64, st);
    }
}

template <class S>
cudaError_t launch_storage(int v, int epi, const D32 &a, cudaStream_t st)
{
    switch (epi) {
    case QS_EPI_PLAIN: return launch_variant<S, QS_EPI_PLAIN>(v, a, st);
    case QS_EPI_CHEB: return launch_variant<S, QS_EPI_CHEB>(v, a, st);
    default: return cudaErrorInvalidValue;
    }
}

template <class S>
cudaError_t batch_launch(const D32B &b, bool one, cudaStream_t st)
{
    if (one) {
        dslash32_batch_one_kernel<S><<<b.off[b.n], 64, 0, st>>>(b);
        return cudaGetLastError();
    }
    static int per_sm = 0, nsm = 0;
    static std::once_flag once;
    std::call_once(once, [] {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, dslash32_batch_kernel<S>, 128, 0);
        if (per_sm < 1) per_sm = 1;
        if (nsm < 1) nsm = 1;
    });
    const unsigned total = b.off[b.n];
    const unsigned grid = total < (unsigned)(per_sm * nsm) ? total : (unsigned)(per_sm * nsm);
    dslash32_batch_kernel<S><<<grid, 128, 0, st>>>(b);
    return cudaGetLastError();
}

}  // namespace

cudaError_t qs_d32_batch_launch(const D32BatchItem *items, int n, int storage, int gamma5, cudaStream_t st)
{
    if (n < 1 || n > QS_BATCH_MAX) return cudaErrorInvalidValue;
    D32B b;
    memset(&b, 0, sizeof(b));
    b.n = n;
    int64_t work = 0;
    for (int i = 0; i < n; ++i) work += items[i].g.Vphys * items[i].nrhs;
    const bool one = work <= QS_ONE_MAX;
    const int tile = one ? QS_BATCH_ONE_TILE : QS_BATCH_TILE;
    unsigned off = 0;
    for (int i = 0; i < n; ++i) {
        D32 &a = b.item[i];
        const D32BatchItem &it = items[i];
        a.g = it.g;
        a.links = reinterpret_cast<const cf *>(it.links);
        a.clov = reinterpret_cast<const cf *>(it.clov);
        a.in = (const char *)it.in;
        a.out = (char *)it.out;
        a.y = a.x = nullptr;
        a.vbytes = qs_d32_vec_bytes(storage, it.g.Ns);
        a.nrhs = it.nrhs;
        a.gamma5 = gamma5;
        a.c = a.s1 = a.s2 = 0.f;
        a.coef = a.dmdev = nullptr;
        a.live = nullptr;
        a.alpha = nullptr;
        a.part = nullptr;
        a.ntile = 0;
        for (int r = 0; r < it.nrhs; ++r) a.dm[r] = (float)(4.0 + it.m0[r]);
        b.off[i] = off;
        const double items_i = (double)((it.g.Vphys + tile - 1) / tile) * it.nrhs;
        if (off + items_i > 4e9) return cudaErrorInvalidValue;
        off += (unsigned)items_i;
    }
    b.off[n] = off;
    cudaError_t e;
    switch (storage) {
    case QS_D32_F32_TILED: e = batch_launch<StF32Tiled>(b, one, st); break;
    case QS_D32_F32_CANON: e = batch_launch<StF32Canon>(b, one, st); break;
    case QS_D32_F16: e = batch_launch<StF16>(b, one, st); break;
    case QS_D32_BF16: e = batch_launch<StBF16>(b, one, st); break;
    default: return cudaErrorInvalidValue;
    }
    qs_note_launches(1);
    return e;
}

int64_t qs_d32_ntile(const Geom &g) { return 2 * ((g.Vphys + 31) / 32); }

int qs_d32_nvariants() { return 7; }

// Device time of an application in FP32 and FP16, thread per site against variant 1: 4^3 x 4, one vector,
// 3.8 and 3.9 us against 5.2 and 5.7; 6^3 x 6, 3 vectors, 4.0 and 4.3 against 6.1 and 6.6; 8^3 x 8, 4 vectors,
// 5.3 and 5.3 against 6.7 and 7.0.
int qs_d32_fixed_variant(const Geom &g, int nrhs) { return g.Vphys * nrhs <= QS_ONE_MAX ? 5 : 1; }

int64_t qs_d32_vec_bytes(int storage, int64_t Ns)
{
    return storage == QS_D32_F16 || storage == QS_D32_BF16 ? Ns * 52 : Ns * 96;
}

cudaError_t qs_d32_launch(const D32Call &c, int variant, cudaStream_t st)
{
    D32 a;
    a.g = c.g;
    a.links = reinterpret_cast<const cf *>(c.links);
    a.clov = reinterpret_cast<const cf *>(c.clov);
    a.in = (const char *)c.in;
    a.out = (char *)c.out;
    a.y = (const char *)c.y;
    a.x = (const char *)c.x;
    a.vbytes = qs_d32_vec_bytes(c.storage, c.g.Ns);
    a.nrhs = c.nrhs;
    a.gamma5 = c.gamma5;
    a.c = (float)c.cheb_c;
    a.s1 = (float)c.cheb_s1;
    a.s2 = (float)c.cheb_s2;
    for (int r = 0; r < c.nrhs; ++r) a.dm[r] = c.m0 ? (float)(4.0 + c.m0[r]) : 0.f;
    a.coef = c.coef_dev;
    a.dmdev = c.dm_dev;
    a.live = c.live;
    a.alpha = c.alpha_dev;
    a.part = c.part;
    a.ntile = (int)qs_d32_ntile(c.g);
    switch (c.storage) {
    case QS_D32_F32_TILED:
        if (c.epi == QS_EPI_NORM) return launch_variant<StF32Tiled, QS_EPI_NORM>(variant, a, st);
        if (c.epi == QS_EPI_RESID) return launch_variant<StF32Tiled, QS_EPI_RESID>(variant, a, st);
        return launch_storage<StF32Tiled>(variant, c.epi, a, st);
    case QS_D32_F32_CANON: return launch_storage<StF32Canon>(variant, c.epi, a, st);
    case QS_D32_F16: return launch_storage<StF16>(variant, c.epi, a, st);
    case QS_D32_BF16: return launch_storage<StBF16>(variant, c.epi, a, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t qs_convert_tiled(int from, int to, const void *in, void *out, int64_t Ns, int k, cudaStream_t st)
{
    cudaError_t e;
    switch (from) {
    case QS_D32_F32_TILED: e = convert_from<StF32Tiled>(to, in, out, Ns, k, st); break;
    case QS_D32_F16: e = convert_from<StF16>(to, in, out, Ns, k, st); break;
    case QS_D32_BF16: e = convert_from<StBF16>(to, in, out, Ns, k, st); break;
    case QS_D32_F64_TILED: e = convert_from<StF64Tiled>(to, in, out, Ns, k, st); break;
    default: return cudaErrorInvalidValue;
    }
    qs_note_launches(1);
    return e;
}

cudaError_t qs_q16_from_f64(int storage, const double *in, void *out, int64_t Ns, int k, cudaStream_t st)
{
    return qs_convert_tiled(QS_D32_F64_TILED, storage, in, out, Ns, k, st);
}

cudaError_t qs_f64_from_q16(int storage, const void *in, double *out, int64_t Ns, int k, cudaStream_t st)
{
    return qs_convert_tiled(storage, QS_D32_F64_TILED, in, out, Ns, k, st);
}
