// Device code of the operator with two threads per site (Sec. 2 operator on the C*-doubled
// lattice): the FP64 operator (dslash.cu), the even-odd one (evenodd.cu) and, with FP32
// arithmetic, the operator on small lattices (dslash32.cu).
//
// Two threads per site: lanes l and l + 16 of a warp take spin q = 0 and 1 of the half spinors.
// (1 -+ g_mu) has rank 2: in the chiral basis g_mu = [[0, e_mu], [e_mu^+, 0]] (e_0 = -1,
// e_k = -i s_k), so (1 - g_mu) psi = (h, -e_mu^+ h), h = psi_up - e_mu psi_dn, and
// (1 + g_mu) psi = (h, +e_mu^+ h), h = psi_up + e_mu psi_dn; each e_mu has one entry per row,
// so spin q of h needs spin q and one lower spin of the neighbour, and the product with the
// link feeds spin q and that lower spin of the result.  Thread q keeps the sums of spin q, of
// spin 2 + q and of spin 3 - q; the last one is its partner's and changes hands once, by a
// shuffle.
//
// What bounds it in FP64: GB300's FP64 pipe issues 0.5 T lane instructions/s (measured, multiply-add
// or add alike), about 1/70 of the FP32 rate, so the only thing that counts is the number of
// FP64 instructions.  A complex multiply-add is four fused ones, conjugations and signs are
// integer operations on the sign bit, the links are stored times -1/2, and nothing is added
// to zero: 1164 per site (426 + 156 per thread), against 1650 before: 16^3 x 32, 32 vectors,
// 27.2 -> 16.1 ms.
#pragma once
#include "dslash.cuh"
#include "stencil.cuh"

__device__ __forceinline__ double qs_flip(double x, unsigned mask)   // mask 0x80000000: -x, 0: x
{
    return __hiloint2double(__double2hiint(x) ^ (int)mask, __double2loint(x));
}
__device__ __forceinline__ float qs_flip(float x, unsigned mask) { return __uint_as_float(__float_as_uint(x) ^ mask); }
__device__ __forceinline__ double2 qs_c2(double x, double y) { return make_double2(x, y); }
__device__ __forceinline__ float2 qs_c2(float x, float y) { return make_float2(x, y); }
// c + a b
template <typename V2>
__device__ __forceinline__ V2 qs_cfma(V2 a, V2 b, V2 c)
{
    return qs_c2(fma(-a.y, b.y, fma(a.x, b.x, c.x)), fma(a.y, b.x, fma(a.x, b.y, c.y)));
}
template <typename V2>
__device__ __forceinline__ V2 qs_cmul(V2 a, V2 b)
{
    return qs_c2(fma(-a.y, b.y, a.x * b.x), fma(a.y, b.x, a.x * b.y));
}

// FP64 vectors: the three colours of one spin of a site, and the FP64 SW blocks
template <class AT>
struct Mem64 {
    typedef double R;
    typedef double2 V2;
    __device__ static void ld3(const double2 *__restrict__ in, int s, int spin, double2 v[3])
    {
#pragma unroll
        for (int i = 0; i < 3; ++i) v[i] = __ldg(in + AT::at(s, 3 * spin + i));
    }
};

// spinor access by doubled site and component.  Canonical [site][12]; site-tiled
// [site / 16][12][site % 16]; and tiled over the sites of one parity, whose index is
// site / 2 (a row of 2L sites holds L of each parity).
struct At64Canon : Mem64<At64Canon> {
    __device__ static int64_t at(int s, int c) { return (int64_t)s * 12 + c; }
};
struct At64Tiled : Mem64<At64Tiled> {
    __device__ static int64_t at(int s, int c) { return ((int64_t)(s >> 4) * 12 + c) * 16 + (s & 15); }
};
struct At64Half : Mem64<At64Half> {
    __device__ static int64_t at(int s, int c) { return At64Tiled::at(s >> 1, c); }
};

struct Lane64 {
    Site c;         // the thread's site
    int q;          // its spin
    unsigned mir;   // 0x80000000 on the mirror half, else 0
    int t;          // +1 for q = 0, -1 for q = 1
};

__device__ __forceinline__ Lane64 qs_lane64(const Geom &g, int s)
{
    Lane64 ln;
    ln.c = site_of(g, s);
    ln.q = (threadIdx.x >> 4) & 1;
    ln.mir = ln.c.x >= g.L ? 0x80000000u : 0u;
    ln.t = ln.q ? -1 : 1;
    return ln;
}

// one hop: up, same (spin 2 + q), cross (spin 3 - q) += or, where the flag says so, =
template <int MU, int STEP, class AT, bool FIRST_UP, bool FIRST_LOW>
__device__ __forceinline__ void qs_hop64(const Geom &g, const typename AT::V2 *__restrict__ links,
                                         const typename AT::V2 *__restrict__ in, const Lane64 &ln, typename AT::V2 up[3],
                                         typename AT::V2 same[3], typename AT::V2 cross[3])
{
    constexpr bool FW = STEP > 0;
    typedef typename AT::R R;
    typedef typename AT::V2 V2;
    int sg;
    const Nb n = nbr_of<MU, STEP>(g, ln.c, &sg);
    const int lo = (MU == 0 || MU == 3) ? 2 + ln.q : 3 - ln.q;
    V2 a[3], b[3], U[9];
    AT::ld3(in, n.s, ln.q, a);
    AT::ld3(in, n.s, lo, b);
    const V2 *lk = links + (int64_t)(MU * 9) * g.Vphys + (FW ? ln.c.p : n.p);
    const unsigned cj = FW ? ln.mir : (n.mir ? 0u : 0x80000000u);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        U[k] = __ldg(lk + (int64_t)k * g.Vphys);
        U[k].y = qs_flip(U[k].y, cj);
    }
    const R f = (R)(FW ? ln.t : -ln.t);
    V2 h[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (MU == 0) h[i] = FW ? qs_c2(a[i].x + b[i].x, a[i].y + b[i].y) : qs_c2(a[i].x - b[i].x, a[i].y - b[i].y);
        else if (MU == 1) h[i] = FW ? qs_c2(a[i].x - b[i].y, a[i].y + b[i].x) : qs_c2(a[i].x + b[i].y, a[i].y - b[i].x);
        else if (MU == 2) h[i] = qs_c2(fma(f, b[i].x, a[i].x), fma(f, b[i].y, a[i].y));
        else h[i] = qs_c2(fma(-f, b[i].y, a[i].x), fma(f, b[i].x, a[i].y));
        if (MU == 0) {
            const unsigned neg = sg < 0 ? 0x80000000u : 0u;   // antiperiodic time
            h[i].x = qs_flip(h[i].x, neg);
            h[i].y = qs_flip(h[i].y, neg);
        }
    }
    V2 *low = (MU == 0 || MU == 3) ? same : cross;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        V2 x;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const V2 u = FW ? U[i * 3 + j] : U[j * 3 + i];
            x = j == 0 ? qs_cmul(u, h[j]) : qs_cfma(u, h[j], x);
        }
        if (FIRST_UP) up[i] = x;
        else up[i] = qs_c2(up[i].x + x.x, up[i].y + x.y);
        V2 l = low[i];
        if (MU == 0) {
            if (FIRST_LOW) l = FW ? x : qs_c2(-x.x, -x.y);
            else l = FW ? qs_c2(l.x + x.x, l.y + x.y) : qs_c2(l.x - x.x, l.y - x.y);
        } else if (MU == 1) {
            if (FIRST_LOW) l = FW ? qs_c2(x.y, -x.x) : qs_c2(-x.y, x.x);
            else l = FW ? qs_c2(l.x + x.y, l.y - x.x) : qs_c2(l.x - x.y, l.y + x.x);
        } else if (MU == 2) {
            l = qs_c2(fma(f, x.x, l.x), fma(f, x.y, l.y));
        } else {
            l = qs_c2(fma(f, x.y, l.x), fma(-f, x.x, l.y));
        }
        low[i] = l;
    }
}

// the sum of all eight hops: up and low are spins q and 2 + q of it.  Every lane of the warp
// must call it.
template <class AT>
__device__ __forceinline__ void qs_hops64(const Geom &g, const typename AT::V2 *__restrict__ links,
                                          const typename AT::V2 *__restrict__ in, const Lane64 &ln,
                                          typename AT::V2 up[3], typename AT::V2 low[3])
{
    typename AT::V2 cross[3];
    qs_hop64<0, +1, AT, true, true>(g, links, in, ln, up, low, cross);
    qs_hop64<0, -1, AT, false, false>(g, links, in, ln, up, low, cross);
    qs_hop64<1, +1, AT, false, true>(g, links, in, ln, up, low, cross);
    qs_hop64<1, -1, AT, false, false>(g, links, in, ln, up, low, cross);
    qs_hop64<2, +1, AT, false, false>(g, links, in, ln, up, low, cross);
    qs_hop64<2, -1, AT, false, false>(g, links, in, ln, up, low, cross);
    qs_hop64<3, +1, AT, false, false>(g, links, in, ln, up, low, cross);
    qs_hop64<3, -1, AT, false, false>(g, links, in, ln, up, low, cross);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        low[i].x += __shfl_xor_sync(0xffffffffu, cross[i].x, 16);
        low[i].y += __shfl_xor_sync(0xffffffffu, cross[i].y, 16);
    }
}

// the SW blocks of one physical site: FP64 [2][36][Vphys] reals, FP32 [2][18][Vphys] pairs
struct SwF64 {
    const double *c;
    int64_t V;
    __device__ SwF64 block(int b) const { return {c + (int64_t)b * 36 * V, V}; }
    __device__ double2 off(int k) const { return make_double2(__ldg(c + (int64_t)(6 + 2 * k) * V), __ldg(c + (int64_t)(7 + 2 * k) * V)); }
    __device__ double diag(int i) const { return __ldg(c + (int64_t)i * V); }
};
struct SwF32 {
    const float2 *c;
    int64_t V;
    __device__ SwF32 block(int b) const { return {c + (int64_t)b * 18 * V, V}; }
    __device__ float2 off(int k) const { return __ldg(c + (int64_t)(3 + k) * V); }
    __device__ float diag(int i) const { return __ldg(reinterpret_cast<const float *>(c + (int64_t)(i >> 1) * V) + (i & 1)); }
};

// rows of spin q of A v for one chiral block b, v of both spins of the block: own (spin q)
// and oth.  The block is stored as 6 real diagonals and 15 strict-lower complex entries; with
// hq = q on the physical site and 1 - q on the mirror (whose block is S conj(A) S, so that
// element (i, j) is t_i t_j conj(A[i'][j']), i' in the other spin half, t = (+, -)) the thread
// needs the Hermitian 3 x 3 part of half hq and the 3 x 3 part between the halves.
// SW is the storage of the blocks (SwF64 or SwF32).
template <class SW, typename V2>
__device__ __forceinline__ void qs_sw64(const SW &sw, const Lane64 &ln, const V2 own[3], const V2 oth[3], V2 out[3])
{
    const int hq = ln.q ^ (ln.mir ? 1 : 0);
    auto ld = [&](int k) { return sw.off(k); };
    V2 s[3];   // (1, 0), (2, 0), (2, 1) of half hq
    s[0] = ld(hq ? 9 : 0);
    s[1] = ld(hq ? 13 : 1);
    s[2] = ld(hq ? 14 : 2);
#pragma unroll
    for (int i = 0; i < 3; ++i) s[i].y = qs_flip(s[i].y, ln.mir);
    auto cj = [](V2 e) { return qs_c2(e.x, -e.y); };
    out[1] = qs_cmul(s[0], own[0]);
    out[0] = qs_cmul(cj(s[0]), own[1]);
    out[2] = qs_cmul(s[1], own[0]);
    out[0] = qs_cfma(cj(s[1]), own[2], out[0]);
    out[2] = qs_cfma(s[2], own[1], out[2]);
    out[1] = qs_cfma(cj(s[2]), own[2], out[1]);
    // between the halves: A[3 + r][c] (hq = 1) or conj(A[3 + c][r]) (hq = 0), times -1 and conjugated on the mirror
    const unsigned fi = hq ? 0u : 0x80000000u;
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const int k1 = qs_tri(3 + r, c), k0 = qs_tri(3 + c, r);
            V2 e = ld(hq ? k1 : k0);
            e.x = qs_flip(e.x, ln.mir);
            e.y = qs_flip(e.y, fi);
            out[r] = qs_cfma(e, oth[c], out[r]);
        }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const auto d = sw.diag(3 * hq + i);
        out[i] = qs_c2(fma(d, own[i].x, out[i].x), fma(d, own[i].y, out[i].y));
    }
}

// up, low += spins q and 2 + q of (dm + A) psi at the thread's site, dm = 4 + m0.  The large term
// dm psi is added last, in one rounding: starting from it, every following sum is rounded at
// its size (relative error against long double 1.8e-16 instead of 1.1e-16 on 4^4 to 6^3 x 4).
template <class AT, class SW>
__device__ __forceinline__ void qs_diag64(const SW &sw0, const typename AT::V2 *__restrict__ in, const Lane64 &ln,
                                          typename AT::R dm, typename AT::V2 up[3], typename AT::V2 low[3])
{
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        typedef typename AT::V2 V2;
        V2 own[3], oth[3], d[3];
        AT::ld3(in, ln.c.s, 2 * b + ln.q, own);
        AT::ld3(in, ln.c.s, 2 * b + 1 - ln.q, oth);
        qs_sw64(sw0.block(b), ln, own, oth, d);
        V2 *o = b ? low : up;
#pragma unroll
        for (int i = 0; i < 3; ++i)
            o[i] = qs_c2(fma(dm, own[i].x, o[i].x + d[i].x), fma(dm, own[i].y, o[i].y + d[i].y));
    }
}
