// Device code of the FP64 operator (Sec. 2 operator on the C*-doubled lattice), shared by the
// full operator (dslash.cu) and the even-odd one (evenodd.cu).
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
// What bounds it: GB300's FP64 pipe issues 0.5 T lane instructions/s (measured, multiply-add
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
// c + a b
__device__ __forceinline__ double2 qs_cfma(double2 a, double2 b, double2 c)
{
    return make_double2(fma(-a.y, b.y, fma(a.x, b.x, c.x)), fma(a.y, b.x, fma(a.x, b.y, c.y)));
}
__device__ __forceinline__ double2 qs_cmul(double2 a, double2 b)
{
    return make_double2(fma(-a.y, b.y, a.x * b.x), fma(a.y, b.x, a.x * b.y));
}

// spinor access by doubled site and component.  Canonical [site][12]; site-tiled
// [site / 16][12][site % 16]; and tiled over the sites of one parity, whose index is
// site / 2 (a row of 2L sites holds L of each parity).
struct At64Canon {
    __device__ static int64_t at(int s, int c) { return (int64_t)s * 12 + c; }
};
struct At64Tiled {
    __device__ static int64_t at(int s, int c) { return ((int64_t)(s >> 4) * 12 + c) * 16 + (s & 15); }
};
struct At64Half {
    __device__ static int64_t at(int s, int c) { return At64Tiled::at(s >> 1, c); }
};

struct Lane64 {
    Site c;         // the thread's site
    int q;          // its spin
    unsigned mir;   // 0x80000000 on the mirror half, else 0
    double t;       // +1 for q = 0, -1 for q = 1
};

__device__ __forceinline__ Lane64 qs_lane64(const Geom &g, int s)
{
    Lane64 ln;
    ln.c = site_of(g, s);
    ln.q = (threadIdx.x >> 4) & 1;
    ln.mir = ln.c.x >= g.L ? 0x80000000u : 0u;
    ln.t = ln.q ? -1.0 : 1.0;
    return ln;
}

// one hop: up, same (spin 2 + q), cross (spin 3 - q) += or, where the flag says so, =
template <int MU, int STEP, class AT, bool FIRST_UP, bool FIRST_LOW>
__device__ __forceinline__ void qs_hop64(const Geom &g, const double2 *__restrict__ links, const double2 *__restrict__ in,
                                         const Lane64 &ln, double2 up[3], double2 same[3], double2 cross[3])
{
    constexpr bool FW = STEP > 0;
    int sg;
    const Nb n = nbr_of<MU, STEP>(g, ln.c, &sg);
    const int lo = (MU == 0 || MU == 3) ? 2 + ln.q : 3 - ln.q;
    double2 a[3], b[3], U[9];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        a[i] = __ldg(in + AT::at(n.s, 3 * ln.q + i));
        b[i] = __ldg(in + AT::at(n.s, 3 * lo + i));
    }
    const double2 *lk = links + (int64_t)(MU * 9) * g.Vphys + (FW ? ln.c.p : n.p);
    const unsigned cj = FW ? ln.mir : (n.mir ? 0u : 0x80000000u);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        U[k] = __ldg(lk + (int64_t)k * g.Vphys);
        U[k].y = qs_flip(U[k].y, cj);
    }
    const double f = FW ? ln.t : -ln.t;
    double2 h[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (MU == 0) h[i] = FW ? make_double2(a[i].x + b[i].x, a[i].y + b[i].y) : make_double2(a[i].x - b[i].x, a[i].y - b[i].y);
        else if (MU == 1) h[i] = FW ? make_double2(a[i].x - b[i].y, a[i].y + b[i].x) : make_double2(a[i].x + b[i].y, a[i].y - b[i].x);
        else if (MU == 2) h[i] = make_double2(fma(f, b[i].x, a[i].x), fma(f, b[i].y, a[i].y));
        else h[i] = make_double2(fma(-f, b[i].y, a[i].x), fma(f, b[i].x, a[i].y));
        if (MU == 0) {
            const unsigned neg = sg < 0 ? 0x80000000u : 0u;   // antiperiodic time
            h[i].x = qs_flip(h[i].x, neg);
            h[i].y = qs_flip(h[i].y, neg);
        }
    }
    double2 *low = (MU == 0 || MU == 3) ? same : cross;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        double2 x;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double2 u = FW ? U[i * 3 + j] : U[j * 3 + i];
            x = j == 0 ? qs_cmul(u, h[j]) : qs_cfma(u, h[j], x);
        }
        if (FIRST_UP) up[i] = x;
        else up[i] = make_double2(up[i].x + x.x, up[i].y + x.y);
        double2 l = low[i];
        if (MU == 0) {
            if (FIRST_LOW) l = FW ? x : make_double2(-x.x, -x.y);
            else l = FW ? make_double2(l.x + x.x, l.y + x.y) : make_double2(l.x - x.x, l.y - x.y);
        } else if (MU == 1) {
            if (FIRST_LOW) l = FW ? make_double2(x.y, -x.x) : make_double2(-x.y, x.x);
            else l = FW ? make_double2(l.x + x.y, l.y - x.x) : make_double2(l.x - x.y, l.y + x.x);
        } else if (MU == 2) {
            l = make_double2(fma(f, x.x, l.x), fma(f, x.y, l.y));
        } else {
            l = make_double2(fma(f, x.y, l.x), fma(-f, x.x, l.y));
        }
        low[i] = l;
    }
}

// the sum of all eight hops: up and low are spins q and 2 + q of it.  Every lane of the warp
// must call it.
template <class AT>
__device__ __forceinline__ void qs_hops64(const Geom &g, const double2 *__restrict__ links, const double2 *__restrict__ in,
                                          const Lane64 &ln, double2 up[3], double2 low[3])
{
    double2 cross[3];
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

// rows of spin q of A v for one chiral block b, v of both spins of the block: own (spin q)
// and oth.  The block is stored as 6 real diagonals and 15 strict-lower complex entries; with
// hq = q on the physical site and 1 - q on the mirror (whose block is S conj(A) S, so that
// element (i, j) is t_i t_j conj(A[i'][j']), i' in the other spin half, t = (+, -)) the thread
// needs the Hermitian 3 x 3 part of half hq and the 3 x 3 part between the halves.
__device__ __forceinline__ void qs_sw64(const double *__restrict__ clov, int64_t V, int p, int b, const Lane64 &ln,
                                        const double2 own[3], const double2 oth[3], double2 out[3])
{
    const int hq = ln.q ^ (ln.mir ? 1 : 0);
    const double *cb = clov + (int64_t)b * 36 * V + p;
    auto ld = [&](int k) { return make_double2(__ldg(cb + (int64_t)(6 + 2 * k) * V), __ldg(cb + (int64_t)(7 + 2 * k) * V)); };
    double2 s[3];   // (1, 0), (2, 0), (2, 1) of half hq
    s[0] = ld(hq ? 9 : 0);
    s[1] = ld(hq ? 13 : 1);
    s[2] = ld(hq ? 14 : 2);
#pragma unroll
    for (int i = 0; i < 3; ++i) s[i].y = qs_flip(s[i].y, ln.mir);
    auto cj = [](double2 e) { return make_double2(e.x, -e.y); };
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
            double2 e = ld(hq ? k1 : k0);
            e.x = qs_flip(e.x, ln.mir);
            e.y = qs_flip(e.y, fi);
            out[r] = qs_cfma(e, oth[c], out[r]);
        }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double d = __ldg(cb + (int64_t)(3 * hq + i) * V);
        out[i] = make_double2(fma(d, own[i].x, out[i].x), fma(d, own[i].y, out[i].y));
    }
}

// up, low += spins q and 2 + q of (dm + A) psi at the thread's site, dm = 4 + m0.  The large term
// dm psi is added last, in one rounding: starting from it, every following sum is rounded at
// its size (relative error against long double 1.8e-16 instead of 1.1e-16 on 4^4 to 6^3 x 4).
template <class AT>
__device__ __forceinline__ void qs_diag64(const Geom &g, const double *__restrict__ clov, const double2 *__restrict__ in,
                                          const Lane64 &ln, double dm, double2 up[3], double2 low[3])
{
#pragma unroll
    for (int b = 0; b < 2; ++b) {
        double2 own[3], oth[3], d[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            own[i] = __ldg(in + AT::at(ln.c.s, 6 * b + 3 * ln.q + i));
            oth[i] = __ldg(in + AT::at(ln.c.s, 6 * b + 3 - 3 * ln.q + i));
        }
        qs_sw64(clov, g.Vphys, ln.c.p, b, ln, own, oth, d);
        double2 *o = b ? low : up;
#pragma unroll
        for (int i = 0; i < 3; ++i)
            o[i] = make_double2(fma(dm, own[i].x, o[i].x + d[i].x), fma(dm, own[i].y, o[i].y + d[i].y));
    }
}
