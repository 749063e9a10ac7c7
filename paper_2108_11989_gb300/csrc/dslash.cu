// The O(a)-improved Wilson-Dirac operator D and Q = gamma_5 D on the C*-doubled
// lattice (Sec. 2 operator, Sec. 3 doublet and Q) in FP64 arithmetic (the FP32-arithmetic
// form for FP32 and 16-bit storage is dslash32.cu).  The site computation, with two threads
// per site, is dslash64.cuh.
#include "dslash64.cuh"

namespace {

// D (or Q) at doubled site s (two threads) for one right-hand side; sites beyond the lattice are
// computed on its last one and not stored
template <class AT>
__device__ __forceinline__ void dslash_site(const Geom &g, const double2 *__restrict__ links,
                                            const double *__restrict__ clov, const double *__restrict__ in_all,
                                            double *__restrict__ out_all, int gamma5, double m0, int r, int s)
{
    const bool on = s < (int)g.Ns;
    const double2 *in = reinterpret_cast<const double2 *>(in_all) + (int64_t)r * g.Ns * 12;
    const Lane64 ln = qs_lane64(g, on ? s : (int)g.Ns - 1);
    double2 up[3], low[3];
    qs_hops64<AT>(g, links, in, ln, up, low);
    qs_diag64<AT>(g, clov, in, ln, 4.0 + m0, up, low);
    if (!on) return;
    double2 *out = reinterpret_cast<double2 *>(out_all) + (int64_t)r * g.Ns * 12;
    const unsigned g5 = gamma5 ? 0x80000000u : 0u;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        out[AT::at(s, 3 * ln.q + i)] = up[i];
        out[AT::at(s, 6 + 3 * ln.q + i)] = make_double2(qs_flip(low[i].x, g5), qs_flip(low[i].y, g5));
    }
}

// A block of NT threads handles NT / 2 consecutive sites of one right-hand side; the right-hand
// side runs fastest over consecutive blocks, so the blocks of one site tile run together and
// share the link and SW-term loads through L2.
template <int NT, int MINB, class AT>
__global__ void __launch_bounds__(NT, MINB) dslash_kernel(DslashArgs<double> a)
{
    const unsigned b = blockIdx.x;
    const int r = (int)(b % (unsigned)a.nrhs);
    const int s = (int)(b / (unsigned)a.nrhs) * (NT / 2) + (int)(threadIdx.x >> 5) * 16 + (int)(threadIdx.x & 15);
    dslash_site<AT>(a.g, a.links, a.clov, a.in, a.out, a.gamma5, a.m0[r], r, s);
}

// Several lattices (configurations of any volume) in one launch: item i owns the
// blocks [off[i], off[i + 1]), laid out as in dslash_kernel.
template <class AT>
__global__ void __launch_bounds__(128, 4) dslash_batch_kernel(const __grid_constant__ BatchArgs<double> a)
{
    const unsigned b = blockIdx.x;
    int i = 0;
#pragma unroll 1
    while (i + 1 < a.n && b >= a.off[i + 1]) ++i;
    const BatchItem<double> &it = a.item[i];
    const unsigned lb = b - a.off[i];
    const int r = (int)(lb % (unsigned)it.nrhs);
    const int s = (int)(lb / (unsigned)it.nrhs) * 64 + (int)(threadIdx.x >> 5) * 16 + (int)(threadIdx.x & 15);
    dslash_site<AT>(it.g, it.links, it.clov, it.in, it.out, a.gamma5, it.m0[r], r, s);
}

template <int NT, int MINB>
cudaError_t launch_variant(const DslashArgs<double> &a, int soa, cudaStream_t st)
{
    const int64_t nb = ((a.g.Ns + NT / 2 - 1) / (NT / 2)) * a.nrhs;
    if (soa) dslash_kernel<NT, MINB, At64Tiled><<<(unsigned)nb, NT, 0, st>>>(a);
    else dslash_kernel<NT, MINB, At64Canon><<<(unsigned)nb, NT, 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace

// Block sizes and registers (blocks per SM); the autotuner in capi.cu picks one per (layout,
// nrhs) by timing.  This kernel serves the FP64 operator; FP32 arithmetic runs in dslash32.cu.
template <>
int qs_dslash_nvariants<double>() { return 3; }

template <>
cudaError_t qs_dslash_launch<double>(DslashArgs<double> a, int nrhs, int variant, int soa, cudaStream_t st)
{
    a.nrhs = nrhs;
    switch (variant) {
    case 0: return launch_variant<32, 12>(a, soa, st);
    case 1: return launch_variant<128, 3>(a, soa, st);
    default: return launch_variant<128, 4>(a, soa, st);
    }
}

// canonical [site][12][re, im] <-> solver [site / 16][12][site % 16][re, im], per vector
__global__ void soa_to_aos_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, int64_t Ns)
{
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;   // canonical complex index
    if (i >= Ns * 12) return;
    int64_t s = i / 12;
    int c = (int)(i % 12);
    out[i] = in[((s >> 4) * 12 + c) * 16 + (s & 15)];
}

cudaError_t qs_soa_to_aos(const double *in, double *out, int64_t Ns, cudaStream_t st)
{
    int64_t n = Ns * 12;
    soa_to_aos_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((const double2 *)in, (double2 *)out, Ns);
    qs_note_launches(1);
    return cudaGetLastError();
}

template <>
cudaError_t qs_dslash_batch_launch<double>(const BatchArgs<double> &a, int soa, cudaStream_t st)
{
    unsigned nb = a.off[a.n];
    if (soa) dslash_batch_kernel<At64Tiled><<<nb, 128, 0, st>>>(a);
    else dslash_batch_kernel<At64Canon><<<nb, 128, 0, st>>>(a);
    qs_note_launches(1);
    return cudaGetLastError();
}
