// Entry points for tests of parts that the C-ABI does not export: the operator's epilogues and
// launch variants, the reductions, and the eigensolver's steps.  solver.cu is included for its
// file-local functions; the rest links against the objects of the library.
#include "../../paper_2108_11989_gb300/csrc/solver.cu"

extern "C" {

QS_API int64_t t_ntile(qs_lattice *lat) { return qs_d32_ntile(lat->g); }
QS_API int t_nvariants() { return qs_d32_nvariants(); }

QS_API int t_fixed_variant(qs_lattice *lat, int nrhs) { return qs_d32_fixed_variant(lat->g, nrhs); }

// one launch of the FP32-arithmetic operator Q with a given variant and epilogue
QS_API int t_d32(qs_lattice *lat, int variant, int storage, int epi, int nrhs, double m0, const void *in, void *out,
                 const void *y, const void *x, double c, double s1, double s2, const float *alpha, const int *live,
                 double *part)
{
    double m[QS_MAX_RHS];
    for (int r = 0; r < nrhs; ++r) m[r] = m0;
    D32Call d;
    memset(&d, 0, sizeof(d));
    d.g = lat->g; d.links = lat->links32; d.clov = lat->clov32;
    d.in = in; d.out = out; d.y = y; d.x = x;
    d.storage = storage; d.nrhs = nrhs; d.gamma5 = 1; d.epi = epi;
    d.cheb_c = c; d.cheb_s1 = s1; d.cheb_s2 = s2;
    d.m0 = m;
    d.alpha_dev = alpha; d.live = live; d.part = part;
    CK(qs_d32_launch(d, variant, lat->stream));
    CK(cudaStreamSynchronize(lat->stream));
    return QS_OK;
}

// |v_r|^2 of k device vectors of nr reals
QS_API int t_norm2(qs_lattice *lat, int f64, const void *v, int k, int64_t nr, double *part, double *out)
{
    if (f64) CK(qs_norm2<double>((const double *)v, k, nr, part, out, lat->stream));
    else CK(qs_norm2<float>((const float *)v, k, nr, part, out, lat->stream));
    CK(cudaStreamSynchronize(lat->stream));
    return QS_OK;
}

// |a_r - theta_r b_r|^2 of k pairs of FP32 device vectors of nr reals
QS_API int t_resid2(qs_lattice *lat, const float *a, const float *b, const double *theta, int k, int64_t nr, double *part,
                    double *out)
{
    CK(qs_resid2<float>(a, b, theta, k, nr, part, out, lat->stream));
    CK(cudaStreamSynchronize(lat->stream));
    return QS_OK;
}

// FP32 CG on Q(m0)^2 for the k device vectors b (solver layout); counts: f32_count, cg_count, iterations
QS_API int t_cg(qs_lattice *lat, int k, double m0, double tol, int maxit, const float *b, float *x, int64_t *counts)
{
    Workspace *w;
    QS_TRY(ws_get(lat, k, &w));
    const int64_t f0 = w->f32_count, c0 = w->cg_count;
    const size_t bytes = (size_t)k * w->nr * sizeof(float);
    CK(cudaMemcpyAsync(w->blk32[0], b, bytes, cudaMemcpyDeviceToDevice, lat->stream));
    int it = 0;
    QS_TRY(cg_f32(lat, w, m0, k, w->blk32[1], w->blk32[0], w->blk32[2], w->blk32[3], tol, maxit, &it));
    CK(cudaMemcpyAsync(x, w->blk32[1], bytes, cudaMemcpyDeviceToDevice, lat->stream));
    CK(cudaStreamSynchronize(lat->stream));
    counts[0] = w->f32_count - f0;
    counts[1] = w->cg_count - c0;
    counts[2] = it;
    return QS_OK;
}

// the Rayleigh-Ritz matrix V^H Q V (k x k complex, host) of the FP32 stage for the k device vectors V
// (solver layout), and the image Q V that it was formed from
QS_API int t_rr32(qs_lattice *lat, int k, double m0, const float *V, float *QV, double *H)
{
    Workspace *w;
    QS_TRY(ws_get(lat, k, &w));
    const size_t bytes = (size_t)k * w->nr * sizeof(float);
    CK(cudaMemcpyAsync(V32(w), V, bytes, cudaMemcpyDeviceToDevice, lat->stream));
    QS_TRY(opQ(lat, w, QS_F32, m0, V32(w), QV, k));   // rayleigh_ritz32 rotates its own copy
    Ritz rz;
    const int s = rayleigh_ritz32(lat, w, m0, k, &rz);
    CK(cudaMemcpy(H, w->Hm, (size_t)k * k * sizeof(double2), cudaMemcpyDeviceToHost));
    return s == QS_OK || s == QS_ENOCONV ? QS_OK : s;
}

}  // extern "C"
