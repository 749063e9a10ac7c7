// Step-proposal network of the learned form of the sign flow: a 3-layer
// perceptron in FP32 (in -> hidden -> hidden -> out, ReLU), trained on the GPU by
// the kernels below (forward, backward, loss, Adam).  The paper itself steps with
// m <- m + c lambda_bar (Sec. 3); a proposal of this network is used only where the
// flow's no-crossing certificate (eq. derivativebound) accepts it.
//
// Parameters are one FP32 array [W1 (h x in), b1, W2 (h x h), b2, W3 (out x h), b3].
// Loss over B rows, targets T (column 0 regression, columns 1.. labels):
//   L = (1/B) sum_b [ (Y_b0 - T_b0)^2 / 2 + sum_{j>=1} (softplus(Y_bj) - T_bj Y_bj) ].
#include "qs_internal.cuh"

#include <stdlib.h>

// A training step is a chain of small products (512 x 192 x 128 at the largest use), bound by
// launches and by the latency of each, so it is cut to eight launches (17 before; batch 512: 150 ->
// 48 us of kernels, 235 -> 111 us a step with the loss read back): bias and ReLU are part of the products, the three weight gradients are one
// launch over slices of the batch, and the Adam kernel adds the slices, in a fixed order.
struct qs_mlp {
    int ni, nh, no, maxB, device;
    cudaStream_t stream;
    size_t np, off[7];
    float *P, *G, *M, *V;
    float *Gp;   // [MLP_SPLIT][np] gradients of the batch slices
    float *A1, *A2, *Y, *dY, *dZ1, *dZ2, *rowloss, *loss;
    int t;
};

namespace {

#define TM 32          // output tile and depth of one step; 256 threads, 2 x 2 outputs each
#define MLP_SPLIT 8    // most slices of the batch in the weight gradients

// C[m][n] = sum_{k0 <= k < k1} A(m, k) B(k, n); A(m, k) = A[m sam + k sak], B(k, n) = B[k sbk + n sbn]
struct Gemm {
    int M, N, K;
    const float *A, *B;
    int sam, sak, sbk, sbn;
    float *C;            // row-major, ld = N
    const float *bias;   // NULL, or added per column
    int relu;            // clamp at 0
    const float *mask;   // NULL, or C is zeroed where mask[m][n] <= 0 (the ReLU's derivative)
    float *asum;         // NULL, or asum[m] = sum_k A(m, k)
};

__device__ __forceinline__ void gemm_block(const Gemm &g, int bm, int bn, int k0, int k1)
{
    __shared__ float as[TM][TM + 1], bs[TM][TM + 1];   // [k][m], [k][n]
    const int t = threadIdx.x, lo = t & 31, hi = t >> 5;
    const int m0 = bm * TM, n0 = bn * TM;
    const bool ak = g.sak == 1, bk = g.sbk == 1;   // consecutive threads along k, or along m / n
    float ra[4], rb[4];
    auto fetch = [&](int kb) {   // the next step's words are in flight while this one is multiplied
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = lo, y = hi + 8 * i;
            const int ka = kb + (ak ? x : y), m = m0 + (ak ? y : x);
            const int kc = kb + (bk ? x : y), n = n0 + (bk ? y : x);
            ra[i] = m < g.M && ka < k1 ? g.A[(int64_t)m * g.sam + (int64_t)ka * g.sak] : 0.f;
            rb[i] = n < g.N && kc < k1 ? g.B[(int64_t)kc * g.sbk + (int64_t)n * g.sbn] : 0.f;
        }
    };
    float c[2][2] = {{0.f, 0.f}, {0.f, 0.f}}, sum = 0.f;
    const int tm = t >> 4, tn = t & 15;
    fetch(k0);
    for (int kb = k0; kb < k1; kb += TM) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = lo, y = hi + 8 * i;
            as[ak ? x : y][ak ? y : x] = ra[i];
            bs[bk ? x : y][bk ? y : x] = rb[i];
        }
        __syncthreads();
        if (kb + TM < k1) fetch(kb + TM);
#pragma unroll
        for (int k = 0; k < TM; ++k) {
            const float a0 = as[k][tm], a1 = as[k][tm + 16], b0 = bs[k][tn], b1 = bs[k][tn + 16];
            c[0][0] = fmaf(a0, b0, c[0][0]);
            c[0][1] = fmaf(a0, b1, c[0][1]);
            c[1][0] = fmaf(a1, b0, c[1][0]);
            c[1][1] = fmaf(a1, b1, c[1][1]);
        }
        if (g.asum && bn == 0 && t < TM) {
#pragma unroll
            for (int k = 0; k < TM; ++k) sum += as[k][t];
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int m = m0 + tm + 16 * i, n = n0 + tn + 16 * j;
            if (m >= g.M || n >= g.N) continue;
            float v = c[i][j] + (g.bias ? g.bias[n] : 0.f);
            if (g.relu) v = fmaxf(v, 0.f);
            if (g.mask && !(g.mask[(int64_t)m * g.N + n] > 0.f)) v = 0.f;
            g.C[(int64_t)m * g.N + n] = v;
        }
    if (g.asum && bn == 0 && t < TM && m0 + t < g.M) g.asum[m0 + t] = sum;
}

__global__ void __launch_bounds__(256) gemm_kernel(Gemm g) { gemm_block(g, blockIdx.y, blockIdx.x, 0, g.K); }

// the three weight gradients over slice blockIdx.y of the batch: C and asum lie in slice s of Gp
struct Grads {
    Gemm g[3];
    int first[4];   // first block of each product
    int slice;      // batch rows per slice
    size_t np;
};

__global__ void __launch_bounds__(256) grads_kernel(const __grid_constant__ Grads a)
{
    int q = 0;
    while (q < 2 && (int)blockIdx.x >= a.first[q + 1]) ++q;
    Gemm g = a.g[q];
    g.C += blockIdx.y * a.np;
    g.asum += blockIdx.y * a.np;
    const int b = (int)blockIdx.x - a.first[q], nn = (g.N + TM - 1) / TM;
    const int k0 = (int)blockIdx.y * a.slice, k1 = min(g.K, k0 + a.slice);
    gemm_block(g, b / nn, b % nn, k0, k1);
}

// one warp per row: dL/dY and the row's loss
__global__ void __launch_bounds__(256) loss_grad_kernel(const float *__restrict__ Y, const float *__restrict__ T, int B, int no,
                                                        float *__restrict__ dY, float *__restrict__ rowloss)
{
    const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= B) return;
    const float *y = Y + (long)b * no, *t = T + (long)b * no;
    float *d = dY + (long)b * no;
    float l = 0.f;
    for (int j = lane; j < no; j += 32) {
        const float z = y[j];
        if (j == 0) {
            const float r = z - t[0];
            l += 0.5f * r * r;
            d[0] = r / B;
        } else {
            const float sp = z > 0.f ? z + log1pf(expf(-z)) : log1pf(expf(z));
            l += sp - t[j] * z;
            d[j] = (1.f / (1.f + expf(-z)) - t[j]) / B;
        }
    }
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) rowloss[b] = l;
}

// G = sum of the batch slices' gradients, one Adam step; the last block: the mean loss
__global__ void __launch_bounds__(256) adam_kernel(float *__restrict__ P, float *__restrict__ G, const float *__restrict__ Gp,
                                                   int nsplit, float *__restrict__ M, float *__restrict__ V, long n, float lr,
                                                   float b1, float b2, float eps, float c1, float c2,
                                                   const float *__restrict__ rowloss, int B, float *__restrict__ loss)
{
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float sh[256];
        float s = 0.f;
        for (int i = threadIdx.x; i < B; i += 256) s += rowloss[i];
        sh[threadIdx.x] = s;
        __syncthreads();
        for (int w = 128; w > 0; w >>= 1) {
            if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
            __syncthreads();
        }
        if (threadIdx.x == 0) *loss = sh[0] / B;
        return;
    }
    const long i = blockIdx.x * 256L + threadIdx.x;
    if (i >= n) return;
    float g = 0.f;
    for (int s = 0; s < nsplit; ++s) g += Gp[s * n + i];
    G[i] = g;
    float m = b1 * M[i] + (1.f - b1) * g;
    float v = b2 * V[i] + (1.f - b2) * g * g;
    M[i] = m;
    V[i] = v;
    P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
}

Gemm product(int M, int N, int K, const float *A, int sam, int sak, const float *B, int sbk, int sbn, float *C)
{
    return {M, N, K, A, B, sam, sak, sbk, sbn, C, nullptr, 0, nullptr, nullptr};
}

cudaError_t run(cudaStream_t st, const Gemm &g)
{
    gemm_kernel<<<dim3((g.N + TM - 1) / TM, (g.M + TM - 1) / TM), 256, 0, st>>>(g);
    qs_note_launches(1);
    return cudaGetLastError();
}

int forward(qs_mlp *n, const float *X, int B, float *Y)
{
    const int ni = n->ni, nh = n->nh, no = n->no;
    const float *W1 = n->P + n->off[0], *W2 = n->P + n->off[2], *W3 = n->P + n->off[4];
    Gemm g = product(B, nh, ni, X, ni, 1, W1, 1, ni, n->A1);
    g.bias = n->P + n->off[1];
    g.relu = 1;
    QS_CUDA(run(n->stream, g));
    g = product(B, nh, nh, n->A1, nh, 1, W2, 1, nh, n->A2);
    g.bias = n->P + n->off[3];
    g.relu = 1;
    QS_CUDA(run(n->stream, g));
    g = product(B, no, nh, n->A2, nh, 1, W3, 1, nh, Y);
    g.bias = n->P + n->off[5];
    QS_CUDA(run(n->stream, g));
    return QS_OK;
}

}  // namespace

extern "C" int qs_mlp_create(int n_in, int n_hidden, int n_out, int max_batch, void *stream, qs_mlp **out)
{
    if (!out || n_in < 1 || n_hidden < 1 || n_out < 2 || max_batch < 1) return QS_EINVAL;
    if ((long)max_batch * (n_hidden > n_out ? n_hidden : n_out) > (1L << 28)) return QS_EINVAL;
    *out = nullptr;
    qs_mlp *n = (qs_mlp *)calloc(1, sizeof(qs_mlp));
    if (!n) return QS_ENOMEM;
    QS_CUDA(cudaGetDevice(&n->device));
    n->ni = n_in; n->nh = n_hidden; n->no = n_out; n->maxB = max_batch;
    n->stream = (cudaStream_t)stream;
    size_t sz[6] = {(size_t)n_hidden * n_in, (size_t)n_hidden, (size_t)n_hidden * n_hidden, (size_t)n_hidden,
                    (size_t)n_out * n_hidden, (size_t)n_out};
    n->off[0] = 0;
    for (int i = 0; i < 6; ++i) n->off[i + 1] = n->off[i] + sz[i];
    n->np = n->off[6];
    size_t hb = (size_t)max_batch * n_hidden, ob = (size_t)max_batch * n_out;
    cudaError_t e = cudaSuccess;
    float **bufs[] = {&n->P, &n->G, &n->M, &n->V};
    e = cudaMalloc(&n->Gp, MLP_SPLIT * n->np * sizeof(float));
    for (float **b : bufs) if (e == cudaSuccess) e = cudaMalloc(b, n->np * sizeof(float));
    float **acts[] = {&n->A1, &n->A2, &n->dZ1, &n->dZ2};
    for (float **b : acts) if (e == cudaSuccess) e = cudaMalloc(b, hb * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->Y, ob * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->dY, ob * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->rowloss, (size_t)max_batch * sizeof(float));
    if (e == cudaSuccess) e = cudaMalloc(&n->loss, sizeof(float));
    if (e == cudaSuccess) e = cudaMemsetAsync(n->P, 0, n->np * sizeof(float), n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->M, 0, n->np * sizeof(float), n->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(n->V, 0, n->np * sizeof(float), n->stream);
    if (e != cudaSuccess) {
        qs_record_cuda_error(e, "qs_mlp_create");
        qs_mlp_destroy(n);
        return e == cudaErrorMemoryAllocation ? QS_ENOMEM : QS_ECUDA;
    }
    *out = n;
    return QS_OK;
}

extern "C" int qs_mlp_destroy(qs_mlp *n)
{
    if (!n) return QS_OK;
    float *all[] = {n->P, n->G, n->M, n->V, n->Gp, n->A1, n->A2, n->dZ1, n->dZ2, n->Y, n->dY, n->rowloss, n->loss};
    for (float *p : all) cudaFree(p);
    free(n);
    return QS_OK;
}

extern "C" int64_t qs_mlp_n_params(const qs_mlp *n) { return n ? (int64_t)n->np : 0; }

cudaStream_t qs_mlp_stream(const qs_mlp *n) { return n->stream; }

extern "C" int qs_mlp_set_params(qs_mlp *n, const float *host)
{
    if (!n || !host) return QS_EINVAL;
    QS_CUDA(cudaMemcpyAsync(n->P, host, n->np * sizeof(float), cudaMemcpyHostToDevice, n->stream));
    QS_CUDA(cudaMemsetAsync(n->M, 0, n->np * sizeof(float), n->stream));
    QS_CUDA(cudaMemsetAsync(n->V, 0, n->np * sizeof(float), n->stream));
    QS_CUDA(cudaStreamSynchronize(n->stream));
    n->t = 0;
    return QS_OK;
}

extern "C" int qs_mlp_get_params(qs_mlp *n, float *host)
{
    if (!n || !host) return QS_EINVAL;
    QS_CUDA(cudaMemcpyAsync(host, n->P, n->np * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    QS_CUDA(cudaStreamSynchronize(n->stream));
    return QS_OK;
}

extern "C" int qs_mlp_get_grads(qs_mlp *n, float *host)
{
    if (!n || !host) return QS_EINVAL;
    QS_CUDA(cudaMemcpyAsync(host, n->G, n->np * sizeof(float), cudaMemcpyDeviceToHost, n->stream));
    QS_CUDA(cudaStreamSynchronize(n->stream));
    return QS_OK;
}

extern "C" int qs_mlp_forward(qs_mlp *n, const float *X, int B, float *Y)
{
    if (!n || !X || !Y || B < 1 || B > n->maxB) return QS_EINVAL;
    return forward(n, X, B, Y);
}

extern "C" int qs_mlp_train_step(qs_mlp *n, const float *X, const float *T, int B, float lr, float *loss)
{
    if (!n || !X || !T || B < 1 || B > n->maxB || !(lr > 0)) return QS_EINVAL;
    const int ni = n->ni, nh = n->nh, no = n->no;
    cudaStream_t st = n->stream;
    QS_TRY(forward(n, X, B, n->Y));
    const float *W2 = n->P + n->off[2], *W3 = n->P + n->off[4];
    loss_grad_kernel<<<(B + 7) / 8, 256, 0, st>>>(n->Y, T, B, no, n->dY, n->rowloss);
    qs_note_launches(1);
    // dZ2 = (dY W3) where A2 > 0, dZ1 = (dZ2 W2) where A1 > 0
    Gemm g = product(B, nh, no, n->dY, no, 1, W3, nh, 1, n->dZ2);
    g.mask = n->A2;
    QS_CUDA(run(st, g));
    g = product(B, nh, nh, n->dZ2, nh, 1, W2, nh, 1, n->dZ1);
    g.mask = n->A1;
    QS_CUDA(run(st, g));
    // dW = dZ^T (layer input), db = column sums of dZ, over slices of at least 64 rows
    Grads a;
    const float *dz[3] = {n->dZ1, n->dZ2, n->dY}, *in[3] = {X, n->A1, n->A2};
    const int m[3] = {nh, nh, no}, nn[3] = {ni, nh, nh};
    a.first[0] = 0;
    for (int q = 0; q < 3; ++q) {
        a.g[q] = product(m[q], nn[q], B, dz[q], 1, m[q], in[q], nn[q], 1, n->Gp + n->off[2 * q]);
        a.g[q].asum = n->Gp + n->off[2 * q + 1];
        a.first[q + 1] = a.first[q] + ((m[q] + TM - 1) / TM) * ((nn[q] + TM - 1) / TM);
    }
    const int nsplit = B >= 64 * MLP_SPLIT ? MLP_SPLIT : (B + 63) / 64;
    a.slice = (B + nsplit - 1) / nsplit;
    a.np = n->np;
    grads_kernel<<<dim3(a.first[3], nsplit), 256, 0, st>>>(a);
    n->t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    adam_kernel<<<(unsigned)((n->np + 255) / 256 + 1), 256, 0, st>>>(
        n->P, n->G, n->Gp, nsplit, n->M, n->V, (long)n->np, lr, b1, b2, 1e-8f, 1.f - powf(b1, (float)n->t),
        1.f - powf(b2, (float)n->t), n->rowloss, B, n->loss);
    qs_note_launches(2);
    QS_CUDA(cudaGetLastError());
    if (loss) {
        QS_CUDA(cudaMemcpyAsync(loss, n->loss, sizeof(float), cudaMemcpyDeviceToHost, st));
        QS_CUDA(cudaStreamSynchronize(st));
    }
    return QS_OK;
}
