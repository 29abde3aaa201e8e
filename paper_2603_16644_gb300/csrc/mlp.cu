// Learned precision proposal (not part of the paper's method; it proposes the
// u_p of Alg. 1 and is checked by a condition estimate):
//   - features of A: column-norm statistics and the diagonal of the
//     preconditioner from an FP8-e4m3 sparse-sign sketch with an FP32 QR;
//   - an MLP d -> 64 -> 64 -> 64 -> 4 (ReLU, softmax cross-entropy) in FP32:
//     forward, backward (sums over chunks of 32 samples, then over the chunks
//     in a fixed order: deterministic) and Adam;
//   - the judge: Hager's 1-norm estimate (Sec. 6.1's estimator, single
//     precision, csrc/hager.cu) of kappa_1(R_s) for a computed
//     preconditioner; a precision
//     u_p is accepted when u_p * kappa_1(R_s) <= 1, the regime of Lemma
//     rscond (eps * kappa(R_s) < 1).
#include "common.cuh"
#include "kernels.cuh"

#include <algorithm>

namespace lsq {

constexpr int MH = 64;   // hidden width
constexpr int MC = 4;    // classes: FP8-e4m3, BF16, FP32, FP64
constexpr int NFEAT = 10;

__host__ __device__ inline int64_t mlp_params(int d) { return (int64_t)MH * d + MH + 2 * ((int64_t)MH * MH + MH) + (int64_t)MC * MH + MC; }

struct MlpPtrs {
    const float *W1, *b1, *W2, *b2, *W3, *b3, *W4, *b4;
};

__device__ inline MlpPtrs mlp_ptrs(const float* p, int d) {
    MlpPtrs q;
    q.W1 = p;
    q.b1 = q.W1 + MH * d;
    q.W2 = q.b1 + MH;
    q.b2 = q.W2 + MH * MH;
    q.W3 = q.b2 + MH;
    q.b3 = q.W3 + MH * MH;
    q.W4 = q.b3 + MH;
    q.b4 = q.W4 + MC * MH;
    return q;
}

// Forward for one sample; z1..z3 are the pre-activations (kept for backward).
__device__ void mlp_fwd1(const MlpPtrs& P, int d, const float* x, float* z1, float* z2, float* z3, float* z4) {
    for (int o = 0; o < MH; ++o) {
        float a = P.b1[o];
        for (int i = 0; i < d; ++i) a = fmaf(P.W1[o * d + i], x[i], a);
        z1[o] = a;
    }
    for (int o = 0; o < MH; ++o) {
        float a = P.b2[o];
        for (int i = 0; i < MH; ++i) a = fmaf(P.W2[o * MH + i], fmaxf(z1[i], 0.0f), a);
        z2[o] = a;
    }
    for (int o = 0; o < MH; ++o) {
        float a = P.b3[o];
        for (int i = 0; i < MH; ++i) a = fmaf(P.W3[o * MH + i], fmaxf(z2[i], 0.0f), a);
        z3[o] = a;
    }
    for (int c = 0; c < MC; ++c) {
        float a = P.b4[c];
        for (int i = 0; i < MH; ++i) a = fmaf(P.W4[c * MH + i], fmaxf(z3[i], 0.0f), a);
        z4[c] = a;
    }
}

__global__ void k_mlp_forward(const float* __restrict__ params, int d, int batch, const float* __restrict__ X,
                              float* __restrict__ logits) {
    extern __shared__ float sp[];
    int64_t np = mlp_params(d);
    for (int64_t q = threadIdx.x; q < np; q += blockDim.x) sp[q] = params[q];
    __syncthreads();
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= batch) return;
    MlpPtrs P = mlp_ptrs(sp, d);
    float z1[MH], z2[MH], z3[MH], z4[MC];
    mlp_fwd1(P, d, X + (int64_t)s * d, z1, z2, z3, z4);
    for (int c = 0; c < MC; ++c) logits[(int64_t)s * MC + c] = z4[c];
}

// Gradient of the mean loss, first pass: one CTA per MB samples runs forward
// and backward for them with the parameters, activations and deltas in shared
// memory and writes its own sum of every parameter's gradient, and of the
// loss, to part[chunk][np + 1]; k_mlp_reduce adds the chunks in order
// (deterministic).  The work is small (0.23 GFLOP at a batch of 4096), so
// latency bounds it: what counts is that many threads share it.  One thread
// per sample and then one thread per parameter walking the whole batch took
// 0.07 + 1.0 ms of a 1.16 ms training step at a batch of 4096; the two passes
// here take the step to 0.05 ms (launches and host calls by then).
// MB = 32: 128 CTAs at a batch of 4096, one sample per lane in the softmax.
constexpr int MB = 32;           // samples per CTA
constexpr int MT = 256;          // threads per CTA
constexpr int MLD = MB + 4;      // [unit][sample] rows, 16-byte aligned, conflict-free by float4
constexpr int MWL = MH + 1;      // weight rows in shared memory
constexpr int MLP_SMEM = (3 * MH * MLD * 2 + MC * MLD + 2 * MH * MWL + MC * MWL + 2 * MH + MC + 8) * (int)sizeof(float);

// out[o][s] = bias[o] + sum_i W[o][i] relu(in[i][s]) for 2 units (lane, lane + 32)
// and 4 samples (4 warp ..) per thread; relu'd inputs are what `in` holds.
__device__ __forceinline__ void mlp_layer(const float* W, const float* bias, const float* in, float* out, int lane,
                                          int warp, bool relu) {
    float a0[4], a1[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) a0[q] = bias[lane], a1[q] = bias[lane + 32];
#pragma unroll 8
    for (int i = 0; i < MH; ++i) {
        const float w0 = W[lane * MWL + i], w1 = W[(lane + 32) * MWL + i];
        const float4 h = *(const float4*)(in + i * MLD + 4 * warp);
        a0[0] = fmaf(w0, h.x, a0[0]), a0[1] = fmaf(w0, h.y, a0[1]), a0[2] = fmaf(w0, h.z, a0[2]), a0[3] = fmaf(w0, h.w, a0[3]);
        a1[0] = fmaf(w1, h.x, a1[0]), a1[1] = fmaf(w1, h.y, a1[1]), a1[2] = fmaf(w1, h.z, a1[2]), a1[3] = fmaf(w1, h.w, a1[3]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        out[lane * MLD + 4 * warp + q] = relu ? fmaxf(a0[q], 0.0f) : a0[q];
        out[(lane + 32) * MLD + 4 * warp + q] = relu ? fmaxf(a1[q], 0.0f) : a1[q];
    }
}

// prev[i][s] = sum_o W[o][i] del[o][s] where act[i][s] > 0, else 0 (the same split).
__device__ __forceinline__ void mlp_back(const float* W, int nout, const float* del, const float* act, float* prev,
                                         int lane, int warp) {
    float a0[4] = {0, 0, 0, 0}, a1[4] = {0, 0, 0, 0};
#pragma unroll 4
    for (int o = 0; o < nout; ++o) {
        const float w0 = W[o * MWL + lane], w1 = W[o * MWL + lane + 32];
        const float4 h = *(const float4*)(del + o * MLD + 4 * warp);
        a0[0] = fmaf(w0, h.x, a0[0]), a0[1] = fmaf(w0, h.y, a0[1]), a0[2] = fmaf(w0, h.z, a0[2]), a0[3] = fmaf(w0, h.w, a0[3]);
        a1[0] = fmaf(w1, h.x, a1[0]), a1[1] = fmaf(w1, h.y, a1[1]), a1[2] = fmaf(w1, h.z, a1[2]), a1[3] = fmaf(w1, h.w, a1[3]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int s = 4 * warp + q;
        prev[lane * MLD + s] = act[lane * MLD + s] > 0.0f ? a0[q] : 0.0f;
        prev[(lane + 32) * MLD + s] = act[(lane + 32) * MLD + s] > 0.0f ? a1[q] : 0.0f;
    }
}

// sum over the CTA's samples of del[o][s] act[i][s] for a 64 x 64 weight
// matrix: 4 x 4 outputs per thread (o = ty + 16 a, i = tx + 16 b).
__device__ __forceinline__ void mlp_outer(const float* del, const float* act, float* __restrict__ g, int tid) {
    const int tx = tid & 15, ty = tid >> 4;
    float c[4][4] = {};
#pragma unroll
    for (int s = 0; s < MB; s += 4) {
        float4 d[4], x[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            d[a] = *(const float4*)(del + (ty + 16 * a) * MLD + s);
            x[a] = *(const float4*)(act + (tx + 16 * a) * MLD + s);
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b)
                c[a][b] = fmaf(d[a].w, x[b].w, fmaf(d[a].z, x[b].z, fmaf(d[a].y, x[b].y, fmaf(d[a].x, x[b].x, c[a][b]))));
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) g[(ty + 16 * a) * MH + tx + 16 * b] = c[a][b];
}

__device__ __forceinline__ float mlp_row_sum(const float* row) {
    float t = 0.0f;
#pragma unroll
    for (int s = 0; s < MB; s += 4) {
        const float4 v = *(const float4*)(row + s);
        t += (v.x + v.y) + (v.z + v.w);
    }
    return t;
}

__global__ void __launch_bounds__(MT) k_mlp_grad_part(const float* __restrict__ params, int d, int batch,
                                                      const float* __restrict__ X, const int32_t* __restrict__ labels,
                                                      float* __restrict__ part) {
    extern __shared__ __align__(16) float msm[];
    float* H1 = msm;                 // relu'd activations [unit][sample]
    float* H2 = H1 + MH * MLD;
    float* H3 = H2 + MH * MLD;
    float* D1 = H3 + MH * MLD;       // deltas
    float* D2 = D1 + MH * MLD;
    float* D3 = D2 + MH * MLD;
    float* D4 = D3 + MH * MLD;       // logits, then deltas of the output
    float* W2 = D4 + MC * MLD;
    float* W3 = W2 + MH * MWL;
    float* W4 = W3 + MH * MWL;
    float* b2 = W4 + MC * MWL;
    float* b3 = b2 + MH;
    float* b4 = b3 + MH;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const MlpPtrs P = mlp_ptrs(params, d);
    const int64_t s0 = (int64_t)blockIdx.x * MB;
    const int ns = (int)min64(MB, batch - s0);
    for (int q = tid; q < MH * MH; q += MT) {
        W2[(q >> 6) * MWL + (q & 63)] = P.W2[q];
        W3[(q >> 6) * MWL + (q & 63)] = P.W3[q];
    }
    if (tid < MC * MH) W4[(tid >> 6) * MWL + (tid & 63)] = P.W4[tid];
    if (tid < MH) b2[tid] = P.b2[tid], b3[tid] = P.b3[tid];
    if (tid < MC) b4[tid] = P.b4[tid];
    // layer 1: W1 and X from global memory (any d); samples past the batch are zero
    for (int o = lane; o < MH; o += 32) {
        float a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = P.b1[o];
        for (int i = 0; i < d; ++i) {
            const float w = P.W1[o * d + i];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int s = 4 * warp + q;
                a[q] = fmaf(w, s < ns ? X[(s0 + s) * d + i] : 0.0f, a[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) H1[o * MLD + 4 * warp + q] = fmaxf(a[q], 0.0f);
    }
    __syncthreads();
    mlp_layer(W2, b2, H1, H2, lane, warp, true);
    __syncthreads();
    mlp_layer(W3, b3, H2, H3, lane, warp, true);
    __syncthreads();
    if (tid < MC * MB) {
        const int c = tid >> 5, s = tid & 31;
        float a = b4[c];
        for (int i = 0; i < MH; ++i) a = fmaf(W4[c * MWL + i], H3[i * MLD + s], a);
        D4[c * MLD + s] = a;
    }
    __syncthreads();
    float* out = part + (int64_t)blockIdx.x * (mlp_params(d) + 1);
    if (warp == 0) {
        // softmax cross-entropy, lane = sample
        float z[MC], mx, se = 0.0f, l = 0.0f;
#pragma unroll
        for (int c = 0; c < MC; ++c) z[c] = D4[c * MLD + lane];
        mx = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));
#pragma unroll
        for (int c = 0; c < MC; ++c) se += expf(z[c] - mx);
        const int y = lane < ns ? labels[s0 + lane] : -1;
#pragma unroll
        for (int c = 0; c < MC; ++c) {
            if (c == y) l = -(z[c] - mx - logf(se));
            D4[c * MLD + lane] = lane < ns ? (expf(z[c] - mx) / se - (c == y ? 1.0f : 0.0f)) / (float)batch : 0.0f;
        }
        for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
        if (lane == 0) out[mlp_params(d)] = l;
    }
    __syncthreads();
    mlp_back(W4, MC, D4, H3, D3, lane, warp);
    __syncthreads();
    mlp_back(W3, MH, D3, H2, D2, lane, warp);
    __syncthreads();
    mlp_back(W2, MH, D2, H1, D1, lane, warp);
    __syncthreads();
    // gradients in the parameter packing W1 b1 W2 b2 W3 b3 W4 b4
    float* g1 = out;
    float* gb1 = g1 + MH * d;
    float* g2 = gb1 + MH;
    float* gb2 = g2 + MH * MH;
    float* g3 = gb2 + MH;
    float* gb3 = g3 + MH * MH;
    float* g4 = gb3 + MH;
    float* gb4 = g4 + MC * MH;
    mlp_outer(D2, H1, g2, tid);
    mlp_outer(D3, H2, g3, tid);
    for (int q = tid; q < MH * d; q += MT) {
        const int o = q / d, i = q % d;
        float t = 0.0f;
        for (int s = 0; s < ns; ++s) t = fmaf(D1[o * MLD + s], X[(s0 + s) * d + i], t);
        g1[q] = t;
    }
    {
        const int c = tid >> 6, i = tid & 63;
        float t = 0.0f;
#pragma unroll
        for (int s = 0; s < MB; ++s) t = fmaf(D4[c * MLD + s], H3[i * MLD + s], t);
        g4[tid] = t;
    }
    if (tid < MH) gb1[tid] = mlp_row_sum(D1 + tid * MLD);
    else if (tid < 2 * MH) gb2[tid - MH] = mlp_row_sum(D2 + (tid - MH) * MLD);
    else if (tid < 3 * MH) gb3[tid - 2 * MH] = mlp_row_sum(D3 + (tid - 2 * MH) * MLD);
    else if (tid < 3 * MH + MC) gb4[tid - 3 * MH] = mlp_row_sum(D4 + (tid - 3 * MH) * MLD);
}

// Second pass: the chunks' sums added in a fixed order (8 contiguous ranges of
// chunks, one per warp, then the 8 sums in order).  One CTA per 32 entries.
__global__ void __launch_bounds__(256) k_mlp_reduce(const float* __restrict__ part, int64_t np, int chunks, int batch,
                                                    float* __restrict__ grad, float* __restrict__ loss) {
    __shared__ float sh[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t q = (int64_t)blockIdx.x * 32 + lane;
    const int c0 = (int)((int64_t)chunks * w / 8), c1 = (int)((int64_t)chunks * (w + 1) / 8);
    float t = 0.0f;
    if (q <= np) {
#pragma unroll 8
        for (int c = c0; c < c1; ++c) t += part[(int64_t)c * (np + 1) + q];
    }
    sh[w][lane] = t;
    __syncthreads();
    if (w == 0 && q <= np) {
        t = ((sh[0][lane] + sh[1][lane]) + (sh[2][lane] + sh[3][lane])) + ((sh[4][lane] + sh[5][lane]) + (sh[6][lane] + sh[7][lane]));
        if (q < np) grad[q] = t;
        else if (loss) *loss = t / (float)batch;
    }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, int64_t count, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= count) return;
    float gq = g[q];
    float a = b1 * m1[q] + (1.0f - b1) * gq;
    float v = b2 * m2[q] + (1.0f - b2) * gq * gq;
    m1[q] = a;
    m2[q] = v;
    p[q] -= lr * (a / c1) / (sqrtf(v / c2) + eps);
}

// ---------------------------------------------------------------------------
// Features (see the oracle for the definitions), one block.
// ---------------------------------------------------------------------------
__global__ void k_colnorm2(const double* __restrict__ A, int64_t m, int64_t lda, double* __restrict__ out) {
    int64_t c = blockIdx.x;
    const double* col = A + c * lda;
    double s = 0.0;
    for (int64_t i = threadIdx.x; i < m; i += blockDim.x) s = fma(col[i], col[i], s);
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    __shared__ double w[32];
    if ((threadIdx.x & 31) == 0) w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += w[q];
        out[c] = t;
    }
}

__global__ void k_features(const double* __restrict__ cn2, const double* __restrict__ Rs, int64_t ldr, int64_t m,
                           int64_t n, float* __restrict__ f) {
    if (threadIdx.x != 0) return;
    double cmax = -1e300, cmin = 1e300, cmean = 0, dmax = -1e300, dmin = 1e300, dmean = 0, fro = 0;
    for (int64_t j = 0; j < n; ++j) {
        double cn = log10(fmax(sqrt(cn2[j]), 1e-300));
        double dj = log10(fmax(fabs(Rs[j + j * ldr]), 1e-300));
        fro += cn2[j];
        cmax = fmax(cmax, cn); cmin = fmin(cmin, cn); cmean += cn;
        dmax = fmax(dmax, dj); dmin = fmin(dmin, dj); dmean += dj;
    }
    cmean /= n;
    dmean /= n;
    double cvar = 0, dvar = 0, sxy = 0, sxx = 0;
    int64_t q0 = n - (n + 3) / 4;
    double tmax = -1e300, tmin = 1e300;
    int64_t small = 0;
    for (int64_t j = 0; j < n; ++j) {
        double cn = log10(fmax(sqrt(cn2[j]), 1e-300));
        double dj = log10(fmax(fabs(Rs[j + j * ldr]), 1e-300));
        double t = (double)j / (double)n - 0.5 * (double)(n - 1) / (double)n;
        cvar += (cn - cmean) * (cn - cmean);
        dvar += (dj - dmean) * (dj - dmean);
        sxy += t * (dj - dmean);
        sxx += t * t;
        if (j >= q0) { tmax = fmax(tmax, dj); tmin = fmin(tmin, dj); }
        small += (dj < dmax - 2.0);
    }
    f[0] = (float)(log2((double)m) / 16.0);
    f[1] = (float)(log2((double)n) / 10.0);
    f[2] = (float)(cmax - cmin);
    f[3] = (float)sqrt(cvar / n);
    f[4] = (float)(dmax - dmin);
    f[5] = (float)sqrt(dvar / n);
    f[6] = (float)(sxx > 0 ? sxy / sxx : 0.0);
    f[7] = (float)(tmax - tmin);
    f[8] = (float)((double)small / (double)n);
    f[9] = (float)(dmin - log10(fmax(sqrt(fro / (double)n), 1e-300)));
}

// Proposal: logits of one feature vector -> class -> precision code.
__global__ void k_propose(const float* __restrict__ logits, int32_t* __restrict__ prec, float* __restrict__ probs) {
    if (threadIdx.x != 0) return;
    int best = 0;
    float mx = logits[0];
    for (int c = 1; c < MC; ++c)
        if (logits[c] > mx) { mx = logits[c]; best = c; }
    const int32_t map[MC] = {LSQ_FP8_E4M3, LSQ_BF16, LSQ_FP32, LSQ_FP64};
    *prec = map[best];
    if (probs) {
        float se = 0.0f;
        for (int c = 0; c < MC; ++c) se += expf(logits[c] - mx);
        for (int c = 0; c < MC; ++c) probs[c] = expf(logits[c] - mx) / se;
    }
}

// ---------------------------------------------------------------------------
// Judge: Hager's estimate of ||R^{-1}||_1 (R upper, FP32 copy), times ||R||_1.
// ---------------------------------------------------------------------------
__global__ void k_to_f32_upper(const double* __restrict__ R, int64_t n, int64_t ldr, float* __restrict__ Rf) {
    int64_t total = n * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = q % n, j = q / n;
        Rf[q] = i <= j ? __double2float_rn(R[i + j * ldr]) : 0.0f;
    }
}

// kappa_1(R) = ||R||_1 gamma (gamma ~ ||R^{-1}||_1) and the judgement
// u_p kappa_1(R) <= 1; a non-finite value or a timed-out solve rejects.
__global__ void k_judge_final(const float* __restrict__ rnorm, const float* __restrict__ gamma,
                              const int32_t* __restrict__ err, int prec, int32_t* __restrict__ accept,
                              double* __restrict__ kappa1) {
    const double k1 = (double)(*rnorm) * (double)(*gamma);
    const double u = prec == LSQ_FP8_E4M3 ? 0x1p-4 : prec == LSQ_BF16 ? 0x1p-8 : prec == LSQ_FP16 ? 0x1p-11
                   : prec == LSQ_FP32 ? 0x1p-24 : 0x1p-53;
    const bool finite = isfinite(k1) && k1 > 0.0 && *err == 0;
    *kappa1 = finite ? k1 : __longlong_as_double(0x7ff0000000000000ll);
    *accept = (finite && u * k1 <= 1.0) ? 1 : 0;
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
lsq_status launch_mlp_forward(const float* params, int d, int batch, const float* X, float* logits, cudaStream_t st) {
    size_t smem = sizeof(float) * (size_t)mlp_params(d);
    if (smem > 200 * 1024) return LSQ_ERR_ARG;
    if (smem > 48 * 1024) LSQ_CUDA_TRY(cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_mlp_forward<<<(unsigned)ceil_div(batch, 64), 64, smem, st>>>(params, d, batch, X, logits);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

// One row of np + 1 sums per MB samples.
size_t mlp_backward_ws_bytes(int d, int batch) {
    return align_up(sizeof(float) * (size_t)ceil_div(batch, MB) * (size_t)(mlp_params(d) + 1), 256) + 256;
}

lsq_status launch_mlp_backward(const float* params, int d, int batch, const float* X, const int32_t* labels,
                               float* grad, float* loss, void* ws, size_t ws_bytes, cudaStream_t st) {
    if (ws_bytes < mlp_backward_ws_bytes(d, batch) || !ws) return LSQ_ERR_NOMEM;
    const int64_t np = mlp_params(d);
    if (sizeof(float) * (size_t)np > 200 * 1024) return LSQ_ERR_ARG;
    float* part = (float*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    const int chunks = (int)ceil_div(batch, MB);
    LSQ_CUDA_TRY(cudaFuncSetAttribute(k_mlp_grad_part, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM));
    k_mlp_grad_part<<<(unsigned)chunks, MT, MLP_SMEM, st>>>(params, d, batch, X, labels, part);
    LSQ_LAUNCH_CHECK();
    k_mlp_reduce<<<(unsigned)ceil_div(np + 1, 32), 256, 0, st>>>(part, np, chunks, batch, grad, loss);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

lsq_status launch_adam(float* p, const float* g, float* m1, float* m2, int64_t count, float lr, float b1, float b2,
                       float eps, int step, cudaStream_t st) {
    float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
    k_adam<<<(unsigned)ceil_div(count, 256), 256, 0, st>>>(p, g, m1, m2, count, lr, b1, b2, eps, c1, c2);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

lsq_status launch_colnorm2(const double* A, int64_t m, int64_t n, int64_t lda, double* out, cudaStream_t st) {
    k_colnorm2<<<(unsigned)n, 256, 0, st>>>(A, m, lda, out);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

lsq_status launch_features_finish(const double* cn2, const double* Rs, int64_t ldr, int64_t m, int64_t n, float* f,
                                  cudaStream_t st) {
    k_features<<<1, 32, 0, st>>>(cn2, Rs, ldr, m, n, f);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

lsq_status launch_propose(const float* logits, int32_t* prec, float* probs, cudaStream_t st) {
    k_propose<<<1, 32, 0, st>>>(logits, prec, probs);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

size_t judge_ws_bytes(int64_t n) { return align_up(sizeof(float) * (size_t)n * n, 256) + 256 + hager_ws_bytes(n) + 256; }

lsq_status launch_judge(const double* Rs, int64_t n, int64_t ldr, int prec, int32_t* accept, double* kappa1, void* ws,
                        size_t ws_bytes, cudaStream_t st) {
    if (!ws || ws_bytes < judge_ws_bytes(n)) return LSQ_ERR_NOMEM;
    float* Rf = (float*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    char* small = (char*)Rf + align_up(sizeof(float) * (size_t)n * n, 256);
    float* rnorm = (float*)small;
    float* gam = (float*)(small + 4);
    int32_t* herr = (int32_t*)(small + 8);
    k_to_f32_upper<<<(unsigned)std::min<int64_t>(ceil_div(n * n, 256), 4096), 256, 0, st>>>(Rs, n, ldr, Rf);
    LSQ_LAUNCH_CHECK();
    lsq_status r;
    if ((r = launch_colnorm1_max(Rf, n, n, true, rnorm, st)) != LSQ_OK) return r;
    LSQ_CUDA_TRY(cudaMemsetAsync(herr, 0, sizeof(int32_t), st));
    if ((r = hager_inv_norm1(Rf, n, n, true, nullptr, gam, herr, small + 256, hager_ws_bytes(n), st)) != LSQ_OK)
        return r;
    k_judge_final<<<1, 1, 0, st>>>(rnorm, gam, herr, prec, accept, kappa1);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

int64_t mlp_param_count_host(int d) { return mlp_params(d); }
int mlp_num_features() { return NFEAT; }

}  // namespace lsq
