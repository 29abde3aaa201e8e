// Preconditioner of Alg. 1: thin QR of the sketch A_s (s x n) in FP32 or
// FP64 arithmetic, R only, then promotion to FP64 and removal of the
// column scaling.  Blocked Householder QR with the compact WY form
// (Schreiber & Van Loan 1989):
//   panel of QNB columns in a cluster of CTAs (Householder vectors as in
//   Golub & Van Loan Alg. 5.1.1, which maps x to +||x|| e1, so diag(R) >= 0),
//   the triangular factor T of  H_1...H_nb = I - V T V^T, and the trailing
//   update C <- (I - V T^T V^T) C as W = V^T C, C -= V (T^T W) in one fused
//   cluster kernel.
#include "common.cuh"
#include "kernels.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

namespace lsq {

constexpr int QNB = 32;        // panel width
constexpr int QPT = 512;       // panel threads

template <typename T>
__device__ __forceinline__ T block_sum(T v, T* red /* >= 32 */) {
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    T t = (T)0;
    for (int w = 0; w < nw; ++w) t += red[w];  // same order in every thread
    return t;
}

// Factor panel columns [k0, k0+nb) of W (s x n, ld), store v below the
// diagonal (v_j = 1 implicit), R on and above, beta[j]; then build T (nb x
// nb upper, ld QNB) and the explicit V (rows k0..s-1, ld ldv).
template <typename T>
__global__ void __launch_bounds__(QPT) k_qr_panel(T* __restrict__ W, int64_t ld, int64_t s, int64_t k0, int nb,
                                                  T* __restrict__ beta, T* __restrict__ Tm, T* __restrict__ V,
                                                  int64_t ldv) {
    __shared__ T red[32];
    __shared__ T wred[QPT / 32][QNB];
    __shared__ T wcol[QNB];
    __shared__ T sh_v1, sh_beta;
    __shared__ int sh_scale;
    __shared__ T Ys[QNB][QNB + 1];
    __shared__ T Vs[32][QNB + 1];
    __shared__ T Ts[QNB][QNB + 1];
    int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int jj = 0; jj < nb; ++jj) {
        int64_t j = k0 + jj;
        T* colj = W + j * ld;
        T sp = (T)0;
        for (int64_t i = j + 1 + tid; i < s; i += QPT) sp = fma(colj[i], colj[i], sp);
        T sigma = block_sum<T>(sp, red);
        if (tid == 0) {
            T x1 = colj[j];
            T mu, b, v1 = (T)1;
            int scale = 0;
            if (sigma == (T)0) {
                mu = fabs(x1);
                b = x1 >= (T)0 ? (T)0 : (T)2;
            } else {
                mu = sqrt(x1 * x1 + sigma);
                v1 = x1 <= (T)0 ? x1 - mu : -sigma / (x1 + mu);
                b = (T)2 * v1 * v1 / (sigma + v1 * v1);
                scale = 1;
            }
            colj[j] = mu;
            beta[j] = b;
            sh_v1 = v1;
            sh_beta = b;
            sh_scale = scale;
        }
        __syncthreads();
        T v1 = sh_v1, b = sh_beta;
        if (sh_scale)
            for (int64_t i = j + 1 + tid; i < s; i += QPT) colj[i] = colj[i] / v1;
        __syncthreads();
        int rem = nb - jj - 1;
        if (rem > 0 && b != (T)0) {
            T acc[QNB];
#pragma unroll
            for (int c = 0; c < QNB; ++c) acc[c] = (T)0;
            // w_c = W[j][c] + sum_{i>j} v_i W[i][c]
            for (int64_t i = j + tid; i < s; i += QPT) {
                T vi = (i == j) ? (T)1 : colj[i];
#pragma unroll
                for (int c = 0; c < QNB; ++c)
                    if (c < rem) acc[c] = fma(vi, W[i + (j + 1 + c) * ld], acc[c]);
            }
#pragma unroll
            for (int c = 0; c < QNB; ++c) {
                T v = acc[c];
                for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (lane == 0) wred[warp][c] = v;
            }
            __syncthreads();
            if (tid < rem) {
                T t = (T)0;
                for (int w = 0; w < QPT / 32; ++w) t += wred[w][tid];
                wcol[tid] = b * t;
            }
            __syncthreads();
            for (int64_t i = j + tid; i < s; i += QPT) {
                T vi = (i == j) ? (T)1 : colj[i];
                for (int c = 0; c < rem; ++c) {
                    T* p = &W[i + (j + 1 + c) * ld];
                    *p = fma(-wcol[c], vi, *p);
                }
            }
        }
        __syncthreads();
    }
    // Y = V^T V over rows k0..s-1 (explicit zeros above, ones on the diagonal)
    int p = tid >> 5, q = lane;  // 16 x 32 threads cover Y in two passes
    T y0 = (T)0, y1 = (T)0;
    for (int64_t r0 = k0; r0 < s; r0 += 32) {
        for (int e = tid; e < 32 * QNB; e += QPT) {
            int rr = e % 32, cc = e / 32;
            int64_t i = r0 + rr;
            T v = (T)0;
            if (cc < nb && i < s) {
                int64_t diag = k0 + cc;
                v = i < diag ? (T)0 : (i == diag ? (T)1 : W[i + diag * ld]);
            }
            Vs[rr][cc] = v;
        }
        __syncthreads();
#pragma unroll 8
        for (int rr = 0; rr < 32; ++rr) {
            y0 = fma(Vs[rr][p], Vs[rr][q], y0);
            y1 = fma(Vs[rr][p + 16], Vs[rr][q], y1);
        }
        // explicit V for the trailing contractions
        for (int e = tid; e < 32 * QNB; e += QPT) {
            int rr = e % 32, cc = e / 32;
            int64_t i = r0 + rr;
            if (i < s) V[(i - k0) + cc * ldv] = Vs[rr][cc];
        }
        __syncthreads();
    }
    Ys[p][q] = y0;
    Ys[p + 16][q] = y1;
    __syncthreads();
    // T: T[j][j] = beta_j, T[0:j, j] = -beta_j T[0:j, 0:j] Y[0:j, j]
    if (warp == 0) {
        for (int c = 0; c < QNB; ++c) Ts[lane][c] = (T)0;
        __syncwarp();
        for (int jj = 0; jj < nb; ++jj) {
            T bj = beta[k0 + jj];
            T t = (T)0;
            if (lane < jj)
                for (int qq = lane; qq < jj; ++qq) t = fma(Ts[lane][qq], Ys[qq][jj], t);
            __syncwarp();
            if (lane < jj) Ts[lane][jj] = -bj * t;
            if (lane == jj) Ts[jj][jj] = bj;
            __syncwarp();
        }
        for (int c = 0; c < QNB; ++c) Tm[lane + c * QNB] = Ts[lane][c];
    }
}

// Same panel factorization by a cluster of QCL CTAs that keep the panel in
// shared memory: CTA r owns rows [r R, (r+1) R) of the panel (local leading
// dimension Rp = R | 1, odd, so that lanes reading different columns of one
// row hit different banks).  Per column j each CTA computes, in one pass over
// its rows below the diagonal, sigma = sum x_i^2 and d_c = sum x_i a_c[i] for
// every later column c (warp = row group, lane = column); the partials and
// the diagonal row (x1, a_c[j], from its owner) are pushed into every CTA's
// shared memory, and after ONE cluster barrier every CTA sums them in rank
// order and gets identical Householder scalars and
//   v^T a_c = a_c[j] + d_c / v1,   w_c = beta v^T a_c
// (v = [1; x(2:)/v1]).  Slots alternate between two buffers by column parity:
// a CTA can only write a buffer again after the next barrier, which every CTA
// reaches after reading it.
constexpr int QCT = 256;
constexpr int QKG = QCT / 64;  // row groups of the previous-panel product (64 threads each)

constexpr int QRC = 32;   // panel rows per warp kept in registers, FP64
constexpr int QRC32 = 64;  // FP32

// The register forms keep u = [v1; x] unscaled: w_c / v1 and the products
// u_i^T u_j stay in range while |v1| lies within 2^+-400, FP32 2^+-45 (columns
// whose squares are in range have norms between about 2^-538 and 2^512, FP32
// 2^-74 and 2^64).  Outside, a column's u is scaled by 1 / v1 before it is used.
// On the exponent field: an FP64 comparison costs a warp 64 cycles.
__device__ __forceinline__ bool qr_far(double av) {
    return (unsigned)(((int)(__double_as_longlong(av) >> 52) & 0x7ff) - (1023 - 400)) > 800u;
}
__device__ __forceinline__ bool qr_far(float av) {
    return (unsigned)((int)(__float_as_uint(av) >> 23 & 0xff) - (127 - 45)) > 90u;
}

// 4 consecutive values from 16-byte aligned shared memory
__device__ __forceinline__ void load4(const float* p, float (&o)[4]) {
    const float4 v = *(const float4*)p;
    o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
}
__device__ __forceinline__ void load4(const double* p, double (&o)[4]) {
    const double2 v0 = *(const double2*)p, v1 = *(const double2*)(p + 2);
    o[0] = v0.x, o[1] = v0.y, o[2] = v1.x, o[3] = v1.y;
}

__device__ __forceinline__ void store4(float* p, float a, float b, float c, float d) { *(float4*)p = make_float4(a, b, c, d); }

// sum_{q < QCL} x[q * stride], pairwise (the same order in every CTA)
template <typename T, int QCL>
__device__ __forceinline__ T tree_sum(const T* x, int stride) {
    T v[QCL];
#pragma unroll
    for (int q = 0; q < QCL; ++q) v[q] = x[q * stride];
#pragma unroll
    for (int h = QCL / 2; h >= 1; h >>= 1)
#pragma unroll
        for (int q = 0; q < h; ++q) v[q] += v[q + h];
    return v[0];
}

// FP64 reciprocal square root and reciprocal for the Householder scalars: an
// FP32 estimate (about 23 bits; operands and estimates moved between FP64 and
// FP32 on the bit patterns, the exponent split off so that any normal FP64
// operand works) refined in FP64, by one third-order step (sqrt) and by two
// Newton steps (reciprocal).  A few units in the last place, 4 to 5 dependent
// FP64 operations each, where the library's correctly rounded sqrt and division
// cost ~650 cycles apiece on this GPU and formed a chain of four per column.
// Subnormal, infinite and NaN operands take the library functions.
__device__ __forceinline__ bool qr_normal(double d) {
    const int e = (int)(((unsigned long long)__double_as_longlong(d) >> 52) & 0x7ff);
    return e != 0 && e != 0x7ff;
}

// 1 / sqrt(d), d > 0
__device__ __forceinline__ double qr_rsqrt(double d) {
    if (!qr_normal(d)) return 1.0 / sqrt(d);
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int e2 = ((int)(b >> 52) - 1023) & ~1;                           // d = m 2^e2, m in [1, 4)
    const unsigned long long mb = b - ((unsigned long long)(long long)e2 << 52);
    const double m = __longlong_as_double((long long)mb);
    const uint32_t fb = (uint32_t)((((mb >> 52) & 0x7ff) - 1023 + 127) << 23) | (uint32_t)((mb >> 29) & 0x7fffff);
    const uint32_t yb = __float_as_uint(rsqrtf(__uint_as_float(fb)));
    double y = __longlong_as_double((long long)(((unsigned long long)((yb >> 23) - 127 + 1023) << 52) |
                                                ((unsigned long long)(yb & 0x7fffff) << 29)));
    const double e = fma(-(m * y), y, 1.0);
    y = fma(y * e, fma(0.375, e, 0.5), y);
    return __longlong_as_double(__double_as_longlong(y) - ((long long)(e2 / 2) << 52));
}

// 1 / d, d > 0 and 1 / d normal
__device__ __forceinline__ double qr_rcp(double d) {
    if (!qr_normal(d)) return 1.0 / d;
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int ed = (int)(b >> 52) - 1023;
    const double m = __longlong_as_double((long long)((b & 0x000fffffffffffffull) | (1023ull << 52)));  // [1, 2)
    const uint32_t fb = (127u << 23) | (uint32_t)((b >> 29) & 0x7fffff);
    const uint32_t yb = __float_as_uint(__frcp_rn(__uint_as_float(fb)));
    double y = __longlong_as_double((long long)(((unsigned long long)((yb >> 23) - 127 + 1023) << 52) |
                                                ((unsigned long long)(yb & 0x7fffff) << 29)));
    y = fma(fma(-m, y, 1.0), y, y);
    y = fma(fma(-m, y, 1.0), y, y);
    return ed < 1021 ? __longlong_as_double(__double_as_longlong(y) - ((long long)ed << 52)) : 1.0 / d;
}

// QCL: CTAs per cluster (1 to 16; 16 is non-portable, else 8).  Dynamic shared
// memory: the local panel (Rp x QNB) and, in the fused form, the previous panel's
// reflector rows and the partial products behind it.
template <typename T, int QCL>
__global__ void __launch_bounds__(QCT)
    k_qr_panel_cl(T* __restrict__ W, int64_t ld, int64_t s, int64_t k0, int nb, T* __restrict__ beta_out,
                  T* __restrict__ Tm, T* __restrict__ V, int64_t ldv, const T* __restrict__ Vp, int64_t ldvp,
                  const T* __restrict__ Tp) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    extern __shared__ __align__(16) unsigned char cl_raw[];
    T* P = reinterpret_cast<T*>(cl_raw);  // local panel, column-major, ld Rp
    __shared__ T all_part[2][QCL][QNB];  // per rank: d_c (sigma at c = j)
    __shared__ T all_row[2][QNB];        // the diagonal row: x1 at j, a_c[j] at c > j
    __shared__ T part[QCT / 32][QNB];
    __shared__ T Ts[QNB][QNB + 1];
    __shared__ T bsh[QNB];
    __shared__ T Wr[QNB][QNB + 1];  // this CTA's partial V_p^T C (read by the whole cluster)
    __shared__ T Ysm[QNB][QNB + 1];  // rank 0: Y = V^T V (strictly upper part), built column by column
    // FP32, per warp: u_jj and the next column on its rows (by the column's parity)
    __shared__ __align__(16) T bcx[2][QCT / 32][std::is_same<T, float>::value ? QRC32 : 4];
    __shared__ T rowbuf[QNB];                      // row jj of the panel (owning CTA)
    __shared__ T scal_sh[4];                       // FP64: mu, b, v1, 1 / v1 of the column (warp 0)
    __shared__ T wc_sh[QNB], f_sh[QNB];            // FP64: w_c and w_c / v1 of the column (warp 0)
    __shared__ int scale_sh;
    const int rank = (int)cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rows = (int)(s - k0);
    const int R = (rows + QCL - 1) / QCL;
    const int Rp = R | 1;
    const int r0 = rank * R;
    const int nloc = r0 < rows ? min(R, rows - r0) : 0;
    T* Yall = P + (int64_t)Rp * QNB;  // fused form only: the staging area behind the panel
    const int chunk = (R + (QCT / 32) - 1) / (QCT / 32);
    const int g0 = warp * chunk, g1 = min(nloc, g0 + chunk);  // this warp's rows
    // loads of all columns of a row in flight before the stores
    for (int i = tid; i < R; i += QCT) {
        T x[QNB];
#pragma unroll
        for (int c = 0; c < QNB; ++c) x[c] = (i < nloc && c < nb) ? W[(k0 + r0 + i) + (k0 + c) * ld] : (T)0;
#pragma unroll
        for (int c = 0; c < QNB; ++c) P[c * Rp + i] = x[c];
    }
    __syncthreads();
    // A CTA may write into another CTA's shared memory only once that CTA is
    // running: without a previous panel (below) the first column's exchange
    // is the first such write, so the cluster meets here first.
    if (Vp == nullptr) cluster.sync();
    if (Vp != nullptr) {
        // The previous panel's reflectors applied to this panel's columns,
        // C <- (I - V_p T_p^T V_p^T) C over rows k0 - QNB .. s - 1 (V_p: QNB
        // columns, ld ldvp, row 0 at k0 - QNB): this CTA's rows in shared
        // memory, the QNB rows above the panel by rank 0 from global memory.
        T* Vl = Yall;                      // [QNB][Rp]: rows QNB + r0 + i of V_p
        T* Wk = Yall + (int64_t)QNB * Rp;    // [QKG][QNB][QNB + 1] row-group partials, then W and W2
        T* Ct = Wk + QKG * QNB * (QNB + 1);  // rank 0: [QNB][QNB + 1] the rows above, then their V_p rows
        T* Vt = Ct + QNB * (QNB + 1);
        for (int i = tid; i < R; i += QCT) {
            T x[QNB];
#pragma unroll
            for (int c = 0; c < QNB; ++c) x[c] = i < nloc ? Vp[(QNB + r0 + i) + c * ldvp] : (T)0;
#pragma unroll
            for (int c = 0; c < QNB; ++c) Vl[c * Rp + i] = x[c];
        }
        if (rank == 0 && tid < QNB) {
            T x[QNB], v[QNB];
#pragma unroll
            for (int c = 0; c < QNB; ++c) {
                x[c] = c < nb ? W[(k0 - QNB + tid) + (k0 + c) * ld] : (T)0;
                v[c] = Vp[tid + c * ldvp];
            }
#pragma unroll
            for (int c = 0; c < QNB; ++c) {
                Ct[tid * (QNB + 1) + c] = x[c];
                Vt[tid * (QNB + 1) + c] = v[c];
            }
        }
        __syncthreads();
        {
            // partial W = V_p^T C: QKG row groups of 64 threads, 4 x 4 blocks
            const int kg = tid >> 6, tl = tid & 63, tp = tl & 7, tq = tl >> 3;
            const int span = (R + QKG - 1) / QKG;
            const int i0 = kg * span, i1 = min(nloc, i0 + span);
            T acc[4][4];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
#pragma unroll 4
            for (int i = i0; i < i1; ++i) {
                T v[4], c[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) v[a] = Vl[(4 * tp + a) * Rp + i];
#pragma unroll
                for (int b = 0; b < 4; ++b) c[b] = P[(4 * tq + b) * Rp + i];
#pragma unroll
                for (int a = 0; a < 4; ++a)
#pragma unroll
                    for (int b = 0; b < 4; ++b) acc[a][b] = fma(v[a], c[b], acc[a][b]);
            }
            if (rank == 0)
#pragma unroll 4
                for (int i = kg * (QNB / QKG); i < (kg + 1) * (QNB / QKG); ++i) {
                    T v[4], c[4];
#pragma unroll
                    for (int a = 0; a < 4; ++a) v[a] = Vt[i * (QNB + 1) + 4 * tp + a];
#pragma unroll
                    for (int b = 0; b < 4; ++b) c[b] = Ct[i * (QNB + 1) + 4 * tq + b];
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) acc[a][b] = fma(v[a], c[b], acc[a][b]);
                }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) Wk[(kg * QNB + 4 * tp + a) * (QNB + 1) + 4 * tq + b] = acc[a][b];
        }
        __syncthreads();
        for (int q = tid; q < QNB * QNB; q += QCT) {
            const int p = q >> 5, c = q & 31;
            Wr[p][c] = tree_sum<T, QKG>(&Wk[p * (QNB + 1) + c], QNB * (QNB + 1));
        }
        cluster.sync();
        // W: the partials of every rank in rank order (the column loop's
        // cluster barriers keep them in place until every CTA has read them)
        T* Wf = Wk;                     // [QNB][QNB + 1]
        T* W2 = Wk + QNB * (QNB + 1);   // [QNB][QNB]
        for (int q = tid; q < QNB * QNB; q += QCT) {
            const int p = q >> 5, c = q & 31;
            T v[QCL];
#pragma unroll
            for (int r = 0; r < QCL; ++r) v[r] = cluster.map_shared_rank(&Wr[0][0], r)[p * (QNB + 1) + c];
#pragma unroll
            for (int h = QCL / 2; h >= 1; h >>= 1)
#pragma unroll
                for (int r = 0; r < h; ++r) v[r] += v[r + h];
            Wf[p * (QNB + 1) + c] = v[0];
        }
        for (int q = tid; q < QNB * QNB; q += QCT) Ts[q & 31][q >> 5] = Tp[q];  // Ts[k][p] = T_p[k, p]
        __syncthreads();
        {
            // T_p^T W: rows warp, warp + 8, ... (T_p is zero below its diagonal)
            T w[QNB * 32 / QCT];
#pragma unroll
            for (int e = 0; e < QNB * 32 / QCT; ++e) w[e] = (T)0;
#pragma unroll 8
            for (int kk = 0; kk < QNB; ++kk) {
                const T f = Wf[kk * (QNB + 1) + lane];
#pragma unroll
                for (int e = 0; e < QNB * 32 / QCT; ++e) w[e] = fma(Ts[kk][warp + e * (QCT / 32)], f, w[e]);
            }
#pragma unroll
            for (int e = 0; e < QNB * 32 / QCT; ++e) W2[(warp + e * (QCT / 32)) * QNB + lane] = w[e];
        }
        __syncthreads();
        // C -= V_p W2, one row per thread; rank 0's rows above the panel follow its own
        const int nrow = nloc + (rank == 0 ? QNB : 0);
        for (int i = tid; i < nrow; i += QCT) {
            const bool own = i < nloc;
            T* cp = own ? P + i : Ct + (i - nloc) * (QNB + 1);
            const T* vp = own ? Vl + i : Vt + (i - nloc) * (QNB + 1);
            const int st = own ? Rp : 1;
            T a[QNB];
#pragma unroll
            for (int c = 0; c < QNB; ++c) a[c] = cp[c * st];
#pragma unroll 2
            for (int p = 0; p < QNB; ++p) {
                const T v = vp[p * st];
#pragma unroll
                for (int c = 0; c < QNB; c += 4) {
                    T w[4];
                    load4(W2 + p * QNB + c, w);
#pragma unroll
                    for (int e = 0; e < 4; ++e) a[c + e] = fma(-v, w[e], a[c + e]);
                }
            }
            if (own) {
#pragma unroll
                for (int c = 0; c < QNB; ++c) P[c * Rp + i] = a[c];
            } else {
#pragma unroll
                for (int c = 0; c < QNB; ++c)
                    if (c < nb) W[(k0 - QNB + i - nloc) + (k0 + c) * ld] = a[c];
            }
        }
        __syncthreads();
    }
    // partial dots of column j over this warp's rows strictly below row j
    // (lane = column c >= j): sum x_j[i] a_c[i]; sigma at c = j
    auto dots = [&](int j) -> T {
        if (!(lane >= j && lane < nb)) return (T)0;
        const T* x = P + j * Rp;
        const T* a = P + lane * Rp;
        T a0 = (T)0, a1 = (T)0, a2 = (T)0, a3 = (T)0;
        int i = max(max(j + 1 - r0, 0), g0);
        for (; i + 4 <= g1; i += 4) {
            a0 = fma(x[i], a[i], a0);
            a1 = fma(x[i + 1], a[i + 1], a1);
            a2 = fma(x[i + 2], a[i + 2], a2);
            a3 = fma(x[i + 3], a[i + 3], a3);
        }
        for (; i < g1; ++i) a0 = fma(x[i], a[i], a0);
        return (a0 + a1) + (a2 + a3);
    };
    // After column j: lanes c > j the partial dots of column j + 1 (rows
    // below j + 1), lanes i < j the partial Y[i][j] = v_i^T v_j = v_i[j] +
    // sum_{r > j} v_i[r] v_j[r] (rows of this warp) in the same pass: both
    // read one broadcast column (x_{j+1} or v_j) against the lane's own.
    auto dots_y = [&](int j) -> T {
        const int jn = j + 1;
        const bool ylane = lane < j, dlane = lane >= jn && lane < nb && jn < nb;
        if (!(ylane || dlane)) return (T)0;
        const T* x = P + (ylane ? j : jn) * Rp;
        const T* a = P + lane * Rp;
        T a0 = (T)0, a1 = (T)0, a2 = (T)0, a3 = (T)0;
        int i = max(max(jn + 1 - r0, 0), g0);
        for (; i + 4 <= g1; i += 4) {
            a0 = fma(x[i], a[i], a0);
            a1 = fma(x[i + 1], a[i + 1], a1);
            a2 = fma(x[i + 2], a[i + 2], a2);
            a3 = fma(x[i + 3], a[i + 3], a3);
        }
        for (; i < g1; ++i) a0 = fma(x[i], a[i], a0);
        T acc2 = (a0 + a1) + (a2 + a3);
        if (ylane) {
            const int lj = j - r0, lj1 = jn - r0;
            if (lj1 >= g0 && lj1 < g1) acc2 = fma(x[lj1], a[lj1], acc2);  // row j + 1
            if (lj >= g0 && lj < g1) acc2 += a[lj];                        // row j: v_j = 1 there
        }
        return acc2;
    };
    // Every per-row step (scaling of v, the update, the next column's dots)
    // stays within the warp's own rows, so a column needs one CTA barrier
    // (the partial dots) and one cluster barrier (their exchange), and for
    // FP64 a second CTA barrier (the scalars from warp 0).
    // Column jj's exchange: the partials of every warp summed (part), pushed
    // with the diagonal row (rowv, from the CTA that owns row jj) into every
    // CTA; after the cluster barrier every CTA forms the same Householder
    // scalars, w_c for each column and (rank 0) column jj - 1 of Y.
    struct Scal {
        T mu, b, v1, rv1, wc;  // R's diagonal entry, beta, v's leading entry before scaling, its reciprocal, w_c
        T f;                   // w_c / v1 (register forms), w_c when far
        T rc;                  // FP32 register form: R[jj][c]
        bool scale;
        bool far;              // register forms: u is scaled by 1 / v1 (qr_far)
    };
    // FP64: the sign of v1 is that of x1 (no cancellation, no case distinction;
    // R's diagonal entry is then -sign(x1) mu, and k_qr_extract makes the
    // diagonal positive by the signs of R's rows), and with mu = sqrt(x1^2 +
    // sigma), |v1| = |x1| + mu:  sigma + v1^2 = 2 mu |v1|, so that beta =
    // 2 v1^2 / (sigma + v1^2) = |v1| / mu needs 1/mu and 1/|v1| only.
    auto scalars64 = [&](int jj, int buf, int owner) -> Scal {
        Scal sc;
        // lane > jj: d_c of this column; lane jj: sigma; lane < jj - 1: u_i^T u_{jj-1}
        const T dsum = tree_sum<T, QCL>(&all_part[buf][0][lane], QNB);
        const T sigma = __shfl_sync(0xffffffffu, dsum, jj);
        const T x1 = all_row[buf][jj];
        const T s2 = fma(x1, x1, sigma);
        sc.scale = sigma != (T)0;
        sc.mu = x1;
        sc.b = (T)0;
        sc.v1 = (T)1;
        sc.rv1 = (T)1;
        sc.wc = sc.f = (T)0;
        sc.far = false;
        if (sc.scale) {
            const T y = (T)qr_rsqrt((double)s2);
            T mu = s2 * y;
            mu = fma((T)0.5 * y, fma(-mu, mu, s2), mu);  // to the last bit
            const T av = fabs(x1) + mu;
            const T r = (T)qr_rcp((double)av);
            sc.v1 = x1 < (T)0 ? -av : av;
            sc.rv1 = x1 < (T)0 ? -r : r;
            sc.mu = x1 < (T)0 ? mu : -mu;
            sc.far = qr_far(av);
            // tau = 2 / u^T u = 1 / (mu |v1|) and beta = |v1| / mu, each corrected
            // once: their errors are common to all rows, so that they would
            // show in R's where those of single entries average out
            T tau = y * r;
            tau = fma(fma(-(tau * mu), av, (T)1), tau, tau);
            T bt = av * y;
            bt = fma(fma(-bt, mu, av), y, bt);
            sc.b = bt;
            if (lane > jj && lane < nb) {
                const T ac = all_row[buf][lane];
                sc.wc = bt * fma(dsum, sc.rv1, ac);
                sc.f = sc.far ? sc.wc : tau * fma(sc.v1, ac, dsum);
            }
        }
        if (rank == 0 && warp == 0 && lane + 1 < jj) Ysm[lane][jj - 1] = dsum;
        if (tid == 0) bsh[jj] = sc.b;  // identical in every CTA of the cluster
        if (rank == owner && tid == 0) beta_out[k0 + jj] = sc.b;
        return sc;
    };
    // The same in FP32, by IEEE operations: two divisions after the root, and
    // w_c and w_c / v1 need none.
    auto scalars32 = [&](int jj, int buf, int owner) -> Scal {
        Scal sc;
        const T dsum = tree_sum<T, QCL>(&all_part[buf][0][lane], QNB);
        const T sigma = __shfl_sync(0xffffffffu, dsum, jj);
        const T x1 = all_row[buf][jj], ac = all_row[buf][lane];
        sc.scale = sigma != (T)0;
        sc.mu = x1;
        sc.b = (T)0;
        sc.v1 = (T)1;
        sc.rv1 = (T)1;
        sc.wc = sc.f = (T)0;
        sc.far = false;
        if (sc.scale) {
            // beta = 2 / v^T v from 1 / v1 as it is used: its error is common to
            // all rows and would show in R
            const T mu = sqrt(fma(x1, x1, sigma)), av = fabs(x1) + mu, rv = (T)1 / av;
            sc.b = (T)2 / fma(sigma * rv, rv, (T)1);
            sc.v1 = x1 < (T)0 ? -av : av;
            sc.rv1 = x1 < (T)0 ? -rv : rv;
            sc.mu = x1 < (T)0 ? mu : -mu;
            sc.far = qr_far(av);
            if (lane > jj && lane < nb) {
                sc.wc = sc.b * fma(dsum, sc.rv1, ac);
                sc.f = sc.far ? sc.wc : sc.wc * sc.rv1;
                sc.rc = ac - sc.wc;
            }
        }
        if (rank == 0 && warp == 0 && lane + 1 < jj) Ysm[lane][jj - 1] = dsum;
        if (tid == 0) bsh[jj] = sc.b;
        if (rank == owner && tid == 0) beta_out[k0 + jj] = sc.b;
        return sc;
    };
    // The Householder scalars of column jj from the exchanged partials (the
    // same in every CTA) and, per lane c > jj, w_c.
    auto scalars = [&](int jj, int buf, int owner) -> Scal {
        Scal sc;
        const T sigma = tree_sum<T, QCL>(&all_part[buf][0][jj], QNB);
        const T x1 = all_row[buf][jj];
        sc.v1 = (T)1;
        sc.rv1 = (T)1;
        sc.scale = sc.far = false;
        if (sigma == (T)0) {
            sc.mu = fabs(x1);
            sc.b = x1 >= (T)0 ? (T)0 : (T)2;
        } else {
            sc.mu = sqrt(x1 * x1 + sigma);
            sc.v1 = x1 <= (T)0 ? x1 - sc.mu : -sigma / (x1 + sc.mu);
            sc.b = (T)2 * sc.v1 * sc.v1 / (sigma + sc.v1 * sc.v1);
            // v is scaled by a reciprocal formed here, in parallel with b
            // (an FP64 division costs ~650 cycles on this GPU)
            sc.rv1 = (T)1 / sc.v1;
            sc.scale = true;
        }
        // lane > jj: d_c of this column; lane < jj - 1: Y[lane][jj - 1] of the previous one
        const T dsum = tree_sum<T, QCL>(&all_part[buf][0][lane], QNB);
        sc.wc = (T)0;
        if (lane > jj && lane < nb) sc.wc = sc.b * (all_row[buf][lane] + (sc.scale ? dsum / sc.v1 : (T)0));
        if (rank == 0 && warp == 0 && lane + 1 < jj) Ysm[lane][jj - 1] = dsum;
        if (tid == 0) bsh[jj] = sc.b;  // identical in every CTA of the cluster
        if (rank == owner && tid == 0) beta_out[k0 + jj] = sc.b;
        return sc;
    };
    auto exchange = [&](int jj, T acc, const T* rowsrc, int rowstride, bool unscaled = false) -> Scal {
        const int buf = jj & 1;
        const int owner = (int)(jj / R);
        part[warp][lane] = acc;
        __syncthreads();
        if (warp == 0) {
            const T t = tree_sum<T, QCT / 32>(&part[0][lane], QNB);
            for (int q = 0; q < QCL; ++q) *cluster.map_shared_rank(&all_part[buf][rank][lane], q) = t;
            if (rank == owner) {
                const T rv = rowsrc[lane * rowstride];
                for (int q = 0; q < QCL; ++q) *cluster.map_shared_rank(&all_row[buf][lane], q) = rv;
            }
        }
        cluster.sync();
        Scal sc;
        if constexpr (std::is_same<T, double>::value) {
            // FP64 instructions issue at a small fraction of the FP32 rate: the
            // scalars and the columns' w_c are formed once per CTA, by warp 0
            // (every warp forming them kept the FP64 pipe 73 % busy on a panel
            // of few rows), and read by the other warps from shared memory.
            if (warp == 0) {
                sc = scalars64(jj, buf, owner);
                if (lane == 0) {
                    scal_sh[0] = sc.mu;
                    scal_sh[1] = sc.b;
                    scal_sh[2] = sc.v1;
                    scal_sh[3] = sc.rv1;
                    scale_sh = (sc.scale ? 1 : 0) | (sc.far ? 2 : 0);
                }
                wc_sh[lane] = sc.wc;
                f_sh[lane] = sc.f;
            }
            __syncthreads();
            sc.mu = scal_sh[0];
            sc.b = scal_sh[1];
            sc.v1 = scal_sh[2];
            sc.rv1 = scal_sh[3];
            sc.scale = (scale_sh & 1) != 0;
            sc.far = (scale_sh & 2) != 0;
            sc.wc = wc_sh[lane];
            sc.f = f_sh[lane];
            return sc;
        }
        return unscaled ? scalars32(jj, buf, owner) : scalars(jj, buf, owner);
    };
    T acc;
    T ysc0 = (T)1, ysc1 = (T)1;  // scales of lane i's entry of Y's last column
    bool done = false;  // columns kept in registers
    if constexpr (std::is_same<T, double>::value) {
      if (chunk <= QRC) {
        // FP64: each thread keeps its column's QRC rows of this warp in
        // registers; per column every lane of a warp takes the raw column jj
        // from lane jj and, after the update, column jj + 1 from lane jj + 1 by
        // shuffles, and forms v, the update and the next dots itself (no
        // divergent single-lane phases, no shared-memory round trips).
        // Measured: the FP64 path 6.2 -> 23.5 solves/s; FP32 broadcasts through
        // shared memory below, which is faster there (3.07 against 4.55 ms per solve).
        // The loops run over QR = 4, 8, ... 32 rows per lane, the fewest that hold
        // the warp's rows: the FP64 pipe takes 16 cycles an instruction and SM, so
        // masked rows are not free (a panel's column costs ~11 thousand cycles
        // with 32 rows per lane, in update and dots alone).
        auto f64_cols = [&](auto qr_tag) {
            constexpr int QR = decltype(qr_tag)::value;
            T a[QR];
#pragma unroll
            for (int q = 0; q < QR; ++q) a[q] = g0 + q < g1 ? P[lane * Rp + g0 + q] : (T)0;
            const int gr0 = r0 + g0;  // global row (from k0) of a[0]
            const int nv = g1 - g0;   // valid rows of this warp (<= 0: none)
            auto row_of = [&](int row) -> T {
                T v = (T)0;
#pragma unroll
                for (int q = 0; q < QR; ++q)
                    if (gr0 + q == row && q < nv) v = a[q];
                return v;
            };
            // column c below row `row` on this warp's rows, from lane c
            // The columns stay as they are in registers: with u = [v1; x] (not
            // scaled to a unit leading entry) the update is a_c -= (w_c / v1) u and
            // u_i^T u_j gives Y up to the scales 1 / v1, so that a column costs two
            // FP64 operations per row and lane (three with v formed by every
            // lane); lane c keeps its own 1 / v1 and R_cc and applies them at the
            // end.
            T xn[QR];
            T myscale = (T)1, myR = (T)0, rprev = (T)1;
            auto column_below = [&](int c, int row) {
#pragma unroll
                for (int q = 0; q < QR; ++q) {
                    const T x = __shfl_sync(0xffffffffu, a[q], c);
                    xn[q] = (q < nv && gr0 + q > row) ? x : (T)0;
                }
            };
            // Y[i][j] = v_i^T v_j from u_i^T u_j (lane i; rank 0, warp 0)
            auto scale_y = [&](int j) {
                if (rank == 0 && warp == 0 && lane < j) Ysm[lane][j] *= myscale * rprev;
            };
            column_below(0, 0);
            if (0 >= gr0 && 0 < gr0 + nv) rowbuf[lane] = row_of(0);
            {
                T s4[4] = {(T)0, (T)0, (T)0, (T)0};  // 4 chains of 8 FMAs
#pragma unroll
                for (int q = 0; q < QR; ++q) s4[q & 3] = fma(xn[q], a[q], s4[q & 3]);
                acc = lane < nb ? (s4[0] + s4[1]) + (s4[2] + s4[3]) : (T)0;
            }
            // column jj after its exchange; FAR: u scaled by 1 / v1 where needed
            auto column = [&](int jj, const Scal& sc, auto far_tag) {
                constexpr bool FAR = decltype(far_tag)::value;
                if (jj > 0) scale_y(jj - 1);
                // u_jj on this warp's rows: 0 above row jj, v1 on it, x below
                T u[QR];
#pragma unroll
                for (int q = 0; q < QR; ++q) {
                    const T x = __shfl_sync(0xffffffffu, a[q], jj);
                    const int gr = gr0 + q;
                    u[q] = (gr < jj || q >= nv) ? (T)0 : (gr == jj ? sc.v1 : x);
                }
                if (FAR && sc.far) {
#pragma unroll
                    for (int q = 0; q < QR; ++q) u[q] *= sc.rv1;
                }
                if (lane == jj) {
                    myscale = sc.rv1;
                    myR = sc.mu;
                }
                rprev = FAR && sc.far ? (T)1 : sc.rv1;
                // later columns: a_c -= w_c v = (w_c / v1) u
                const bool upd = lane > jj && lane < nb && sc.b != (T)0;
                const T f = sc.f;
                if (upd) {
#pragma unroll
                    for (int q = 0; q < QR; ++q) a[q] = fma(-f, u[q], a[q]);
                }
                const int jn = jj + 1;
                if (jn < nb) {
                    column_below(jn, jn);
                    if (jn >= gr0 && jn < gr0 + nv) rowbuf[lane] = row_of(jn);
                }
                // lanes c > jj: dots of column jj + 1; lanes i < jj: u_i^T u_jj
                const bool ylane = lane < jj, dlane = lane >= jn && lane < nb && jn < nb;
                T s4[4] = {(T)0, (T)0, (T)0, (T)0};
#pragma unroll
                for (int q = 0; q < QR; ++q) s4[q & 3] = fma(ylane ? u[q] : xn[q], a[q], s4[q & 3]);
                acc = (ylane || dlane) ? (s4[0] + s4[1]) + (s4[2] + s4[3]) : (T)0;
            };
            // from the first far column on in a loop of its own: the branch alone
            // cost a panel of few rows 5 %
            int jj = 0;
            Scal sc;
            for (; jj < nb; ++jj) {
                sc = exchange(jj, acc, rowbuf, 1);
                if (sc.far) break;
                column(jj, sc, std::false_type{});
            }
            while (jj < nb) {
                column(jj, sc, std::true_type{});
                if (++jj < nb) sc = exchange(jj, acc, rowbuf, 1);
            }
            ysc0 = myscale * rprev;  // of Y's last column, formed below
            // R on and above the diagonal, v below it
            if (lane < nb) {
#pragma unroll
                for (int q = 0; q < QR; ++q) {
                    const int gr = gr0 + q;
                    a[q] = gr > lane ? a[q] * myscale : (gr == lane ? myR : a[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < QR; ++q)
                if (q < nv) P[lane * Rp + g0 + q] = a[q];
        };
        if (chunk <= 4) f64_cols(std::integral_constant<int, 4>{});
        else if (chunk <= 8) f64_cols(std::integral_constant<int, 8>{});
        else if (chunk <= 12) f64_cols(std::integral_constant<int, 12>{});
        else if (chunk <= 16) f64_cols(std::integral_constant<int, 16>{});
        else if (chunk <= 20) f64_cols(std::integral_constant<int, 20>{});
        else if (chunk <= 24) f64_cols(std::integral_constant<int, 24>{});
        else if (chunk <= 28) f64_cols(std::integral_constant<int, 28>{});
        else f64_cols(std::integral_constant<int, QRC>{});
        done = true;
      }
    } else {
        // Each thread keeps its column's QR rows of this warp in registers; per
        // column the warp broadcasts u_jj and x_{jj+1} through its own buffers,
        // read 4 rows per load.  The columns stay unscaled as in the FP64 form:
        // with v formed and stored back, a row's place compared at each of five
        // passes over 32 rows and three dependent divisions, a column cost 3000
        // cycles beside its exchange whatever the rows of the warp: the panels of a
        // 1200 x 400 sketch 105 us each, 68 us so (with the previous panel's product
        // above spread over the CTA).  QR = 8 ... 64 is the fewest that hold the rows.
        auto f32_cols = [&](auto qr_tag) {
            constexpr int QR = decltype(qr_tag)::value;
            T a[QR];
#pragma unroll
            for (int q = 0; q < QR; ++q) a[q] = g0 + q < g1 ? P[lane * Rp + g0 + q] : (T)0;
            const int gr0 = r0 + g0;  // global row (from k0) of a[0]
            const int nv = g1 - g0;   // valid rows of this warp (<= 0: none); a is zero beyond
            auto row_of = [&](int row) -> T {
                T v = (T)0;
#pragma unroll
                for (int q = 0; q < QR; ++q)
                    if (gr0 + q == row) v = a[q];
                return v;
            };
            // lane c: its column below row `row`
            auto put_below = [&](T* x, int row) {
                if (gr0 > row) {
#pragma unroll
                    for (int q = 0; q < QR; q += 4) store4(x + q, a[q], a[q + 1], a[q + 2], a[q + 3]);
                } else {
#pragma unroll
                    for (int q = 0; q < QR; ++q) x[q] = gr0 + q > row ? a[q] : (T)0;
                }
            };
            auto dot = [&](const T* x) -> T {
                constexpr int CH = QR > 32 ? 8 : 4;  // chains
                T s4[CH];
#pragma unroll
                for (int e = 0; e < CH; ++e) s4[e] = (T)0;
#pragma unroll
                for (int q = 0; q < QR; q += 4) {
                    T xv[4];
                    load4(x + q, xv);
#pragma unroll
                    for (int e = 0; e < 4; ++e) s4[(q + e) % CH] = fma(xv[e], a[q + e], s4[(q + e) % CH]);
                }
                T r = (s4[0] + s4[1]) + (s4[2] + s4[3]);
                if constexpr (CH == 8) r += (s4[4] + s4[5]) + (s4[6] + s4[7]);
                return r;
            };
            T myscale = (T)1, myR = (T)0, rprev = (T)1;
            if (lane == 0) put_below(&bcx[0][warp][0], 0);
            if (0 >= gr0 && 0 < gr0 + nv) rowbuf[lane] = row_of(0);
            __syncwarp();
            acc = dot(&bcx[0][warp][0]);
            if (lane >= nb) acc = (T)0;
            for (int jj = 0; jj < nb; ++jj) {
                const Scal sc = exchange(jj, acc, rowbuf, 1, true);
                // Y[i][j] = v_i^T v_j from u_i^T u_j (lane i; rank 0, warp 0)
                if (rank == 0 && warp == 0 && lane < jj - 1) Ysm[lane][jj - 1] = Ysm[lane][jj - 1] * myscale * rprev;
                T* u = &bcx[jj & 1][warp][0];
                T* xn = &bcx[(jj + 1) & 1][warp][0];
                if (jj >= gr0 && jj < gr0 + nv) {  // the leading entry of u_jj
                    if (lane == 0) u[jj - gr0] = sc.v1;
                    __syncwarp();
                }
                if (sc.far) {
                    for (int q = lane; q < QR; q += 32) u[q] *= sc.rv1;
                    __syncwarp();
                }
                if (lane == jj) {
                    myscale = sc.rv1;
                    myR = sc.mu;
                }
                rprev = sc.far ? (T)1 : sc.rv1;
                if (lane > jj && lane < nb && sc.b != (T)0) {
                    const T f = sc.f;
#pragma unroll
                    for (int q = 0; q < QR; q += 4) {
                        T uv[4];
                        load4(u + q, uv);
#pragma unroll
                        for (int e = 0; e < 4; ++e) a[q + e] = fma(-f, uv[e], a[q + e]);
                    }
                    // R's row without the roundings of f and v1
                    if (jj >= gr0 && jj < gr0 + nv) {
#pragma unroll
                        for (int q = 0; q < QR; ++q) a[q] = gr0 + q == jj ? sc.rc : a[q];
                    }
                }
                const int jn = jj + 1;
                if (jn < nb) {
                    if (lane == jn) put_below(xn, jn);
                    if (jn >= gr0 && jn < gr0 + nv) rowbuf[lane] = row_of(jn);
                }
                __syncwarp();
                // lanes c > jj: dots of column jj + 1; lanes i < jj: u_i^T u_jj
                const bool ylane = lane < jj, dlane = lane >= jn && lane < nb && jn < nb;
                acc = dot(ylane ? u : xn);
                if (!(ylane || dlane)) acc = (T)0;
            }
            // lane < nb - 1: the scales of Y's last column, formed below
            if (rank == 0 && warp == 0) {
                ysc0 = myscale;
                ysc1 = rprev;
            }
            // R on and above the diagonal, v below it
            if (lane < nb) {
#pragma unroll
                for (int q = 0; q < QR; ++q) {
                    const int gr = gr0 + q;
                    a[q] = gr > lane ? a[q] * myscale : (gr == lane ? myR : a[q]);
                }
            }
#pragma unroll
            for (int q = 0; q < QR; ++q)
                if (q < nv) P[lane * Rp + g0 + q] = a[q];
        };
        done = true;
        if (chunk <= 8) f32_cols(std::integral_constant<int, 8>{});
        else if (chunk <= 16) f32_cols(std::integral_constant<int, 16>{});
        else if (chunk <= 24) f32_cols(std::integral_constant<int, 24>{});
        else if (chunk <= 32) f32_cols(std::integral_constant<int, 32>{});
        else if (chunk <= QRC32) f32_cols(std::integral_constant<int, QRC32>{});
        else done = false;
    }
    if (!done) {
        acc = dots(0);
        for (int jj = 0; jj < nb; ++jj) {
            T* xj = P + jj * Rp;
            T* ac = P + lane * Rp;
            const int owner = (int)(jj / R);
            const Scal sc = exchange(jj, acc, P + (jj - r0), Rp);
            const T b = sc.b, wc = sc.wc;
            if (rank == owner && tid == 0) xj[jj - r0] = sc.mu;  // the diagonal entry is not read again (v there is 1)
            // v below the diagonal, this warp's rows
            const int ib = max(jj + 1 - r0, 0);
            if (sc.scale)
                for (int i = max(ib, g0) + lane; i < g1; i += 32) xj[i] = xj[i] * sc.rv1;
            __syncwarp();
            if (lane > jj && lane < nb && b != (T)0) {
                const int id = max(jj - r0, 0);  // owned rows >= the diagonal
                const int dr = jj - r0;           // local index of the diagonal row
                int i = max(id, g0);
                // blocks of 8 rows: all loads before the stores (the column of v and
                // the updated column never overlap)
                for (; i + 8 <= g1; i += 8) {
                    T v[8], av[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        v[q] = (i + q == dr) ? (T)1 : xj[i + q];
                        av[q] = ac[i + q];
                    }
#pragma unroll
                    for (int q = 0; q < 8; ++q) ac[i + q] = fma(-wc, v[q], av[q]);
                }
                for (; i < g1; ++i) {
                    const T vi = (i == dr) ? (T)1 : xj[i];
                    ac[i] = fma(-wc, vi, ac[i]);
                }
            }
            __syncwarp();
            acc = dots_y(jj);
        }
    }
    // Y[:, nb - 1] of the last column: one more reduction, into rank 0
    part[warp][lane] = acc;
    __syncthreads();
    if (warp == 0) {
        const T t = tree_sum<T, QCT / 32>(&part[0][lane], QNB);
        *cluster.map_shared_rank(&all_part[nb & 1][rank][lane], 0) = t;
    }
    cluster.sync();
    if (rank == 0 && warp == 0 && lane + 1 < nb)
        Ysm[lane][nb - 1] = tree_sum<T, QCL>(&all_part[nb & 1][0][lane], QNB) * ysc0 * ysc1;
    // write R / v back to W and the explicit V (0 above, 1 on the diagonal)
    for (int i = tid; i < nloc; i += QCT) {
        const int64_t gi = r0 + i;
#pragma unroll 8
        for (int c = 0; c < QNB; ++c) {
            if (c < nb) {
                const T pv = P[c * Rp + i];
                W[(k0 + gi) + (k0 + c) * ld] = pv;
                V[gi + c * ldv] = gi < c ? (T)0 : (gi == c ? (T)1 : pv);
            } else {
                V[gi + c * ldv] = (T)0;
            }
        }
    }
    __syncthreads();
    if (rank == 0) {
        __syncthreads();
        if (warp == 0) {
            // column by column: T[0:j, j] = -beta_j T[0:j, 0:j] Y[0:j, j]; lane = row
            T trow[QNB];
#pragma unroll
            for (int jj = 0; jj < QNB; ++jj) {
                T t4[4] = {(T)0, (T)0, (T)0, (T)0};  // 4 chains: the latency of 496 dependent FMAs is long in FP64
                if (jj < nb)
#pragma unroll
                    for (int qq = 0; qq < jj; ++qq) t4[qq & 3] = fma(trow[qq], Ysm[qq][jj], t4[qq & 3]);
                const T t = (t4[0] + t4[1]) + (t4[2] + t4[3]);
                const T bj = jj < nb ? bsh[jj] : (T)0;
                trow[jj] = lane < jj ? -bj * t : (lane == jj ? bj : (T)0);
            }
#pragma unroll
            for (int c = 0; c < QNB; ++c) Tm[lane + c * QNB] = trow[c];
        }
    }
}

// ---------------------------------------------------------------------------
// Trailing update C <- (I - V T^T V^T) C in one launch.  A cluster of QUC CTAs
// owns a block of 32 columns of C; its CTAs take the 128-row sub-tiles of the
// block in turn (rank, rank + QUC, ...).  Per CTA:
//   1. W_r = V^T C over its sub-tiles (32 x 32), four row groups of 64 threads
//      with 4 x 4 register tiles, summed in a fixed order;
//   2. W = sum_r W_r over the cluster (rank order, read through distributed
//      shared memory), W2 = T^T W (T upper, so W2[p] uses T[0..p][p]);
//   3. C -= V W2 over its sub-tiles, written back coalesced.
// Sub-tiles are staged in shared memory as [32 columns][128 rows] with the
// 4-element groups of a row XOR-swizzled by (column / 4), so that both the
// transposing stores and the 4-wide reads of either phase are free of bank
// conflicts.  V columns >= nb load as zero (so do rows >= rows, columns >= nt).
// ---------------------------------------------------------------------------
constexpr int QUC = 8;    // CTAs per cluster
constexpr int QUR = 128;  // rows per sub-tile
constexpr int QUT = 256;  // threads per CTA

template <typename T>
struct alignas(4 * sizeof(T)) QuVec {
    T v[4];
};

// position of (column c, row i) in a swizzled [32][QUR] sub-tile
__device__ __forceinline__ int qu_idx(int c, int i) { return c * QUR + ((((i >> 2) ^ (c >> 2)) << 2) | (i & 3)); }

template <typename T>
static size_t qu_smem_bytes() {
    // V and C sub-tiles (the row-group partials of phase 1 reuse them), the
    // cluster-visible partial W_r, the summed W, W2 and T
    return sizeof(T) * (2 * 32 * QUR + 3 * 32 * 33 + 32 * 32);
}

// A sub-tile in registers: thread t holds row t mod QUR of columns
// t / QUR + 2 j, j < 16, of V and C (consecutive threads read consecutive rows).
template <typename T>
struct QuRegs {
    T v[16], c[16];
};

template <typename T>
__device__ __forceinline__ void qu_fetch(QuRegs<T>& rg, const T* __restrict__ V, int64_t ldv, int nb,
                                         const T* __restrict__ C, int64_t ldc, int64_t ncols, int64_t rows,
                                         int64_t r0) {
    const int i = threadIdx.x & (QUR - 1), c0 = threadIdx.x >> 7;
    const int64_t gi = r0 + i;
    const bool ok = gi < rows;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        const int c = c0 + 2 * j;
        rg.v[j] = (ok && c < nb) ? V[gi + c * ldv] : (T)0;
        rg.c[j] = (ok && c < ncols) ? C[gi + c * ldc] : (T)0;
    }
}

template <typename T>
__device__ __forceinline__ void qu_put(const QuRegs<T>& rg, T* __restrict__ Vs, T* __restrict__ Cs) {
    const int i = threadIdx.x & (QUR - 1), c0 = threadIdx.x >> 7;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        Vs[qu_idx(c0 + 2 * j, i)] = rg.v[j];
        Cs[qu_idx(c0 + 2 * j, i)] = rg.c[j];
    }
}

template <typename T, int CL>
__global__ void __launch_bounds__(QUT)
    k_qr_update(T* __restrict__ C, int64_t ldc, int64_t nt, const T* __restrict__ V, int64_t ldv, int nb,
                const T* __restrict__ Tm, int64_t rows) {
    extern __shared__ __align__(16) unsigned char qu_raw[];
    T* Vs = (T*)qu_raw;
    T* Cs = Vs + 32 * QUR;
    T* Wr = Cs + 32 * QUR;  // [32][33] this CTA's partial, read by the whole cluster
    T* Wf = Wr + 32 * 33;   // [32][33] the cluster sum
    T* Ts = Wf + 32 * 33;   // [32][33] T
    T* W2 = Ts + 32 * 33;   // [32][32] T^T W
    T* Wk = Vs;             // [4][32][33] row-group partials (after phase 1)
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank();
    const int64_t c0 = (int64_t)(blockIdx.x / CL) * 32;
    const int64_t ncols = min64(32, nt - c0);
    T* Cb = C + c0 * ldc;
    const int tid = threadIdx.x;
    const int64_t nsub = (rows + QUR - 1) / QUR;
    for (int q = tid; q < 32 * 32; q += QUT) Ts[(q & 31) * 33 + (q >> 5)] = Tm[q];  // Ts[k][p] = T[k, p]

    // 1. W_r = V^T C over this CTA's sub-tiles (the next sub-tile is fetched
    // into registers while the current one is used)
    QuRegs<T> rg;
    if (rank < nsub) qu_fetch<T>(rg, V, ldv, nb, Cb, ldc, ncols, rows, (int64_t)rank * QUR);
    {
        const int kg = tid >> 6, tl = tid & 63, tp = tl & 7, tq = tl >> 3;
        T acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
        for (int64_t sb = rank; sb < nsub; sb += CL) {
            __syncthreads();
            qu_put<T>(rg, Vs, Cs);
            __syncthreads();
            if (sb + CL < nsub) qu_fetch<T>(rg, V, ldv, nb, Cb, ldc, ncols, rows, (sb + CL) * QUR);
#pragma unroll 2
            for (int s4 = 0; s4 < QUR / 16; ++s4) {
                const int i = kg * (QUR / 4) + 4 * s4;
                QuVec<T> va[4], cb[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) va[a] = *(const QuVec<T>*)(Vs + qu_idx(4 * tp + a, i));
#pragma unroll
                for (int b = 0; b < 4; ++b) cb[b] = *(const QuVec<T>*)(Cs + qu_idx(4 * tq + b, i));
#pragma unroll
                for (int w = 0; w < 4; ++w)
#pragma unroll
                    for (int a = 0; a < 4; ++a)
#pragma unroll
                        for (int b = 0; b < 4; ++b) acc[a][b] = fma(va[a].v[w], cb[b].v[w], acc[a][b]);
            }
        }
        __syncthreads();
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) Wk[(kg * 32 + 4 * tp + a) * 33 + 4 * tq + b] = acc[a][b];
        __syncthreads();
        for (int q = tid; q < 32 * 32; q += QUT) {
            const int p = q >> 5, c = q & 31;
            Wr[p * 33 + c] = ((Wk[p * 33 + c] + Wk[(32 + p) * 33 + c]) + Wk[(64 + p) * 33 + c]) + Wk[(96 + p) * 33 + c];
        }
    }
    // the first sub-tile of step 3 (C is not written before step 3)
    if (rank < nsub) qu_fetch<T>(rg, V, ldv, nb, Cb, ldc, ncols, rows, (int64_t)rank * QUR);
    // 2. W = sum over the cluster, W2 = T^T W
    cluster.sync();
    for (int q = tid; q < 32 * 32; q += QUT) {
        const int p = q >> 5, c = q & 31;
        T w = (T)0;
        for (int r = 0; r < CL; ++r) w += cluster.map_shared_rank(Wr, r)[p * 33 + c];
        Wf[p * 33 + c] = w;
    }
    // this CTA's reads of the other CTAs' partials are done; they may exit
    // once every CTA has arrived (waited for at the end)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    __syncthreads();
    for (int q = tid; q < 32 * 32; q += QUT) {
        const int p = q >> 5, c = q & 31;
        T w = (T)0;
        for (int k = 0; k <= p; ++k) w = fma(Ts[k * 33 + p], Wf[k * 33 + c], w);
        W2[p * 32 + c] = w;
    }
    // 3. C -= V W2 over this CTA's sub-tiles
    {
        const int ti = tid & 31, tq = tid >> 5;  // rows 4 ti .. 4 ti + 3, columns 4 tq .. 4 tq + 3
        for (int64_t sb = rank; sb < nsub; sb += CL) {
            __syncthreads();
            qu_put<T>(rg, Vs, Cs);
            __syncthreads();
            if (sb + CL < nsub) qu_fetch<T>(rg, V, ldv, nb, Cb, ldc, ncols, rows, (sb + CL) * QUR);
            QuVec<T> cv[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) cv[b] = *(const QuVec<T>*)(Cs + qu_idx(4 * tq + b, 4 * ti));
#pragma unroll 4
            for (int p = 0; p < 32; ++p) {
                const QuVec<T> v = *(const QuVec<T>*)(Vs + qu_idx(p, 4 * ti));
                const QuVec<T> w = *(const QuVec<T>*)(W2 + p * 32 + 4 * tq);
#pragma unroll
                for (int b = 0; b < 4; ++b)
#pragma unroll
                    for (int a = 0; a < 4; ++a) cv[b].v[a] = fma(-v.v[a], w.v[b], cv[b].v[a]);
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) *(QuVec<T>*)(Cs + qu_idx(4 * tq + b, 4 * ti)) = cv[b];
            __syncthreads();
            const int64_t r0 = sb * QUR;
            for (int e = tid; e < 32 * QUR; e += QUT) {
                const int i = e & (QUR - 1), c = e >> 7;
                if (r0 + i < rows && c < ncols) Cb[(r0 + i) + c * ldc] = Cs[qu_idx(c, i)];
            }
        }
    }
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename TI, typename T>
__global__ void k_qr_load(const TI* __restrict__ As, int64_t s, int64_t n, int64_t ldas, T* __restrict__ W) {
    int64_t total = s * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = q % s, j = q / s;
        W[q] = (T)As[i + j * ldas];
    }
}

template <typename T>
__global__ void k_qr_extract(const T* __restrict__ W, int64_t ld, int64_t n, const int32_t* __restrict__ colexp,
                             double* __restrict__ Rs, int64_t ldr) {
    int64_t total = n * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = q % n, j = q / n;
        if (i <= j) {
            // row i times the sign of its diagonal entry (FP64 panels leave either)
            double v = (double)W[i + j * ld];
            if (W[i + i * ld] < (T)0) v = -v;
            Rs[i + j * ldr] = colexp ? ldexp(v, -colexp[j]) : v;
        }
    }
}

__global__ void k_check_diag(const double* __restrict__ Rs, int64_t n, int64_t ldr, int32_t* __restrict__ info) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double d = Rs[j + j * ldr];
    if (!(d > 0.0) || !isfinite(d)) set_info_once(info, (int32_t)(j + 1));
}

// Dynamic shared memory of the cluster panel: the local panel and, after it,
// rank 0's V^T V partials of every rank or (fused: the previous panel's
// update applied first) the local rows of V_p and the row-group partials.
template <typename T>
static size_t qr_cluster_smem(int64_t rows, int qcl, bool fused) {
    const size_t Rp = (size_t)(ceil_div(rows, qcl) | 1);
    // the fused form also stages the previous panel's V rows and the W
    // partials (Vl, Wk, Ct, Vt behind the local panel)
    const size_t pre = Rp * QNB + (size_t)(QKG + 2) * QNB * (QNB + 1);
    return sizeof(T) * (Rp * QNB + (fused ? pre : 0));
}

struct QrCluster {
    int qcl = 0;         // CTAs per cluster, 0: single-CTA panel kernel
    bool fused = false;  // each panel applies the previous panel's update to its own columns
};

// The panel kernel of a cluster size.
template <typename T>
static auto qr_panel_kernel(int qcl) {
    if constexpr (std::is_same<T, float>::value) {
        switch (qcl) {
        case 1: return k_qr_panel_cl<T, 1>;
        case 2: return k_qr_panel_cl<T, 2>;
        case 4: return k_qr_panel_cl<T, 4>;
        default: break;
        }
    }
    return qcl == 16 ? k_qr_panel_cl<T, 16> : k_qr_panel_cl<T, 8>;
}

// CTAs per cluster.  FP32: the fewest that leave a CTA at most 64 rows (8 a
// warp), and 16 beyond 512.  A column costs an exchange whose price grows with
// the cluster while the rows of a small sketch are little work: with 16 CTAs
// whatever the size a 1000 x 100 solve took 685 us, 660 with at most 128 rows a
// CTA and 654 with 64.  FP64, whose pipe bounds a CTA: 16.  16 CTAs where the
// device can schedule that with the panel's shared memory (non-portable size),
// else 8; 0 if neither fits (the single-CTA panel kernel then runs).  The fused
// form (each panel applies the previous panel's update to its own columns) is
// preferred where its shared memory fits.  Decided once per precision and size.
template <typename T>
static QrCluster qr_cluster_query(int64_t s) {
    const size_t lim = 200 * 1024;
    const int64_t rows_per_cta = 64;
    for (bool fused : {true, false}) {
        bool tried16 = false;
        for (int qcl : {1, 2, 4, 8, 16, 8}) {
            // ascending while too many rows per CTA; the last 8 is the fallback for 16
            if (qcl < 16 && !tried16 && (sizeof(T) == 8 || ceil_div(s, qcl) > rows_per_cta)) continue;
            tried16 = tried16 || qcl == 16;
            const size_t sm = qr_cluster_smem<T>(s, qcl, fused);
            if (sm > lim) continue;
            auto kern = qr_panel_kernel<T>(qcl);
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) != cudaSuccess ||
                (qcl > 8 &&
                 cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
                cudaGetLastError();
                continue;
            }
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = qcl;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(qcl);
            cfg.blockDim = dim3(QCT);
            cfg.dynamicSmemBytes = sm;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int nclusters = 0;
            if (cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters >= 1) {
                QrCluster q;
                q.qcl = qcl;
                q.fused = fused;
                return q;
            }
            cudaGetLastError();
        }
    }
    return QrCluster();
}

template <typename T>
static QrCluster qr_cluster_size(int64_t s) {
    static std::mutex mu;
    static int64_t last_s = -1;
    static int last_dev = -1;
    static QrCluster last_q;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (s != last_s || dev != last_dev) {
        last_q = qr_cluster_query<T>(s);
        last_s = s;
        last_dev = dev;
    }
    return last_q;
}

template <typename T>
static cudaError_t qr_launch_cluster(int qcl, size_t smem, cudaStream_t st, T* W, int64_t s, int64_t k0, int nb,
                                     T* beta, T* Tm, T* V, int64_t rows, const T* Vp, int64_t ldvp, const T* Tp) {
    auto kern = qr_panel_kernel<T>(qcl);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = qcl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(qcl);
    cfg.blockDim = dim3(QCT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, W, s, s, k0, nb, beta, Tm, V, rows, Vp, ldvp, Tp);
}

// V and T are double-buffered by panel parity (a panel's V and T are read by
// its trailing update and by the next panel while the next panel writes the
// other buffer).
struct QrLayout {
    size_t w, beta, tm[2], v[2];
    size_t total;
};

static QrLayout qr_layout(int64_t s, int64_t n, int es) {
    QrLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
    L.w = take((size_t)s * n * es);
    L.beta = take((size_t)n * es);
    for (int b = 0; b < 2; ++b) {
        L.tm[b] = take((size_t)QNB * QNB * es);
        L.v[b] = take((size_t)s * QNB * es);
    }
    L.total = off;
    return L;
}

// Whether clusters of 16 update CTAs (non-portable size) can be scheduled
// with the update's shared memory; decided once per device.
template <typename T>
static bool qu_cluster16_ok() {
    static std::mutex mu;
    static int known[64] = {};  // 0 unknown, 1 yes, 2 no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lk(mu);
    if (known[dev] == 0) {
        const size_t sm = qu_smem_bytes<T>();
        auto kern = k_qr_update<T, 16>;
        bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm) == cudaSuccess &&
                  cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
        if (ok) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 16;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(16);
            cfg.blockDim = dim3(QUT);
            cfg.dynamicSmemBytes = sm;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int nclusters = 0;
            ok = cudaOccupancyMaxActiveClusters(&nclusters, kern, &cfg) == cudaSuccess && nclusters >= 1;
        }
        cudaGetLastError();
        known[dev] = ok ? 1 : 2;
    }
    return known[dev] == 1;
}

// C (rows x nt, ld s) <- (I - V T^T V^T) C.  A cluster per 32 columns; FP64
// updates of few columns (at most 7 column tiles, 56 CTAs with 8 per cluster)
// take 16 CTAs per cluster when there are rows for 16 (2048 or more), so that
// twice the SMs share them.  That is the unblocked FP64 QR (n <= 256, or the
// digit-sliced products off): the blocked one spreads such updates over the chip
// (qr_apply_wide below), with scratch that the unblocked one does not have.
template <typename T>
static lsq_status qr_apply(const T* V, const T* Tm, int nb, int64_t rows, T* C, int64_t s, int64_t nt,
                           cudaStream_t st) {
    if (nt <= 0) return LSQ_OK;
    const size_t sm = qu_smem_bytes<T>();
    const int64_t ctiles = ceil_div(nt, 32);
    const bool wide = std::is_same<T, double>::value && ctiles * 16 <= device_sm_count() &&
                      ceil_div(rows, QUR) >= 16 && qu_cluster16_ok<T>();
    const int cl = wide ? 16 : 8;
    auto kern = wide ? k_qr_update<T, 16> : k_qr_update<T, 8>;
    LSQ_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(ctiles * cl));
    cfg.blockDim = dim3(QUT);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LSQ_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, C, s, nt, V, rows, nb, Tm, rows));
    note_launch();
    return LSQ_OK;
}

// ---------------------------------------------------------------------------
// FP64 update of a few column tiles, C <- (I - V T^T V^T) C, in three launches
// that spread the rows over the whole chip.  The FP64 pipe (2 FMA a cycle and
// SM) bounds it: 64 rows x rows of C of work each way.  The cluster form above
// has 16 SMs per 32 columns, and the form fused into the next panel (which
// applies V to that panel's 32 columns) the 16 SMs of the panel: 100 us + 150 us
// a panel of 3000 rows on average; with the three launches here the QR of a
// 4000 x 2000 matrix went from 44.4 to 32.4 ms.
//   1. W_z = V^T C over 64-row chunks z, one CTA per chunk and 32 columns;
//   2. W = sum_z W_z (fixed order), W2 = T^T W, one CTA per 8 columns;
//   3. C -= V W2, one CTA per chunk and 32 columns.
// ---------------------------------------------------------------------------
constexpr int QWR = 64;         // rows per chunk
constexpr int QW_MIN = 512;     // fewer rows: the fused and the cluster form (one launch)

__global__ void __launch_bounds__(256) k_qr_wpart(const double* __restrict__ V, int64_t ldv, int nb,
                                                  const double* __restrict__ C, int64_t ldc, int64_t nt, int64_t rows,
                                                  double* __restrict__ Wp) {
    __shared__ double sm[4 * 32 * 33];
    double* Vs = sm;                     // [32][QWR + 1]
    double* Cs = sm + 32 * (QWR + 1);
    static_assert(2 * 32 * (QWR + 1) <= 4 * 32 * 33, "the partials reuse the tiles");
    const int tid = threadIdx.x, i = tid & (QWR - 1), c0 = tid >> 6;
    const int64_t r0 = (int64_t)blockIdx.x * QWR, j0 = (int64_t)blockIdx.y * 32;
    const bool ok = r0 + i < rows;
    double v[8], x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int c = c0 + 4 * j;
        v[j] = ok && c < nb ? V[r0 + i + c * ldv] : 0.0;
        x[j] = ok && j0 + c < nt ? C[r0 + i + (j0 + c) * ldc] : 0.0;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        Vs[(c0 + 4 * j) * (QWR + 1) + i] = v[j];
        Cs[(c0 + 4 * j) * (QWR + 1) + i] = x[j];
    }
    __syncthreads();
    // four row groups of 64 threads with 4 x 4 tiles
    const int kg = tid >> 6, tp = tid & 7, tq = (tid & 63) >> 3;
    double acc[4][4] = {};
#pragma unroll 4
    for (int k = kg * (QWR / 4); k < (kg + 1) * (QWR / 4); ++k) {
        double a[4], b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            a[q] = Vs[(tp + 8 * q) * (QWR + 1) + k];
            b[q] = Cs[(tq + 8 * q) * (QWR + 1) + k];
        }
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[p][q] = fma(a[p], b[q], acc[p][q]);
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) sm[(kg * 32 + tp + 8 * p) * 33 + tq + 8 * q] = acc[p][q];
    __syncthreads();
    double* out = Wp + ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * 1024;
    for (int q = tid; q < 1024; q += 256) {
        const int e = (q >> 5) * 33 + (q & 31);
        out[q] = (sm[e] + sm[32 * 33 + e]) + (sm[64 * 33 + e] + sm[96 * 33 + e]);
    }
}

__global__ void __launch_bounds__(256) k_qr_wred(const double* __restrict__ Wp, int nch, const double* __restrict__ Tm,
                                                 double* __restrict__ W2) {
    __shared__ double Wf[32][8];
    const int p = threadIdx.x >> 3, cl = threadIdx.x & 7, c = (int)blockIdx.y * 8 + cl;
    const double* src = Wp + (int64_t)blockIdx.x * nch * 1024 + p * 32 + c;
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    int z = 0;
    for (; z + 4 <= nch; z += 4)
#pragma unroll
        for (int q = 0; q < 4; ++q) s[q] += src[(int64_t)(z + q) * 1024];
    for (; z < nch; ++z) s[0] += src[(int64_t)z * 1024];
    Wf[p][cl] = (s[0] + s[1]) + (s[2] + s[3]);
    __syncthreads();
    double w0 = 0.0, w1 = 0.0;
    for (int k = 0; k <= p; k += 2) {
        w0 = fma(Tm[k + p * QNB], Wf[k][cl], w0);
        if (k < p) w1 = fma(Tm[k + 1 + p * QNB], Wf[k + 1][cl], w1);
    }
    W2[(int64_t)blockIdx.x * 1024 + p * 32 + c] = w0 + w1;
}

__global__ void __launch_bounds__(256) k_qr_wapply(const double* __restrict__ V, int64_t ldv, int nb,
                                                   double* __restrict__ C, int64_t ldc, int64_t nt, int64_t rows,
                                                   const double* __restrict__ W2) {
    __shared__ double Vs[32][QWR];
    __shared__ __align__(16) double Ws[32][32];
    const int tid = threadIdx.x, i = tid & (QWR - 1), g = tid >> 6;
    const int64_t r0 = (int64_t)blockIdx.x * QWR, j0 = (int64_t)blockIdx.y * 32;
    const bool ok = r0 + i < rows;
    double v[8], x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int c = g + 4 * j;
        v[j] = ok && c < nb ? V[r0 + i + c * ldv] : 0.0;
        x[j] = ok && j0 + 8 * g + j < nt ? C[r0 + i + (j0 + 8 * g + j) * ldc] : 0.0;
    }
    for (int q = tid; q < 1024; q += 256) Ws[q >> 5][q & 31] = W2[(int64_t)blockIdx.y * 1024 + q];
#pragma unroll
    for (int j = 0; j < 8; ++j) Vs[g + 4 * j][i] = v[j];
    __syncthreads();
#pragma unroll 4
    for (int p = 0; p < 32; ++p) {
        const double vv = Vs[p][i];
#pragma unroll
        for (int j = 0; j < 8; ++j) x[j] = fma(-vv, Ws[p][8 * g + j], x[j]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
        if (ok && j0 + 8 * g + j < nt) C[r0 + i + (j0 + 8 * g + j) * ldc] = x[j];
}

// Scratch of qr_apply_wide: the partials of every chunk and 32 columns, then W2.
static size_t qr_wide_bytes(int64_t rows, int64_t nt) {
    return sizeof(double) * 1024 * (size_t)ceil_div(nt, 32) * (size_t)(ceil_div(rows, QWR) + 1);
}

static lsq_status qr_apply_wide(const double* V, const double* Tm, int nb, int64_t rows, double* C, int64_t s,
                                int64_t nt, double* scratch, cudaStream_t st) {
    if (nt <= 0) return LSQ_OK;
    const unsigned nch = (unsigned)ceil_div(rows, QWR), ct = (unsigned)ceil_div(nt, 32);
    double* W2 = scratch + (int64_t)1024 * ct * nch;
    k_qr_wpart<<<dim3(nch, ct), 256, 0, st>>>(V, rows, nb, C, s, nt, rows, scratch);
    LSQ_LAUNCH_CHECK();
    k_qr_wred<<<dim3(ct, 4), 256, 0, st>>>(scratch, (int)nch, Tm, W2);
    LSQ_LAUNCH_CHECK();
    k_qr_wapply<<<dim3(nch, ct), 256, 0, st>>>(V, rows, nb, C, s, nt, rows, W2);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

// Internal streams for the look-ahead QR (one pair per device): panels on a
// high-priority stream, the wide trailing updates on a low-priority one.
struct QrStreams {
    cudaStream_t hi = nullptr, lo = nullptr;
    bool ok = false;
};
static std::mutex g_qr_mu;

static QrStreams* qr_streams() {
    static QrStreams per_dev[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    QrStreams& q = per_dev[dev];
    if (!q.ok) {
        int lo_p = 0, hi_p = 0;
        if (cudaDeviceGetStreamPriorityRange(&lo_p, &hi_p) != cudaSuccess) return nullptr;
        if (cudaStreamCreateWithPriority(&q.hi, cudaStreamNonBlocking, hi_p) != cudaSuccess) return nullptr;
        if (cudaStreamCreateWithPriority(&q.lo, cudaStreamNonBlocking, lo_p) != cudaSuccess) return nullptr;
        q.ok = true;
    }
    return &q;
}

// ---------------------------------------------------------------------------
// FP64 QR with the trailing updates on the tensor cores.  The columns are
// taken in blocks of QTB: inside a block, 32-column panels and their
// rank-32 updates as above (restricted to the block); then the block's
// reflectors H_1 ... H_b = I - V T V^T update every later column at once,
//   W = V^T C,  X = T^T W,  C <- C - V X,
// each an FP64-accurate digit-sliced product (csrc/oz_trsm.cu).  T is formed
// from S = T^{-1} = striu(V^T V) + diag(1/beta) (Puglisi 1992; Joffrain et al.
// 2006: the triangular factor of the compact WY form is the inverse of that
// matrix) and the panels' own T factors, the inverses of its diagonal blocks (a
// zero beta, H = I, gives a zero row and column of T).
// ---------------------------------------------------------------------------
constexpr int QTB = 256;  // columns per block of the tensor-core form

static bool qr_tc_blocked(int es, int64_t n) { return es == 8 && n > QTB && fp64_emulation_enabled() && ot_trsm_supported(); }

struct QrTcLayout {
    size_t vx, vt, gw, part, tt, tp, xp, err, ot, ot_bytes, total;
};

static QrTcLayout qr_tc_layout(int64_t s, int64_t n) {
    QrTcLayout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
    L.vx = take(sizeof(double) * (size_t)s * QTB);
    L.vt = take(sizeof(double) * (size_t)s * QTB);
    L.gw = take(sizeof(double) * QTB * (size_t)n);  // -V^T [V C] (V and C: at most n columns)
    L.part = take(ot_gemm_long_part_bytes(QTB, n, s));
    L.tt = take(sizeof(double) * QTB * QTB);
    L.tp = take(sizeof(double) * QNB * QTB);  // the T factors of the block's panels
    L.xp = take(sizeof(double) * QTB * (size_t)n);
    L.err = take(sizeof(int32_t));
    L.ot_bytes = std::max(ot_gemm_long_ws_bytes(QTB, n, s),
                          ot_update_ws_bytes(std::max<int64_t>(s, QTB), std::max<int64_t>(n, QTB), QTB));
    L.ot = take(L.ot_bytes);
    L.total = off;
    return L;
}

// The block's reflectors as explicit V (rows x nb, ld rows) and V^T (nb x
// rows, ld nb): unit diagonal, zero above, Householder vectors below (the
// lower part of W's columns j0 .. j0 + nb - 1 from row j0).
__global__ void k_qr_vblock(const double* __restrict__ W, int64_t ld, int64_t j0, int64_t rows, int nb,
                            double* __restrict__ Vx, double* __restrict__ Vt) {
    const int64_t total = rows * nb;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = q % rows, c = q / rows;
        const double v = r < c ? 0.0 : (r == c ? 1.0 : W[(j0 + r) + (j0 + c) * ld]);
        Vx[q] = v;
        Vt[c + r * nb] = v;
    }
}

// T^T (ld nb) of the block from Gn = -V^T V (ld nb) and the T factors of its
// panels (Tp: panel q's 32 x 32 T at Tp + 1024 q, column-major, zero below the
// diagonal and past its columns).  With S = T^{-1} = striu(V^T V) + diag(1/beta),
// column j of T by back substitution over 32-row blocks,
//   t_I = -T_II sum_{J > I} S[I, J] t_J,   t_J(j) = T_JJ[:, j] in j's own block:
// the diagonal blocks of S are inverted already (the panels' T), so that a block
// takes two matrix-vector products and no chain of 32 steps (one warp per
// column walking its 256 rows one by one took 232 us).  One warp
// per column, lane = row of the block.
__global__ void __launch_bounds__(32) k_qr_tblock(const double* __restrict__ Gn, const double* __restrict__ Tp, int nb,
                                                   double* __restrict__ Tt) {
    __shared__ double t[QTB];
    __shared__ double rhs[QNB];
    const int j = blockIdx.x, lane = threadIdx.x, jb = j / QNB;
    t[jb * QNB + lane] = Tp[1024 * jb + lane + (j % QNB) * QNB];
    for (int I = jb + 1; I * QNB < nb; ++I) t[I * QNB + lane] = 0.0;
    __syncwarp();
    for (int I = jb - 1; I >= 0; --I) {
        const int i = I * QNB + lane;  // only the last block can be ragged, and I is not it
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        const int p1 = min(nb, (jb + 1) * QNB);
        int p = (I + 1) * QNB;
        for (; p + 4 <= p1; p += 4)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[q] = fma(-Gn[i + (int64_t)(p + q) * nb], t[p + q], s[q]);
        for (; p < p1; ++p) s[0] = fma(-Gn[i + (int64_t)p * nb], t[p], s[0]);
        rhs[lane] = (s[0] + s[1]) + (s[2] + s[3]);
        __syncwarp();
        double w[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int q = 0; q < QNB; ++q) w[q & 3] = fma(Tp[1024 * I + lane + q * QNB], rhs[q], w[q & 3]);
        t[i] = -((w[0] + w[1]) + (w[2] + w[3]));
        __syncwarp();
    }
    for (int i = lane; i < nb; i += 32) Tt[j + (int64_t)i * nb] = t[i];
}

__global__ void k_qr_err_to_info(const int32_t* __restrict__ err, int32_t* __restrict__ info) {
    if (*err != 0 && *info == 0) *info = -2;
}

// C (rows x nt, ld s) <- (I - V T^T V^T) C for the block of nb reflectors
// stored in W's columns j0 .. j0 + nb - 1 (C: W's rows j0.., columns j0 + nb..).
static lsq_status qr_tc_trailing(double* W, int64_t s, int64_t j0, int nb, int64_t n, char* base, const QrTcLayout& L,
                                 cudaStream_t st) {
    const int64_t rows = s - j0, nt = n - j0 - nb;
    if (nt <= 0) return LSQ_OK;
    double* Vx = (double*)(base + L.vx);
    double* Vt = (double*)(base + L.vt);
    double* Gn = (double*)(base + L.gw);
    double* Wn = Gn + (int64_t)nb * nb;
    double* Tt = (double*)(base + L.tt);
    double* Xp = (double*)(base + L.xp);
    int32_t* err = (int32_t*)(base + L.err);
    char* ows = base + L.ot;
    double* C = W + j0 + (j0 + nb) * s;
    lsq_status r;
    k_qr_vblock<<<(unsigned)std::min<int64_t>(ceil_div(rows * nb, 256), 8192), 256, 0, st>>>(W, s, j0, rows, nb, Vx,
                                                                                              Vt);
    LSQ_LAUNCH_CHECK();
    // [Gn Wn] = -V^T [V C]
    if ((r = ot_gemm_long(Vt, nb, Vx, rows, nb, C, s, nt, Gn, nb, rows, (double*)(base + L.part), ows, L.ot_bytes, err,
                          st)) != LSQ_OK)
        return r;
    k_qr_tblock<<<(unsigned)nb, 32, 0, st>>>(Gn, (const double*)(base + L.tp), nb, Tt);
    LSQ_LAUNCH_CHECK();
    // Xp = 0 - T^T Wn = T^T (V^T C)
    LSQ_CUDA_TRY(cudaMemsetAsync(Xp, 0, sizeof(double) * nb * (size_t)nt, st));
    if ((r = ot_gemm_update(Tt, nb, Wn, 1, nb, Xp, nb, Xp, nb, nb, nt, nb, ows, L.ot_bytes, err, st)) != LSQ_OK)
        return r;
    // C <- C - V Xp
    return ot_gemm_update(Vx, rows, Xp, 1, nb, C, s, C, s, rows, nt, nb, ows, L.ot_bytes, err, st);
}

size_t qr_ws_bytes(int64_t s, int64_t n, int prec) {
    int es = prec == LSQ_FP64 ? 8 : 4;
    size_t b = qr_layout(s, n, es).total + 256;
    if (qr_tc_blocked(es, n)) b += qr_tc_layout(s, n).total + 256;
    return b;
}

// FP64 QR by blocks of QTB columns (see qr_tc_trailing): the panels and
// rank-32 updates inside a block on the panel stream as in qr_run, the
// block's update of every later column on the tensor cores.  W holds A_s.
static lsq_status qr_blocked_f64(double* W, double* beta, int64_t s, int64_t n, const int32_t* colexp, double* Rs,
                                 int64_t ldr, int32_t* info, char* base, const QrLayout& L, char* tcb,
                                 cudaStream_t st) {
    const QrTcLayout TL = qr_tc_layout(s, n);
    int32_t* err = (int32_t*)(tcb + TL.err);
    LSQ_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int32_t), st));
    const QrCluster qc = qr_cluster_size<double>(s);
    const int qcl = qc.qcl;
    int k = 0;  // panel counter: the parity of the V and T buffers
    lsq_status r = LSQ_OK;
    for (int64_t j0 = 0; j0 < n && r == LSQ_OK; j0 += QTB) {
        const int64_t j1 = std::min<int64_t>(n, j0 + QTB);
        const double* Vprev = nullptr;
        const double* Tprev = nullptr;
        int64_t ldvprev = 0;
        for (int64_t k0 = j0; k0 < j1; k0 += QNB, ++k) {
            const int b = k & 1;
            const int nb = (int)std::min<int64_t>(QNB, j1 - k0);
            const int64_t rows = s - k0;
            double* Tm = (double*)(tcb + TL.tp) + 1024 * ((k0 - j0) / QNB);
            double* V = (double*)(base + L.v[b]);
            if (qcl > 0) {
                const size_t clsm = qr_cluster_smem<double>(rows, qcl, qc.fused);
                if (qr_launch_cluster<double>(qcl, clsm, st, W, s, k0, nb, beta, Tm, V, rows, Vprev, ldvprev, Tprev) !=
                    cudaSuccess)
                    return LSQ_ERR_CUDA;
            } else {
                k_qr_panel<double><<<1, QPT, 0, st>>>(W, s, s, k0, nb, beta, Tm, V, rows);
            }
            note_launch();
            if (cudaGetLastError() != cudaSuccess) return LSQ_ERR_CUDA;
            // the rest of the block's columns
            const int64_t nt = j1 - k0 - nb;
            if (nt <= 0) {
                ++k;
                break;
            }
            const int64_t nn = std::min<int64_t>(QNB, nt), nw = nt - nn;
            double* C = W + k0 + (k0 + nb) * s;
            // the digit-sliced products' scratch is free until the block ends
            const bool wide = rows > QW_MIN && qr_wide_bytes(rows, nt) <= TL.ot_bytes;
            const bool fuse_next = !wide && qcl > 0 && qc.fused && nb == QNB;
            r = wide        ? qr_apply_wide(V, Tm, nb, rows, C, s, nt, (double*)(tcb + TL.ot), st)
                : fuse_next ? qr_apply<double>(V, Tm, nb, rows, C + nn * s, s, nw, st)
                            : qr_apply<double>(V, Tm, nb, rows, C, s, nt, st);
            if (r != LSQ_OK) return r;
            Vprev = fuse_next ? V : nullptr;
            Tprev = fuse_next ? Tm : nullptr;
            ldvprev = rows;
        }
        // the block's reflectors on every later column
        r = qr_tc_trailing(W, s, j0, (int)(j1 - j0), n, tcb, TL, st);
    }
    if (r != LSQ_OK) return r;
    k_qr_extract<double><<<(unsigned)std::min<int64_t>(ceil_div(n * n, 256), 4096), 256, 0, st>>>(W, s, n, colexp, Rs,
                                                                                                ldr);
    LSQ_LAUNCH_CHECK();
    if (info) {
        k_check_diag<<<(unsigned)ceil_div(n, 128), 128, 0, st>>>(Rs, n, ldr, info);
        LSQ_LAUNCH_CHECK();
        k_qr_err_to_info<<<1, 1, 0, st>>>(err, info);
        LSQ_LAUNCH_CHECK();
    }
    return LSQ_OK;
}

template <typename T>
static lsq_status qr_run(const void* As, int64_t s, int64_t n, int64_t ldas, int as_prec, const int32_t* colexp,
                         double* Rs, int64_t ldr, int32_t* info, void* ws, size_t ws_bytes, cudaStream_t st) {
    int es = sizeof(T);
    QrLayout L = qr_layout(s, n, es);
    char* base = (char*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    if (!ws || L.total + ((char*)base - (char*)ws) > ws_bytes) return LSQ_ERR_NOMEM;
    T* W = (T*)(base + L.w);
    T* beta = (T*)(base + L.beta);
    unsigned g = (unsigned)std::min<int64_t>(ceil_div(s * n, 256), 8192);
    if (as_prec == LSQ_FP64)
        k_qr_load<double, T><<<g, 256, 0, st>>>((const double*)As, s, n, ldas, W);
    else
        k_qr_load<float, T><<<g, 256, 0, st>>>((const float*)As, s, n, ldas, W);
    LSQ_LAUNCH_CHECK();
    if constexpr (std::is_same<T, double>::value) {
        if (qr_tc_blocked(es, n)) {
            char* tcb = base + align_up(L.total, 256);
            if (L.total + 256 + qr_tc_layout(s, n).total + ((char*)base - (char*)ws) > ws_bytes) return LSQ_ERR_NOMEM;
            return qr_blocked_f64(W, beta, s, n, colexp, Rs, ldr, info, base, L, tcb, st);
        }
    }
    // look-ahead: while panel k + 1 is factored (high-priority stream), the
    // wide part of panel k's trailing update runs on the low-priority stream;
    // the narrow part (the next panel's columns) goes first on the panel
    // stream.  Not while the caller's stream is being captured into a graph, nor
    // in the batched solver, where concurrent problems must not share streams.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    LSQ_CUDA_TRY(cudaStreamIsCapturing(st, &cap));
    QrStreams* qs =
        (cap == cudaStreamCaptureStatusNone && !FanoutScope::active() && n > 2 * QNB) ? qr_streams() : nullptr;
    std::unique_lock<std::mutex> lk(g_qr_mu, std::defer_lock);
    cudaEvent_t ev_fork = nullptr, ev_p = nullptr, ev_w[2] = {nullptr, nullptr}, ev_join = nullptr;
    auto cleanup = [&]() {
        for (cudaEvent_t e : {ev_fork, ev_p, ev_w[0], ev_w[1], ev_join})
            if (e) cudaEventDestroy(e);
    };
    cudaStream_t sh = st, sl = st;
    if (qs) {
        lk.lock();
        bool good = cudaEventCreateWithFlags(&ev_fork, cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventCreateWithFlags(&ev_p, cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventCreateWithFlags(&ev_w[0], cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventCreateWithFlags(&ev_w[1], cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventCreateWithFlags(&ev_join, cudaEventDisableTiming) == cudaSuccess &&
                    cudaEventRecord(ev_fork, st) == cudaSuccess && cudaStreamWaitEvent(qs->hi, ev_fork, 0) == cudaSuccess &&
                    cudaStreamWaitEvent(qs->lo, ev_fork, 0) == cudaSuccess;
        if (!good) {
            cleanup();
            return LSQ_ERR_CUDA;
        }
        sh = qs->hi;
        sl = qs->lo;
    }
    lsq_status r = LSQ_OK;
    const QrCluster qc = qr_cluster_size<T>(s);
    const int qcl = qc.qcl;
    // the previous panel's V and T when this panel applies its update itself
    const T* Vprev = nullptr;
    const T* Tprev = nullptr;
    int64_t ldvprev = 0;
    int k = 0;
    for (int64_t k0 = 0; k0 < n && r == LSQ_OK; k0 += QNB, ++k) {
        const int b = k & 1;
        int nb = (int)std::min<int64_t>(QNB, n - k0);
        int64_t rows = s - k0;
        T* Tm = (T*)(base + L.tm[b]);
        T* V = (T*)(base + L.v[b]);
        const size_t clsm = qcl > 0 ? qr_cluster_smem<T>(rows, qcl, qc.fused) : 0;
        // Householder panel: sum over its columns of 4 (rows - j)(nb - j) flops
        double pflops = 0.0;
        for (int j = 0; j < nb; ++j) pflops += 4.0 * (double)(rows - j) * (double)(nb - j);
        stage_mark(ST_K_QRPANEL, true, sh);
        if (qcl > 0) {
            if (qr_launch_cluster<T>(qcl, clsm, sh, W, s, k0, nb, beta, Tm, V, rows, Vprev, ldvprev, Tprev) !=
                cudaSuccess) {
                r = LSQ_ERR_CUDA;
                break;
            }
        } else {
            k_qr_panel<T><<<1, QPT, 0, sh>>>(W, s, s, k0, nb, beta, Tm, V, rows);
        }
        note_launch();
        if (cudaGetLastError() != cudaSuccess) {
            r = LSQ_ERR_CUDA;
            break;
        }
        stage_mark(ST_K_QRPANEL, false, sh, pflops);
        const int64_t nt = n - k0 - nb;
        if (nt <= 0) break;
        const int64_t nn = std::min<int64_t>(QNB, nt), nw = nt - nn;  // narrow / wide columns
        T* C = W + k0 + (k0 + nb) * s;
        // the next panel's columns (narrow part): by the next panel kernel
        // itself when fused (a full panel only: V then has QNB columns), else
        // a separate update on the panel stream
        const bool fuse_next = qcl > 0 && qc.fused && nb == QNB;
        if (qs) {
            // the wide part on the low-priority stream, after this panel
            if (cudaEventRecord(ev_p, sh) != cudaSuccess || cudaStreamWaitEvent(sl, ev_p, 0) != cudaSuccess) {
                r = LSQ_ERR_CUDA;
                break;
            }
            r = qr_apply<T>(V, Tm, nb, rows, C + nn * s, s, nw, sl);
            if (r != LSQ_OK || cudaEventRecord(ev_w[b], sl) != cudaSuccess) {
                r = r != LSQ_OK ? r : LSQ_ERR_CUDA;
                break;
            }
            // the next panel's columns also hold the previous panel's wide
            // update, and the next panel overwrites that update's V and T
            if (k >= 1 && cudaStreamWaitEvent(sh, ev_w[b ^ 1], 0) != cudaSuccess) {
                r = LSQ_ERR_CUDA;
                break;
            }
            if (!fuse_next) r = qr_apply<T>(V, Tm, nb, rows, C, s, nn, sh);
        } else {
            r = fuse_next ? qr_apply<T>(V, Tm, nb, rows, C + nn * s, s, nw, st)
                          : qr_apply<T>(V, Tm, nb, rows, C, s, nt, st);
        }
        Vprev = fuse_next ? V : nullptr;
        Tprev = fuse_next ? Tm : nullptr;
        ldvprev = rows;
    }
    if (qs) {
        // join both internal streams back into the caller's stream
        bool good = cudaEventRecord(ev_join, sh) == cudaSuccess && cudaStreamWaitEvent(st, ev_join, 0) == cudaSuccess &&
                    cudaEventRecord(ev_fork, sl) == cudaSuccess && cudaStreamWaitEvent(st, ev_fork, 0) == cudaSuccess;
        cleanup();
        if (!good && r == LSQ_OK) r = LSQ_ERR_CUDA;
    }
    if (r != LSQ_OK) return r;
    k_qr_extract<T><<<(unsigned)std::min<int64_t>(ceil_div(n * n, 256), 4096), 256, 0, st>>>(W, s, n, colexp, Rs, ldr);
    LSQ_LAUNCH_CHECK();
    if (info) {
        k_check_diag<<<(unsigned)ceil_div(n, 128), 128, 0, st>>>(Rs, n, ldr, info);
        LSQ_LAUNCH_CHECK();
    }
    return LSQ_OK;
}

lsq_status launch_precond_qr(const void* As, int64_t s, int64_t n, int64_t ldas, int as_prec, int qr_prec,
                             const int32_t* colexp, double* Rs, int64_t ldr, int32_t* info, void* ws, size_t ws_bytes,
                             cudaStream_t st) {
    if (qr_prec == LSQ_FP64) return qr_run<double>(As, s, n, ldas, as_prec, colexp, Rs, ldr, info, ws, ws_bytes, st);
    return qr_run<float>(As, s, n, ldas, as_prec, colexp, Rs, ldr, info, ws, ws_bytes, st);
}

}  // namespace lsq
