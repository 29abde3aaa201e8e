// n x n factorizations and vector triangular solves for Eqs. e_pne / e_hpne:
//   - blocked right-looking Cholesky G = L L^T (FP64 for PNE; FP32 for the
//     condition estimate of Sec. 6.1): diagonal block in shared memory, panel
//     solve one thread per row, trailing update as an FP64-accurate
//     tensor-core product (FP64 with workspace) or a register-tiled rank-nb
//     product on the CUDA cores;
//   - blocked right-looking LU with partial pivoting (first largest |pivot|,
//     as LAPACK's getrf) for HPNE;
//   - triangular solves L y = c, L^T y = c, U y = c, unit L y = c as a
//     wavefront over 32-row blocks, one CTA each.
// A device status word (info) is written on breakdown; every later kernel of
// the same factorization and the solves return early once it is set.
#include "common.cuh"
#include "kernels.cuh"
#include "trsv_block.cuh"

#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

namespace lsq {

constexpr int CNB = 64;   // Cholesky block
constexpr int LNB = 32;   // LU panel width

// ---------------------------------------------------------------------------
// Generic register-tiled rank-K update  C(i, j) -= sum_k P(i, k) Q(j, k)
// with element strides; 64x64 tiles, K <= 64 staged once.  lower: only tiles
// with tile_i >= tile_j (and entries i >= j written).
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_rank_update(T* __restrict__ C, int64_t ldc, const T* __restrict__ P,
                                                     int64_t psi, int64_t psk, const T* __restrict__ Q, int64_t qsj,
                                                     int64_t qsk, int64_t M, int64_t N, int K, bool lower,
                                                     int64_t tilesN, const int32_t* __restrict__ info) {
    if (info && *info != 0) return;
    __shared__ T Ps[32][64 + 1];
    __shared__ T Qs[32][64 + 1];
    int64_t t = blockIdx.x, ti, tj;
    if (lower) {
        int64_t r = (int64_t)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
        while ((r + 1) * (r + 2) / 2 <= t) ++r;
        while (r * (r + 1) / 2 > t) --r;
        ti = r;
        tj = t - r * (r + 1) / 2;
    } else {
        ti = t / tilesN;
        tj = t % tilesN;
    }
    int64_t i0 = ti * 64, j0 = tj * 64;
    int tid = threadIdx.x;
    int tx = tid & 15, ty = tid >> 4;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = (T)0;
    for (int kc = 0; kc < K; kc += 32) {
        int kn = min(32, K - kc);
        __syncthreads();
        for (int q = tid; q < 64 * 32; q += 256) {
            int r = q % 64, k = q / 64;
            int64_t gi = i0 + r, gj = j0 + r;
            bool kin = k < kn;
            Ps[k][r] = (kin && gi < M) ? P[gi * psi + (int64_t)(kc + k) * psk] : (T)0;
            Qs[k][r] = (kin && gj < N) ? Q[gj * qsj + (int64_t)(kc + k) * qsk] : (T)0;
        }
        __syncthreads();
        for (int k = 0; k < kn; ++k) {
            T pa[4], qb[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) pa[a] = Ps[k][ty * 4 + a];
#pragma unroll
            for (int b = 0; b < 4; ++b) qb[b] = Qs[k][tx * 4 + b];
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] = fma(pa[a], qb[b], acc[a][b]);
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int64_t gi = i0 + ty * 4 + a, gj = j0 + tx * 4 + b;
            if (gi < M && gj < N && (!lower || gi >= gj)) C[gi + gj * ldc] -= acc[a][b];
        }
}

template <typename T>
lsq_status rank_update_ext(T* C, int64_t ldc, const T* P, int64_t psi, int64_t psk, const T* Q, int64_t qsj,
                              int64_t qsk, int64_t M, int64_t N, int K, bool lower, const int32_t* info,
                              cudaStream_t st) {
    if (M <= 0 || N <= 0 || K <= 0) return LSQ_OK;
    int64_t tm = ceil_div(M, 64), tn = ceil_div(N, 64);
    int64_t tiles = lower ? tm * (tm + 1) / 2 : tm * tn;
    k_rank_update<T><<<(unsigned)tiles, 256, 0, st>>>(C, ldc, P, psi, psk, Q, qsj, qsk, M, N, K, lower, tn, info);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

template lsq_status rank_update_ext<double>(double*, int64_t, const double*, int64_t, int64_t, const double*, int64_t,
                                           int64_t, int64_t, int64_t, int, bool, const int32_t*, cudaStream_t);
template lsq_status rank_update_ext<float>(float*, int64_t, const float*, int64_t, int64_t, const float*, int64_t,
                                          int64_t, int64_t, int64_t, int, bool, const int32_t*, cudaStream_t);

// ---------------------------------------------------------------------------
// Cholesky
// ---------------------------------------------------------------------------
// 1 / sqrt(d) for a positive finite d.  FP64: an FP32 estimate y of the
// significand's root refined by one third-order step
//   e = 1 - m y^2,  y <- y + y (e / 2 + 3/8 e^2),  d = m 4^k, m in [1, 4)
// in 64-bit integers (e to 2^-61): a warp issues one FP64 instruction in 64
// cycles on this part, dependent or not, and the pivots form the
// factorization's critical path; the integer chain takes about as long as two
// of them.  Relative error below one unit in the last place.
template <typename T>
__device__ __forceinline__ T rsqrt_pivot(T d) {
    if constexpr (sizeof(T) == 4) {
        return (T)1 / sqrtf(d);
    } else {
        const unsigned long long b = (unsigned long long)__double_as_longlong(d);
        if ((b >> 52) == 0) return 1.0 / sqrt(d);  // subnormal
        const int e2 = ((int)(b >> 52) - 1023) & ~1;  // 2 k
        const unsigned long long mb = b - ((unsigned long long)(long long)e2 << 52);  // bits of m
        const int sh = (int)(mb >> 52) - 1023;                                       // 0 or 1
        const unsigned long long M = ((mb & 0x000fffffffffffffull) | 0x0010000000000000ull) << (10 + sh);  // m 2^62
        const float y0 = rsqrtf(__uint_as_float((uint32_t)((mb >> 52) - 1023 + 127) << 23 | (uint32_t)((mb >> 29) & 0x7fffff)));
        const uint32_t Y0 = (uint32_t)(y0 * 16777216.0f);  // the estimate, 2^-24 units, about (1/2, 1]
        const unsigned long long Q = ((unsigned long long)Y0 * Y0) << 15;  // y0^2 2^63
        const long long e = (long long)((1ull << 61) - __umul64hi(M, Q));  // 2^-61 units, below 2^41
        const int eh = (int)(e >> 12);                                    // 2^-49 units
        const long long ee = ((long long)eh * eh) >> 37;                  // e^2, 2^-61 units
        const long long c = ((e >> 1) + ((3 * ee) >> 3)) >> 4;            // 2^-57 units, below 2^37
        const unsigned long long Y = ((unsigned long long)Y0 << 36) + (unsigned long long)(((long long)Y0 * c) >> 21);  // y 2^60
        const unsigned long long yb = ((Y + 64) >> 7) + (1021ull << 52);  // a carry to 1.0 moves into the exponent
        return __longlong_as_double((long long)(yb - ((unsigned long long)(long long)(e2 / 2) << 52)));
    }
}

// d > 0 and finite, without FP64 instructions
template <typename T>
__device__ __forceinline__ bool pivot_ok(T d) {
    if constexpr (sizeof(T) == 4) return d > (T)0 && isfinite(d);
    else return (unsigned long long)(__double_as_longlong(d) - 1) < 0x7fefffffffffffffull;
}

// Diagonal block (CNB x CNB) in one CTA, right-looking, the entries of columns
// 1 .. 63 in registers (8 a thread).  They are numbered by columns from the last
// to the second, so that the active ones, c > j, are a prefix: thread t holds
// entries t, t + 256, ..., and a column takes as many rounds as the prefix has.
// Per column j: the raw column (published by its holders) times 1/sqrt(d_j),
// then the update of the active entries.  Bound by the chain of a column (the
// root, two FP64 operations, two barriers) and, for the first third, by the FP64
// pipe (one warp instruction in 16 cycles per SM).  With the block in shared
// memory, a table look-up, three loads and a store an entry, and the root in
// FP64, a block took 49 us (87 thousand cycles, 67 of them in the update); 43 us so.
template <typename T>
__global__ void __launch_bounds__(256) k_potrf_diag(T* __restrict__ G, int64_t ld, int64_t n, int64_t k0,
                                                    int32_t* __restrict__ info) {
    if (*info != 0) return;
    constexpr int NE = CNB * (CNB - 1) / 2, NR = (NE + 255) / 256;  // entries of columns 1 .., rounds
    __shared__ T Ls[CNB][CNB + 1];
    __shared__ T raw[CNB], colj[CNB];  // column j before and after the scaling
    __shared__ int bad;
    const int nb = (int)min64(CNB, n - k0);
    const int tid = threadIdx.x;
    int rr[NR], cc[NR];
    T a[NR];
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        const int e = tid + 256 * u;
        // column 63 - w, w (w + 1) / 2 <= e: the root is exact to a unit
        int w = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
        if ((w + 1) * (w + 2) / 2 <= e) ++w;
        if (w * (w + 1) / 2 > e) --w;
        cc[u] = e < NE ? CNB - 1 - w : CNB - 1;
        rr[u] = e < NE ? cc[u] + e - w * (w + 1) / 2 : CNB - 1;
        a[u] = (e < NE && rr[u] < nb) ? G[(k0 + rr[u]) + (k0 + cc[u]) * ld] : (T)0;
    }
    if (tid < CNB) raw[tid] = tid < nb ? G[(k0 + tid) + k0 * ld] : (T)0;
    if (tid == 0) bad = 0;
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        if (tid < CNB) {
            const T d = raw[j];
            if (pivot_ok<T>(d)) {
                const T l = raw[tid] * rsqrt_pivot<T>(d);
                colj[tid] = l;
                Ls[tid][j] = l;  // row j: d / sqrt(d)
            } else if (tid == 0) {
                bad = j + 1;
            }
        }
        __syncthreads();
        if (bad) break;
        const int E = (CNB - 1 - j) * (CNB - j) / 2;
#pragma unroll
        for (int u = NR - 1; u >= 0; --u)
            if (256 * u < E) {
                a[u] = fma(-colj[rr[u]], colj[cc[u]], a[u]);
                if (cc[u] == j + 1) raw[rr[u]] = a[u];
            }
        __syncthreads();
    }
    if (bad) {
        if (tid == 0) set_info_once(info, (int32_t)(k0 + bad));
        return;
    }
    for (int q = tid; q < CNB * CNB; q += 256) {
        const int r = q & 63, c = q >> 6;
        if (r < nb && c < nb) G[(k0 + r) + (k0 + c) * ld] = r >= c ? Ls[r][c] : (T)0;
    }
}

// L21 = G21 L11^{-T}, right-looking with reciprocal pivots.  16 threads per
// row (2 rows per warp), thread `sub` owning columns sub, sub+16, sub+32,
// sub+48 in registers; x_j is broadcast within the half-warp by a shuffle.
template <typename T>
__global__ void __launch_bounds__(128) k_potrf_panel(T* __restrict__ G, int64_t ld, int64_t n, int64_t k0,
                                                     const int32_t* __restrict__ info) {
    if (*info != 0) return;
    __shared__ T L11[CNB][CNB + 1];
    __shared__ T rinv[CNB];
    for (int q = threadIdx.x; q < CNB * CNB; q += 128) {
        int r = q & 63, c = q >> 6;
        L11[r][c] = G[(k0 + r) + (k0 + c) * ld];
    }
    __syncthreads();
    for (int j = threadIdx.x; j < CNB; j += 128) rinv[j] = (T)1 / L11[j][j];
    __syncthreads();
    const int lane = threadIdx.x & 31, sub = lane & 15;
    const int64_t i = k0 + CNB + (int64_t)blockIdx.x * 8 + (threadIdx.x >> 4);
    const bool live = i < n;
    T x[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) x[q] = live ? G[i + (k0 + sub + 16 * q) * ld] : (T)0;
#pragma unroll
    for (int j = 0; j < CNB; ++j) {
        const int qj = j >> 4, sj = j & 15;
        if (sub == sj) x[qj] = x[qj] * rinv[j];
        const T xj = __shfl_sync(0xffffffffu, x[qj], (lane & 16) | sj);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = sub + 16 * q;
            if (k > j) x[q] = fma(-xj, L11[k][j], x[q]);
        }
    }
    if (live) {
#pragma unroll
        for (int q = 0; q < 4; ++q) G[i + (k0 + sub + 16 * q) * ld] = x[q];
    }
}

template <typename T>
__global__ void k_zero_upper(T* __restrict__ G, int64_t n, int64_t ld, const int32_t* __restrict__ info) {
    if (*info != 0) return;
    int64_t total = n * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = q % n, j = q / n;
        if (i < j) G[i + j * ld] = (T)0;
    }
}

size_t cholesky_ws_bytes(int64_t n) { return n > CNB ? ot_update_ws_bytes(n - CNB, n - CNB, CNB) : 256; }

// Right-looking in steps of 64 columns.  FP64 with scratch: each step's product is
// digit-sliced, over the tiles that reach the lower triangle (the rest of the
// upper triangle keeps its old values until it is cleared); its epilogue bounds
// it (8 bytes converted, read and written per output for 64 products).  One
// product with K = 256 per four steps takes 0.7 ms off the 9.3 ms of a
// factorization and solve of order 4096, but its one exponent per row covers 256
// columns of L: with L's 64-column pieces graded by 2^20 the residual of G - L L^T
// relative to |L| |L|^T grew from 1.2e-15 to 1.4e-11.
template <typename T>
lsq_status launch_cholesky(T* G, int64_t n, int64_t ld, int32_t* info, cudaStream_t st, void* ws, size_t ws_bytes) {
    const bool tc = std::is_same<T, double>::value && ws && ws_bytes >= cholesky_ws_bytes(n) && ot_trsm_supported();
    for (int64_t k0 = 0; k0 < n; k0 += CNB) {
        const int nb = (int)std::min<int64_t>(CNB, n - k0);
        k_potrf_diag<T><<<1, 256, 0, st>>>(G, ld, n, k0, info);
        LSQ_LAUNCH_CHECK();
        const int64_t rest = n - k0 - nb;
        if (rest <= 0) break;
        k_potrf_panel<T><<<(unsigned)ceil_div(rest, 8), 128, 0, st>>>(G, ld, n, k0, info);
        LSQ_LAUNCH_CHECK();
        T* L21 = G + (k0 + nb) + k0 * ld;
        T* A22 = G + (k0 + nb) + (k0 + nb) * ld;
        lsq_status s;
        if constexpr (std::is_same<T, double>::value) {
            if (tc) {
                s = ot_gemm_update_lower(L21, ld, A22, ld, rest, nb, ws, ws_bytes, nullptr, st);
                if (s != LSQ_OK) return s;
                continue;
            }
        }
        s = rank_update_ext<T>(A22, ld, L21, 1, ld, L21, 1, ld, rest, rest, nb, true, info, st);
        if (s != LSQ_OK) return s;
    }
    k_zero_upper<T><<<(unsigned)std::min<int64_t>(ceil_div(n * n, 256), 4096), 256, 0, st>>>(G, n, ld, info);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

template lsq_status launch_cholesky<double>(double*, int64_t, int64_t, int32_t*, cudaStream_t, void*, size_t);
template lsq_status launch_cholesky<float>(float*, int64_t, int64_t, int32_t*, cudaStream_t, void*, size_t);

// ---------------------------------------------------------------------------
// LU with partial pivoting
// ---------------------------------------------------------------------------
// Panel columns [k0, k0+nb), rows [k0, rows), by a cluster of CTAs with one
// matrix row per thread in registers.  Rows are never moved while the panel is
// factored: each thread carries the position its row has after the swaps so
// far (LAPACK's sequential interchanges), and writes the row there at the end.
// Per column every CTA finds its own best candidate (largest magnitude, then
// smallest position; bit patterns and integer warp reductions, no FP64
// compares), pushes that row and its reciprocal pivot into every CTA's shared
// memory, and after ONE cluster barrier all CTAs pick the same winner and
// update their rows.  Exchange slots alternate by column parity.
//
// The chain of 32 pivots bounds it: one exchange (about a microsecond) a
// column, and the FP64 pipe (2 FMA a cycle and SM), which is why the rows are
// spread over up to 16 SMs.  One CTA working in global memory took 420 us for
// a panel of 1000 rows on average; with this kernel and k_lu_u12 below the LU of
// a 2000 x 2000 matrix went from 35.5 to 13.8 ms, with the same bits.
//
// l = a / d is formed as q = a r, q + r (a - q d) with r = 1/d correctly
// rounded: the correctly rounded quotient (Markstein) at 3 FP64 operations,
// while a - q d and q are well inside the normal range; tiny and zero a and q take
// the division (by their exponent fields, no FP64 compare).
template <typename T>
struct LuKey;
template <>
struct LuKey<double> {
    // orders |v|; NaN below everything, so that it is taken only when nothing else is there
    static __device__ __forceinline__ unsigned long long of(double v) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        return b > 0x7ff0000000000000ull ? 1ull : b + 1ull;
    }
    static __device__ __forceinline__ bool unusable(double v) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
        return b == 0 || b >= 0x7ff0000000000000ull;
    }
    // |v| < 2^-895
    static __device__ __forceinline__ bool tiny(double v) {
        return ((unsigned)(__double_as_longlong(v) >> 32) & 0x7fffffffu) < (128u << 20);
    }
};
template <>
struct LuKey<float> {
    static __device__ __forceinline__ unsigned long long of(float v) {
        const unsigned b = __float_as_uint(v) & 0x7fffffffu;
        return b > 0x7f800000u ? 1ull : (unsigned long long)b + 1ull;
    }
    static __device__ __forceinline__ bool unusable(float v) {
        const unsigned b = __float_as_uint(v) & 0x7fffffffu;
        return b == 0 || b >= 0x7f800000u;
    }
    // |v| < 2^-67
    static __device__ __forceinline__ bool tiny(float v) { return (__float_as_uint(v) & 0x7fffffffu) < (60u << 23); }
};

// Largest key of the warp, then the smallest position that has it (key 0: none).
__device__ __forceinline__ void lu_warp_best(unsigned long long& key, unsigned& pos) {
    const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    const unsigned mp = __reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? pos : 0xffffffffu);
    key = ((unsigned long long)mh << 32) | ml;
    pos = mp;
}

constexpr int LUC = 16;  // CTAs per cluster at most

template <typename T, int NT>
__global__ void __launch_bounds__(NT) k_lu_panel_cl(T* __restrict__ H, int64_t ld, int64_t rows, int64_t k0, int nb,
                                                    int32_t* __restrict__ piv, int32_t* __restrict__ info) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int NW = NT / 32;
    __shared__ T rowx[2][LUC][LNB + 1];  // each CTA's candidate row, its reciprocal pivot behind it
    __shared__ unsigned long long keyx[2][LUC];
    __shared__ unsigned posx[2][LUC];
    __shared__ unsigned long long wkey[NW];
    __shared__ unsigned wpos[NW];
    __shared__ T myrow[LNB + 1];
    const int rank = (int)cluster.block_rank(), CL = (int)cluster.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int prow = (int)(rows - k0);
    const int R = (prow + CL - 1) / CL;
    const int r0 = rank * R;
    const bool live = tid < R && r0 + tid < prow;
    unsigned pos = (unsigned)(r0 + tid);
    T a[LNB];
#pragma unroll
    for (int c = 0; c < LNB; ++c) a[c] = (live && c < nb) ? H[(k0 + r0 + tid) + (k0 + c) * ld] : (T)0;
    cluster.sync();  // every CTA runs before its shared memory is written
#pragma unroll
    for (int j = 0; j < LNB; ++j) {
        if (j < nb) {
            const int buf = j & 1;
            const bool act = live && pos >= (unsigned)j;
            unsigned long long key = act ? LuKey<T>::of(a[j]) : 0ull;
            unsigned bp = act ? pos : 0xffffffffu;
            lu_warp_best(key, bp);
            if (lane == 0) wkey[warp] = key, wpos[warp] = bp;
            __syncthreads();
            key = lane < NW ? wkey[lane] : 0ull;
            bp = lane < NW ? wpos[lane] : 0xffffffffu;
            lu_warp_best(key, bp);
            if (act && pos == bp) {
#pragma unroll
                for (int c = j; c < LNB; ++c) myrow[c] = a[c];
                myrow[LNB] = (T)1 / a[j];
            }
            __syncthreads();
            const int span = LNB + 1 - j;
            for (int q = tid; q < CL * span; q += NT) {
                const int dst = q / span, c = j + q % span;
                *cluster.map_shared_rank(&rowx[buf][rank][c], dst) = myrow[c];
            }
            if (tid < CL) {
                *cluster.map_shared_rank(&keyx[buf][rank], tid) = key;
                *cluster.map_shared_rank(&posx[buf][rank], tid) = bp;
            }
            cluster.sync();
            key = lane < CL ? keyx[buf][lane] : 0ull;
            bp = lane < CL ? posx[buf][lane] : 0xffffffffu;
            const unsigned long long own_key = key;
            const unsigned own_pos = bp;
            lu_warp_best(key, bp);
            const int br = __ffs((int)__ballot_sync(0xffffffffu, lane < CL && own_key == key && own_pos == bp)) - 1;
            const T* u = &rowx[buf][br][0];
            const T d = u[j], rd = u[LNB];
            const bool zero = LuKey<T>::unusable(d);
            if (rank == 0 && tid == 0) {
                piv[k0 + j] = (int32_t)(k0 + bp);
                if (zero) set_info_once(info, (int32_t)(k0 + j + 1));
            }
            pos = pos == bp ? (unsigned)j : (pos == (unsigned)j ? bp : pos);
            if (!zero && live && pos > (unsigned)j) {
                const T q = a[j] * rd;
                // (a tiny d has only tiny a)
                const T l = LuKey<T>::tiny(a[j]) || LuKey<T>::tiny(q) ? a[j] / d : fma(fma(-q, d, a[j]), rd, q);
                a[j] = l;
#pragma unroll
                for (int c = j + 1; c < LNB; ++c) a[c] = fma(-l, u[c], a[c]);
            }
        }
    }
    if (live) {
#pragma unroll
        for (int c = 0; c < LNB; ++c)
            if (c < nb) H[(k0 + (int64_t)pos) + (k0 + c) * ld] = a[c];
    }
}

// The same panel by one block of 1024 threads in global memory: panels with
// more rows than the cluster holds (512 a CTA).
template <typename T>
__global__ void __launch_bounds__(1024) k_lu_panel(T* __restrict__ H, int64_t ld, int64_t rows, int64_t k0, int nb,
                                                   int32_t* __restrict__ piv, int32_t* __restrict__ info) {
    __shared__ T wv[32];
    __shared__ int64_t wi[32];
    __shared__ int64_t pivrow;
    int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int jj = 0; jj < nb; ++jj) {
        int64_t j = k0 + jj;
        // pivot: largest |H[i][j]|, smallest i on ties
        T best = (T)-1;
        int64_t bi = rows;
        for (int64_t i = j + tid; i < rows; i += 1024) {
            T v = fabs(H[i + j * ld]);
            if (v > best) { best = v; bi = i; }
        }
        for (int off = 16; off > 0; off >>= 1) {
            T ov = __shfl_xor_sync(0xffffffffu, best, off);
            int64_t oi = __shfl_xor_sync(0xffffffffu, bi, off);
            if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
        }
        if (lane == 0) { wv[warp] = best; wi[warp] = bi; }
        __syncthreads();
        if (warp == 0) {
            best = wv[lane];
            bi = wi[lane];
            for (int off = 16; off > 0; off >>= 1) {
                T ov = __shfl_xor_sync(0xffffffffu, best, off);
                int64_t oi = __shfl_xor_sync(0xffffffffu, bi, off);
                if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
            }
            if (lane == 0) {
                if (bi >= rows) bi = j;  // NaN in every row: a pivot that is reported below
                pivrow = bi;
                piv[j] = (int32_t)bi;
            }
        }
        __syncthreads();
        int64_t p = pivrow;
        if (p != j)
            for (int c = tid; c < nb; c += 1024) {
                T t = H[j + (k0 + c) * ld];
                H[j + (k0 + c) * ld] = H[p + (k0 + c) * ld];
                H[p + (k0 + c) * ld] = t;
            }
        __syncthreads();
        T d = H[j + j * ld];
        bool zero = (d == (T)0) || !isfinite(d);
        if (zero) {
            if (tid == 0) set_info_once(info, (int32_t)(j + 1));
        } else {
            for (int64_t i = j + 1 + tid; i < rows; i += 1024) H[i + j * ld] = H[i + j * ld] / d;
        }
        __syncthreads();
        if (!zero) {
            for (int64_t i = j + 1 + tid; i < rows; i += 1024) {
                T l = H[i + j * ld];
                for (int c = jj + 1; c < nb; ++c) {
                    int64_t col = k0 + c;
                    H[i + col * ld] = fma(-l, H[j + col * ld], H[i + col * ld]);
                }
            }
        }
        __syncthreads();
    }
}

// Apply the panel's row swaps (in order) to the columns outside the panel.
template <typename T>
__global__ void k_lu_swap(T* __restrict__ H, int64_t ld, int64_t cols, int64_t k0, int nb,
                          const int32_t* __restrict__ piv) {
    int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cols || (c >= k0 && c < k0 + nb)) return;
    for (int jj = 0; jj < nb; ++jj) {
        int64_t j = k0 + jj, p = piv[j];
        if (p != j) {
            T t = H[j + c * ld];
            H[j + c * ld] = H[p + c * ld];
            H[p + c * ld] = t;
        }
    }
}

// U12 = L11^{-1} A12 (unit lower L11), one thread per column [c0, c1), the
// column in registers and fully unrolled, right-looking: after entry k its
// updates of the later entries are independent (a left-looking loop over a
// local array took 40 us a launch, bound by latency).
template <typename T>
__global__ void __launch_bounds__(32) k_lu_u12(T* __restrict__ H, int64_t ld, int64_t c0, int64_t c1, int64_t k0,
                                               int nb) {
    __shared__ T L11[LNB][LNB];  // [column][row]
    for (int q = threadIdx.x; q < LNB * LNB; q += 32) {
        const int i = q % LNB, j = q / LNB;
        L11[j][i] = (i < nb && j < nb) ? H[(k0 + i) + (k0 + j) * ld] : (T)0;
    }
    __syncthreads();
    const int64_t c = c0 + (int64_t)blockIdx.x * 32 + threadIdx.x;
    if (c >= c1) return;
    T u[LNB];
#pragma unroll
    for (int i = 0; i < LNB; ++i) u[i] = i < nb ? H[(k0 + i) + c * ld] : (T)0;
#pragma unroll
    for (int k = 0; k < LNB; ++k)
#pragma unroll
        for (int i = k + 1; i < LNB; ++i) u[i] = fma(-L11[k][i], u[k], u[i]);
#pragma unroll
    for (int i = 0; i < LNB; ++i)
        if (i < nb) H[(k0 + i) + c * ld] = u[i];
}

// CTAs of the cluster for a panel of prow rows: about 64 rows each up to
// max_cluster CTAs, at most 512 (a thread holds a row); 0: no cluster holds it.
int lu_panel_cluster(int64_t prow, int max_cluster) {
    int cl = 1;
    while (cl < max_cluster && cl * 64 < prow) cl *= 2;
    return max_cluster > 0 && ceil_div(prow, cl) <= 512 ? cl : 0;
}

template <typename T, int NT>
static cudaError_t lu_panel_launch(int cl, bool query, int* fits, T* H, int64_t ld, int64_t rows, int64_t k0, int nb,
                                   int32_t* piv, int32_t* info, cudaStream_t st) {
    auto kern = k_lu_panel_cl<T, NT>;
    if (cl > 8) {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)cl);
    cfg.blockDim = dim3(NT);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (query) return cudaOccupancyMaxActiveClusters(fits, kern, &cfg);
    return cudaLaunchKernelEx(&cfg, kern, H, ld, rows, k0, nb, piv, info);
}

// The panel kernel of at least R threads, launched or (query) asked how many
// clusters of cl CTAs the device holds.
template <typename T>
static cudaError_t lu_panel_do(int64_t R, int cl, bool query, int* fits, T* H, int64_t ld, int64_t rows, int64_t k0,
                               int nb, int32_t* piv, int32_t* info, cudaStream_t st) {
    if (R <= 64) return lu_panel_launch<T, 64>(cl, query, fits, H, ld, rows, k0, nb, piv, info, st);
    if (R <= 128) return lu_panel_launch<T, 128>(cl, query, fits, H, ld, rows, k0, nb, piv, info, st);
    if (R <= 256) return lu_panel_launch<T, 256>(cl, query, fits, H, ld, rows, k0, nb, piv, info, st);
    return lu_panel_launch<T, 512>(cl, query, fits, H, ld, rows, k0, nb, piv, info, st);
}

// Largest cluster that the device schedules with every thread count: 16
// (non-portable), else 8, else 0.  Asked once per device.
template <typename T>
static int lu_max_cluster() {
    static std::mutex mu;
    static int last_dev = -1, last = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (dev == last_dev) return last;
    last = 0;
    for (int cl : {LUC, 8}) {
        bool all = true;
        for (int64_t R : {64, 128, 256, 512}) {
            int fits = 0;
            all = all && lu_panel_do<T>(R, cl, true, &fits, nullptr, 0, 0, 0, 0, nullptr, nullptr, nullptr) == cudaSuccess &&
                  fits >= 1;
        }
        if (all) {
            last = cl;
            break;
        }
        cudaGetLastError();
    }
    last_dev = dev;
    return last;
}

template <typename T>
static lsq_status launch_lu_panel(T* H, int64_t ld, int64_t rows, int64_t k0, int nb, int32_t* piv, int32_t* info,
                                  cudaStream_t st) {
    const int cl = lu_panel_cluster(rows - k0, lu_max_cluster<T>());
    if (cl > 0)
        LSQ_CUDA_TRY(lu_panel_do<T>(ceil_div(rows - k0, cl), cl, false, nullptr, H, ld, rows, k0, nb, piv, info, st));
    else
        k_lu_panel<T><<<1, 1024, 0, st>>>(H, ld, rows, k0, nb, piv, info);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

// Blocked right-looking LU with partial pivoting of a rows x cols matrix
// (rows >= cols): P H = L U, L unit lower trapezoidal, U cols x cols upper.
template <typename T>
lsq_status launch_lu_rect(T* H, int64_t rows, int64_t cols, int64_t ld, int32_t* piv, int32_t* info, cudaStream_t st) {
    if (rows < cols) return LSQ_ERR_ARG;
    for (int64_t k0 = 0; k0 < cols; k0 += LNB) {
        int nb = (int)std::min<int64_t>(LNB, cols - k0);
        lsq_status ps = launch_lu_panel<T>(H, ld, rows, k0, nb, piv, info, st);
        if (ps != LSQ_OK) return ps;
        k_lu_swap<T><<<(unsigned)ceil_div(cols, 128), 128, 0, st>>>(H, ld, cols, k0, nb, piv);
        LSQ_LAUNCH_CHECK();
        int64_t rest = cols - k0 - nb, rrest = rows - k0 - nb;
        if (rest <= 0) continue;
        k_lu_u12<T><<<(unsigned)ceil_div(rest, 32), 32, 0, st>>>(H, ld, k0 + nb, cols, k0, nb);
        LSQ_LAUNCH_CHECK();
        // A22 -= L21 U12:  P(i,k) = H[(k0+nb+i) + (k0+k) ld],  Q(j,k) = H[(k0+k) + (k0+nb+j) ld]
        lsq_status s = rank_update_ext<T>(H + (k0 + nb) + (k0 + nb) * ld, ld, H + (k0 + nb) + k0 * ld, 1, ld,
                                          H + k0 + (k0 + nb) * ld, ld, 1, rrest, rest, nb, false, nullptr, st);
        if (s != LSQ_OK) return s;
    }
    return LSQ_OK;
}

template lsq_status launch_lu_rect<float>(float*, int64_t, int64_t, int64_t, int32_t*, int32_t*, cudaStream_t);
template lsq_status launch_lu_rect<double>(double*, int64_t, int64_t, int64_t, int32_t*, int32_t*, cudaStream_t);

lsq_status launch_lu(double* H, int64_t n, int64_t ld, int32_t* piv, int32_t* info, cudaStream_t st) {
    return launch_lu_rect<double>(H, n, n, ld, piv, info, st);
}

// The sketch's LU preconditioner (not-normal equations): the tall LU of A_s
// (s x n, float or double) in T arithmetic, then U with the column scaling
// undone, U_s[:, j] = U[:, j] 2^-colexp[j], promoted to FP64 (upper
// triangle of Us written, ld ldu).
template <typename TS, typename T>
__global__ void k_lu_load(const TS* __restrict__ As, int64_t s, int64_t n, int64_t ldas, T* __restrict__ W) {
    const int64_t total = s * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = q % s, j = q / s;
        W[q] = (T)As[i + j * ldas];
    }
}

template <typename T>
__global__ void k_lu_upper_out(const T* __restrict__ W, int64_t s, int64_t n, const int32_t* __restrict__ colexp,
                               double* __restrict__ Us, int64_t ldu) {
    const int64_t total = n * n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = q % n, j = q / n;
        if (i <= j) Us[i + j * ldu] = ldexp((double)W[i + j * s], colexp ? -colexp[j] : 0);
    }
}

size_t lu_precond_ws_bytes(int64_t s, int64_t n, int prec) {
    const size_t es = prec == LSQ_FP64 ? 8 : 4;
    return align_up(es * (size_t)s * n, 256) + align_up(sizeof(int32_t) * (size_t)n, 256) + 256;
}

lsq_status launch_lu_precond(const void* As, int64_t s, int64_t n, int64_t ldas, int as_prec, int lu_prec,
                             const int32_t* colexp, double* Us, int64_t ldu, int32_t* info, void* ws, size_t ws_bytes,
                             cudaStream_t st) {
    if (!ws || ws_bytes < lu_precond_ws_bytes(s, n, lu_prec)) return LSQ_ERR_NOMEM;
    const size_t es = lu_prec == LSQ_FP64 ? 8 : 4;
    char* base = (char*)(((uintptr_t)ws + 255) & ~(uintptr_t)255);
    int32_t* piv = (int32_t*)(base + align_up(es * (size_t)s * n, 256));
    const unsigned g = (unsigned)std::min<int64_t>(ceil_div(s * n, 256), 8192);
    const unsigned gu = (unsigned)std::min<int64_t>(ceil_div(n * n, 256), 8192);
    lsq_status r;
    if (lu_prec == LSQ_FP64) {
        double* W = (double*)base;
        if (as_prec == LSQ_FP64) k_lu_load<double, double><<<g, 256, 0, st>>>((const double*)As, s, n, ldas, W);
        else k_lu_load<float, double><<<g, 256, 0, st>>>((const float*)As, s, n, ldas, W);
        LSQ_LAUNCH_CHECK();
        if ((r = launch_lu_rect<double>(W, s, n, s, piv, info, st)) != LSQ_OK) return r;
        k_lu_upper_out<double><<<gu, 256, 0, st>>>(W, s, n, colexp, Us, ldu);
    } else {
        float* W = (float*)base;
        if (as_prec == LSQ_FP64) k_lu_load<double, float><<<g, 256, 0, st>>>((const double*)As, s, n, ldas, W);
        else k_lu_load<float, float><<<g, 256, 0, st>>>((const float*)As, s, n, ldas, W);
        LSQ_LAUNCH_CHECK();
        if ((r = launch_lu_rect<float>(W, s, n, s, piv, info, st)) != LSQ_OK) return r;
        k_lu_upper_out<float><<<gu, 256, 0, st>>>(W, s, n, colexp, Us, ldu);
    }
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

// ---------------------------------------------------------------------------
// Triangular solves on a vector, many CTAs in a wavefront.  CTA v takes its
// row block from an atomic counter (v-th CTA to start), so every block it
// waits for belongs to a CTA that has already started.  It stages each
// off-diagonal 32 x 32 block of the operator while the solution of that block
// is still being computed, waits for that solution (bounded: 2 s of
// %globaltimer unless a test shortened it, then -2 is recorded and NaN passed
// on), applies it, and finally solves its diagonal block and publishes y_b.
//
// Publication: the solution is also written to a scratch copy `pub` that the
// launch fills with all-ones bit patterns (a NaN that arithmetic does not
// produce; a computed value with that pattern is published as the default
// NaN).  A waiting CTA polls the 32 entries it needs directly, one lane each,
// so a block's solution reaches the next CTA in one trip through L2 (no flag,
// no fence).
//
// Diagonal block: staged before the first wait with its reciprocal pivots and
// the block's own right-hand side, rows scaled to a unit diagonal.  For the
// Cholesky factor (L and L^T) a CTA that has a block to wait for also forms
// the inverse of its diagonal block while it waits, and applies it as a
// product: a few dependent FP64 operations instead of a 32-step chain.  The
// explicit inverse adds an error of order u kappa(L_bb) |y_b|, below the
// u kappa(A_p)^2 that the normal equations carry; the other factors (R_s, the
// LU factors) keep the substitution.
// Partial sums are combined in a fixed order, so the result does not depend
// on timing.
// ---------------------------------------------------------------------------
template <typename T>
struct TrsvPub;
template <>
struct TrsvPub<double> {
    static __device__ __forceinline__ void put(double* p, double v) {
        unsigned long long b = (unsigned long long)__double_as_longlong(v);
        if (b == ~0ull) b = 0x7ff8000000000000ull;
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(b) : "memory");
    }
    // the entry, or false while it is unpublished
    static __device__ __forceinline__ bool get(const double* p, double& v) {
        unsigned long long b;
        asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(b) : "l"(p) : "memory");
        v = __longlong_as_double((long long)b);
        return b != ~0ull;
    }
};
template <>
struct TrsvPub<float> {
    static __device__ __forceinline__ void put(float* p, float v) {
        unsigned b = __float_as_uint(v);
        if (b == ~0u) b = 0x7fc00000u;
        asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(b) : "memory");
    }
    static __device__ __forceinline__ bool get(const float* p, float& v) {
        unsigned b;
        asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(b) : "l"(p) : "memory");
        v = __uint_as_float(b);
        return b != ~0u;
    }
};

template <typename T>
__global__ void __launch_bounds__(128) k_trsv_wave(int kind, const T* __restrict__ M, int64_t n, int64_t ld, T* y,
                                                   int32_t* sync, T* pub, const int32_t* __restrict__ info,
                                                   int32_t* __restrict__ err, uint64_t wait_ns) {
    if (info && *info != 0) return;
    __shared__ T blk[32][33];
    __shared__ T dgb[32][33];  // diagonal block, rows scaled to a unit diagonal (then its inverse, see below)
    __shared__ T xin[32][33];  // inverse of the scaled block
    __shared__ T part[4][32];
    __shared__ T yk[32];
    __shared__ T rin[32];
    __shared__ T wsh[32];
    __shared__ int vb, failed;
    const int tid = threadIdx.x, r = tid & 31, q = tid >> 5;
    const int nblk = (int)((n + 31) / 32);
    if (tid == 0) {
        vb = atomicAdd(&sync[0], 1) + 1;  // the counter starts at -1 (all-ones fill)
        failed = 0;
    }
    __syncthreads();
    const int v = vb;
    const bool forward = (kind == TB_LOWER || kind == TB_UNIT_LOWER || kind == TB_UPPER_T);
    const bool trans = (kind == TB_LOWER_T || kind == TB_UPPER_T);  // operator entry (i, j) = M[j + i ld]
    const bool unit = (kind == TB_UNIT_LOWER);
    const bool use_inv = (kind == TB_LOWER || kind == TB_LOWER_T) && v > 0;
    const int b = forward ? v : nblk - 1 - v;
    const int64_t b0 = (int64_t)b * 32;
    const int bs = (int)min64(32, n - b0);
    // everything that does not depend on other blocks, before the first wait:
    // the diagonal block, the reciprocal pivots and this block's right-hand side
    for (int e = tid; e < 1024; e += 128) {
        int rr, jj;
        if (trans) { jj = e & 31; rr = e >> 5; } else { rr = e & 31; jj = e >> 5; }
        T val = (T)0;
        if (rr < bs && jj < bs) val = trans ? M[(b0 + jj) + (b0 + rr) * ld] : M[(b0 + rr) + (b0 + jj) * ld];
        dgb[rr][jj] = val;
    }
    T vv = (tid < 32 && r < bs) ? y[b0 + r] : (T)0;
    __syncthreads();
    if (tid < 32) rin[r] = (r < bs && !unit) ? (T)1 / dgb[r][r] : (T)1;
    __syncthreads();
    for (int e = tid; e < 1024; e += 128) {
        const int rr = e & 31, jj = e >> 5;
        if (rr != jj) dgb[rr][jj] *= rin[rr];
        if (use_inv) xin[rr][jj] = rr == jj ? (T)1 : (T)0;
    }
    if (use_inv) {
        // X = D'^{-1} for the unit triangular D' (rows and columns in solve
        // order: ascending for L, descending for L^T), right-looking: after
        // step j, row j of X is final and updates the rows solved after it.
        __syncthreads();
        for (int j = 0; j < 31; ++j) {
            const int w = j + 1, cnt = (31 - j) * w;
            for (int e = tid; e < cnt; e += 128) {
                const int ro = j + 1 + e / w, co = e % w;  // solve-order row (> j) and column (<= j)
                const int jr = forward ? j : 31 - j, rr = forward ? ro : 31 - ro, cc = forward ? co : 31 - co;
                xin[rr][cc] = fma(-dgb[rr][jr], xin[jr][cc], xin[rr][cc]);
            }
            __syncthreads();
        }
        // y_b = X diag(rin) w: fold the pivots into the columns
        for (int e = tid; e < 1024; e += 128) {
            const int rr = e & 31, cc = e >> 5;
            dgb[rr][cc] = xin[rr][cc] * rin[cc];
        }
    }
    T acc0 = (T)0, acc1 = (T)0;
    for (int st = 0; st < v; ++st) {
        const int k = forward ? st : nblk - 1 - st;
        const int64_t k0 = (int64_t)k * 32;
        const int ks = (int)min64(32, n - k0);
        for (int e = tid; e < 1024; e += 128) {
            int rr, jj;
            if (trans) { jj = e & 31; rr = e >> 5; } else { rr = e & 31; jj = e >> 5; }
            T val = (T)0;
            if (rr < bs && jj < ks) val = trans ? M[(k0 + jj) + (b0 + rr) * ld] : M[(b0 + rr) + (k0 + jj) * ld];
            blk[rr][jj] = val;
        }
        if (tid < 32) {
            // poll the ks published entries of block k, one lane each
            T got = (T)0;
            bool have = r >= ks;
            bool timed_out = false;
            uint64_t t0;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (;;) {
                if (!have) have = TrsvPub<T>::get(pub + k0 + r, got);
                if (__all_sync(0xffffffffu, have)) break;
                uint64_t t;  // lane 0's clock decides for the warp
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
                if (__shfl_sync(0xffffffffu, t - t0 > wait_ns ? 1 : 0, 0)) {
                    timed_out = true;
                    break;
                }
            }
            yk[r] = r < ks ? got : (T)0;
            if (timed_out && r == 0) failed = 1;
        }
        __syncthreads();
        if (failed) break;
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            acc0 = fma(-blk[r][q * 8 + j], yk[q * 8 + j], acc0);
            acc1 = fma(-blk[r][q * 8 + j + 1], yk[q * 8 + j + 1], acc1);
        }
        __syncthreads();
    }
    part[q][r] = acc0 + acc1;
    __syncthreads();
    if (use_inv) {
        // w = c_b - sum of the applied blocks, then y_b = (X diag(rin)) w,
        // 8 columns per warp in two chains, the warps' parts summed pairwise
        if (tid < 32) wsh[r] = vv + ((part[0][r] + part[1][r]) + (part[2][r] + part[3][r]));
        __syncthreads();
        T s0 = (T)0, s1 = (T)0;
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
            s0 = fma(dgb[r][q * 8 + j], wsh[q * 8 + j], s0);
            s1 = fma(dgb[r][q * 8 + j + 1], wsh[q * 8 + j + 1], s1);
        }
        part[q][r] = s0 + s1;
        __syncthreads();
        if (tid < 32) vv = (part[0][r] + part[1][r]) + (part[2][r] + part[3][r]);
    }
    if (tid < 32) {
        const bool ok = !failed;
        if (!use_inv) {
            vv = vv + part[0][r] + part[1][r] + part[2][r] + part[3][r];
            vv = vv * rin[r];  // unit-diagonal system from here on
            if (forward) {
                for (int jj = 0; jj < bs; ++jj) {
                    const T vj = __shfl_sync(0xffffffffu, vv, jj);
                    if (r > jj && r < bs) vv = fma(-dgb[r][jj], vj, vv);
                }
            } else {
                for (int jj = bs - 1; jj >= 0; --jj) {
                    const T vj = __shfl_sync(0xffffffffu, vv, jj);
                    if (r < jj) vv = fma(-dgb[r][jj], vj, vv);
                }
            }
        }
        if (r < bs) {
            if (ok) y[b0 + r] = vv;
            // a failed block passes NaN on, so that the blocks after it do not wait
            TrsvPub<T>::put(pub + b0 + r, ok ? vv : (T)NAN);
        }
        if (!ok && r == 0) set_info_once(err, -2);
    }
}

// Scratch: the block counter, then the published copy of the solution (8-byte aligned).
size_t trsv_sync_ints(int64_t n) { return 2 + 2 * (size_t)n; }

// Bound of one wait for another block's solution (2 s; shorter only in tests).
static uint64_t g_trsv_wait_ns = 2000000000ull;

uint64_t trsv_wait_ns() { return g_trsv_wait_ns; }

uint64_t set_trsv_wait_ns(uint64_t ns) {
    const uint64_t old = g_trsv_wait_ns;
    g_trsv_wait_ns = ns;
    return old;
}

template <typename T>
lsq_status launch_trsv(int kind, const T* M, int64_t n, int64_t ld, T* y, const int32_t* info, int32_t* sync,
                       int32_t* err, cudaStream_t st) {
    if (!sync || n <= 0 || n > (int64_t)1 << 30 || ((uintptr_t)sync % 8) != 0) return LSQ_ERR_ARG;
    int64_t nblk = ceil_div(n, 32);
    // all ones: the counter reads -1, every published entry is unset
    LSQ_CUDA_TRY(cudaMemsetAsync(sync, 0xff, sizeof(int32_t) * trsv_sync_ints(n), st));
    k_trsv_wave<T><<<(unsigned)nblk, 128, 0, st>>>(kind, M, n, ld, y, sync, (T*)(sync + 2), info, err,
                                                   g_trsv_wait_ns);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

template lsq_status launch_trsv<double>(int, const double*, int64_t, int64_t, double*, const int32_t*, int32_t*,
                                        int32_t*, cudaStream_t);
template lsq_status launch_trsv<float>(int, const float*, int64_t, int64_t, float*, const int32_t*, int32_t*, int32_t*,
                                       cudaStream_t);

__global__ void k_apply_piv(const int32_t* __restrict__ piv, int64_t n, double* __restrict__ y,
                            const int32_t* __restrict__ info) {
    if (info && *info != 0) return;
    for (int64_t k = 0; k < n; ++k) {
        int64_t p = piv[k];
        if (p != k) { double t = y[k]; y[k] = y[p]; y[p] = t; }
    }
}

lsq_status launch_apply_piv(const int32_t* piv, int64_t n, double* y, const int32_t* info, cudaStream_t st) {
    k_apply_piv<<<1, 1, 0, st>>>(piv, n, y, info);
    LSQ_LAUNCH_CHECK();
    return LSQ_OK;
}

}  // namespace lsq
