// Blocked Cholesky factorisation S = L L^T (arXiv:1705.11191 Eq. 8) and the blocked
// triangular solves with L used for the standard form H~ = L^{-1} H L^{-T} and the
// back-substitution c = L^{-T} c~ (Eq. 9).
//
// Right-looking blocked algorithm with block nb = kTriBlock: the nb x nb diagonal block is
// factorised and inverted by one CTA in shared memory; the panel below it is multiplied
// by the inverse (a GEMM) and the trailing matrix gets a lower-triangular rank-nb update
// (a GEMM restricted to the lower triangle). The triangular solves reuse the inverted
// diagonal blocks so that every O(n^3) flop is in a GEMM.
#include "common.cuh"
#include "kernels.h"
#include "packets.cuh"

namespace egb {

// One CTA: factor the jb x jb diagonal block at a (lower triangle read), write L back
// (upper part of the block zeroed) and its inverse to inv (ld ldi).
//
// Symmetric elimination with the inverse formed in the same pass: after step k the rows i > k
// hold the Schur complement in the columns c > k and, in the columns c <= k, the rows of the
// unit lower-triangular inverse (row i -= (a_ik / d_k) row k, with the identity understood in
// the columns already eliminated). L = columns / sqrt(d_k), inverse = rows / sqrt(d_i). Thread
// (row i, every fourth column) keeps its 16 entries in registers; a step publishes the pivot row
// and 1 / d_k through shared memory and has one block barrier. The steps are unrolled by register
// (four steps, one per column of a quad, in a loop), so that column k needs no search through the
// registers. What bounds it: 64 dependent steps, each a reciprocal, a barrier and a rank-1 update
// (in binary64 up to 4096 FMAs at two a clock). Factorising in shared memory with three barriers a
// step and then inverting column by column took 85 us (binary32) and 210 us (binary64) a block, with
// 16 consecutive columns a thread, picked out by predicated moves, 40 and 96 us, this 23 and 76 us.
template <typename T>
__global__ void __launch_bounds__(4 * kTriBlock)
potrf_diag_kernel(int jb, T *a, int lda, T *inv, int ldi, int *status, int pivot_base)
{
    constexpr int B = kTriBlock, CPT = B / 4;
    __shared__ __align__(16) T prow[2][4][CPT];  // pivot row: [part][q] is column 4 q + part
    __shared__ T prec[2];                        // 1 / d_k
    __shared__ T piv[B];                         // d_k
    __shared__ T Ls[B][B + 1];                   // a_ik (i > k), by column
    __shared__ int bad;
    const int tid = threadIdx.x, lane = tid & 31, quad = lane & ~3;
    const int i = tid >> 2, part = tid & 3;
    T E[CPT];
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        const int c = 4 * q + part, hi = max(i, c), lo = min(i, c);
        E[q] = hi < jb ? a[(size_t)hi + (size_t)lo * lda] : (i == c ? T(1) : T(0));
    }
    if (tid == 0) bad = -1;
    // row k of the next pivot and its reciprocal, published by the row's four threads; e is the entry
    // of the thread's column in the quad of column k
    auto publish = [&](int k, T e) {
        if (i == k) {
#pragma unroll
            for (int q = 0; q < CPT; ++q) prow[k & 1][part][q] = E[q];
            if (part == (k & 3)) {
                T d = e;
                if (!(d > T(0)) || !isfinite(d)) {
                    if (bad < 0) bad = k;
                    d = T(1);  // keep going with a harmless pivot; the status reports the failure
                }
                piv[k] = d;
                prec[k & 1] = recip(d);
            }
        }
    };
    __syncthreads();
    publish(0, E[0]);
    __syncthreads();
#pragma unroll
    for (int qk = 0; qk < CPT; ++qk)
#pragma unroll 1
        for (int pk = 0; pk < 4; ++pk) {
            const int k = 4 * qk + pk;
            const T aik = __shfl_sync(0xffffffffu, E[qk], quad | pk);
            if (i > k) {
                const T f = aik * prec[k & 1];
                if (part == 0) Ls[k][i] = aik;
#pragma unroll
                for (int q = 0; q < CPT; ++q) E[q] = fma(-f, prow[k & 1][part][q], E[q]);
                if (part == pk) E[qk] = -f;
            } else if (i == k && part == pk) {
                E[qk] = T(1);  // row k is finished: its entry k of the unit triangular inverse
            }
            if (k + 1 < B) publish(k + 1, pk < 3 ? E[qk] : E[qk + 1 < CPT ? qk + 1 : qk]);
            __syncthreads();
            // row k enters the following steps with a 1 in column k; the others read it here
        }
    if (tid == 0 && bad >= 0) report_error(status, ELSI_ERR_NOT_PD, pivot_base + bad);
    // L and the inverse; Ls holds a_ik, scaled by 1 / sqrt(d_k)
    T *rs = &prow[0][0][0];
    if (tid < B) rs[tid] = T(1) / dsqrt(piv[tid]);
    __syncthreads();
    const T ri = rs[i];
#pragma unroll
    for (int q = 0; q < CPT; ++q) {
        const int c = 4 * q + part;
        if (i < jb && c < jb) inv[(size_t)i + (size_t)c * ldi] = c <= i ? ri * E[q] : T(0);
    }
    for (int e = tid; e < jb * jb; e += 4 * B) {
        const int r = e % jb, c = e / jb;
        a[(size_t)r + (size_t)c * lda] = r > c ? Ls[c][r] * rs[c] : (r == c ? dsqrt(piv[c]) : T(0));
    }
}

template <typename T>
__global__ void zero_upper_kernel(int n, T *a, int lda)
{
    size_t total = (size_t)n * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        int i = (int)(e % n), j = (int)(e / n);
        if (i < j) a[(size_t)i + (size_t)j * lda] = T(0);
    }
}

template <typename T>
static cudaError_t launch_potrf_diag(cudaStream_t st, int jb, T *a, int lda, T *inv, int ldi,
                                     int *status, int base)
{
    EGB_COUNT_LAUNCH();
    potrf_diag_kernel<T><<<1, 4 * kTriBlock, 0, st>>>(jb, a, lda, inv, ldi, status, base);
    return cudaGetLastError();
}

// Left-looking over panels of kTriPanel columns: the panel's diagonal block is factored by
// kTriBlock blocks (updates inside the block), the rows below it are solved against the
// panel's L (right triangular solve by blocks), and the trailing matrix gets one rank-
// kTriPanel update per panel.
template <typename T>
cudaError_t potrf(cudaStream_t st, int n, T *a, int lda, T *inv_diag, int *status)
{
    const int nb = kTriBlock, np = kTriPanel;
    cudaError_t e;
    for (int p0 = 0; p0 < n; p0 += np) {
        const int p1 = (n - p0 < np) ? n : p0 + np;
        // (1) diagonal block [p0, p1)
        for (int j0 = p0; j0 < p1; j0 += nb) {
            const int jb = (p1 - j0 < nb) ? p1 - j0 : nb;
            T *a11 = a + j0 + (size_t)j0 * lda;
            T *inv11 = inv_diag + j0;  // ld = n
            if ((e = launch_potrf_diag<T>(st, jb, a11, lda, inv11, n, status, j0)) != cudaSuccess) return e;
            const int m2 = p1 - j0 - jb;
            if (m2 > 0) {
                T *a21 = a + (j0 + jb) + (size_t)j0 * lda;
                T *a22 = a + (j0 + jb) + (size_t)(j0 + jb) * lda;
                if ((e = tri_apply<T>(st, 1, 0, jb, m2, inv11, n, a21, lda)) != cudaSuccess) return e;
                if ((e = gemm<T>(st, 0, 1, m2, m2, jb, T(-1), a21, lda, a21, lda, T(1), a22, lda, 1)) != cudaSuccess) return e;
            }
        }
        const int m2 = n - p1;
        if (m2 <= 0) continue;
        // (2) rows below: X L_pp^T = A21, block column by block column
        T *a21 = a + p1 + (size_t)p0 * lda;
        for (int j0 = p0; j0 < p1; j0 += nb) {
            const int jb = (p1 - j0 < nb) ? p1 - j0 : nb;
            T *xj = a + p1 + (size_t)j0 * lda;
            if (j0 > p0) {
                // A21_j -= X_{p0..j0} L_{j, p0..j0}^T
                if ((e = gemm<T>(st, 0, 1, m2, jb, j0 - p0, T(-1), a21, lda, a + j0 + (size_t)p0 * lda, lda,
                                 T(1), xj, lda)) != cudaSuccess) return e;
            }
            if ((e = tri_apply<T>(st, 1, 0, jb, m2, inv_diag + j0, n, xj, lda)) != cudaSuccess) return e;
        }
        // (3) A22 -= L21 L21^T (lower triangle), K = panel width
        T *a22 = a + p1 + (size_t)p1 * lda;
        if ((e = gemm<T>(st, 0, 1, m2, m2, p1 - p0, T(-1), a21, lda, a21, lda, T(1), a22, lda, 1)) != cudaSuccess) return e;
    }
    size_t total = (size_t)n * n;
    int grid = (int)((total + 255) / 256);
    if (grid > 152 * 16) grid = 152 * 16;
    EGB_COUNT_LAUNCH();
    zero_upper_kernel<T><<<grid, 256, 0, st>>>(n, a, lda);
    return cudaGetLastError();
}

// Rows [r0, r1) of the triangular solve in two parts: the first part to be solved, its product with
// the rest of L taken from the other part (K = its rows), the other part; blocks of kTriBlock rows
// are multiplied by their inverses. From n = 4096 the parts are halves (a power of two blocks): every row
// of B is read and written once per level, log2(n / 64) times in all, and most of the operations are
// in products with a long K. Below, the first part is a panel of 256 rows, then a block: more rows of
// the products in flight at a time. Standard form and back-substitution by halves against panels:
// n = 16384 61 and 30 ms against 82 and 40, n = 5000 (binary64) 33.7 and 4.8 against 37.9 and 4.6,
// n = 4096 4.0 and 1.9 against 4.3 and 2.1; n = 2000 1.55 and 0.82 against 1.38 and 0.75. In between, binary32
// n = 2800 2.52 and 1.23 against 2.46 and 1.20, 3500 3.41 and 1.60 against 3.36 and 1.61, 3800 3.74 and 1.80
// against 3.96 and 1.91; binary64 n = 2000 4.83 and 1.09 against 5.08 and 1.13, 3200 11.5 and 2.2 against 12.7
// and 2.1, 4095 19.1 and 3.1 against 22.4 and 3.1 (there halves would pay from 2000 on: 1 % of a solve).
template <typename T>
static cudaError_t trsm_range(cudaStream_t st, int trans, bool halves, int r0, int r1, int ncol, const T *L,
                              int ldl, const T *inv_diag, int ldi, T *B, int ldb, const T *ka, const T *kb)
{
    const int nb = kTriBlock, rows = r1 - r0;
    if (rows <= nb) return tri_apply<T>(st, 0, trans, rows, ncol, inv_diag + r0, ldi, B + r0, ldb);
    int mid;
    if (halves) {
        int half = nb;
        while (2 * half < rows) half *= 2;
        mid = r0 + half;
    } else {
        const int step = rows > kTriPanel ? kTriPanel : nb;
        mid = trans ? r0 + (rows - 1) / step * step : r0 + step;
    }
    const T *l21 = L + mid + (size_t)r0 * ldl;  // rows [mid, r1), columns [r0, mid)
    cudaError_t e;
    if (!trans) {
        if ((e = trsm_range<T>(st, trans, halves, r0, mid, ncol, L, ldl, inv_diag, ldi, B, ldb, ka, kb)) != cudaSuccess) return e;
        if ((e = gemm<T>(st, 0, 0, r1 - mid, ncol, mid - r0, T(-1), l21, ldl, B + r0, ldb, T(1), B + mid, ldb)) != cudaSuccess) return e;
        return trsm_range<T>(st, trans, halves, mid, r1, ncol, L, ldl, inv_diag, ldi, B, ldb, ka, kb);
    }
    if ((e = trsm_range<T>(st, trans, halves, mid, r1, ncol, L, ldl, inv_diag, ldi, B, ldb, ka, kb)) != cudaSuccess) return e;
    if ((e = gemm<T>(st, 1, 0, mid - r0, ncol, r1 - mid, T(-1), l21, ldl, B + mid, ldb, T(1), B + r0, ldb, 0,
                     ka ? ka + mid : nullptr, kb ? kb + mid : nullptr)) != cudaSuccess) return e;
    return trsm_range<T>(st, trans, halves, r0, mid, ncol, L, ldl, inv_diag, ldi, B, ldb, ka, kb);
}

template <typename T>
cudaError_t trsm_left_lower(cudaStream_t st, int trans, int n, int ncol, const T *L, int ldl,
                            const T *inv_diag, T *B, int ldb, T *scales)
{
    if (n <= 0 || ncol <= 0) return cudaSuccess;
    const T *ka = nullptr, *kb = nullptr;
    if constexpr (sizeof(T) == 8) {
        if (trans) {
            cudaError_t e = row_scales(st, n, ncol, L, ldl, true, scales, &ka, &kb);
            if (e != cudaSuccess) return e;
        }
    }
    return trsm_range<T>(st, trans, n >= 4096, 0, n, ncol, L, ldl, inv_diag, n, B, ldb, ka, kb);
}

template cudaError_t potrf<double>(cudaStream_t, int, double *, int, double *, int *);
template cudaError_t potrf<float>(cudaStream_t, int, float *, int, float *, int *);
template cudaError_t trsm_left_lower<double>(cudaStream_t, int, int, int, const double *, int,
                                             const double *, double *, int, double *);
template cudaError_t trsm_left_lower<float>(cudaStream_t, int, int, int, const float *, int,
                                            const float *, float *, int, float *);

}  // namespace egb
