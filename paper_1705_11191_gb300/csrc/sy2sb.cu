// Full -> band reduction B = Q1^T H~ Q1 (arXiv:1705.11191 Eq. 11, first line; step (1)
// of the two-stage tridiagonalisation in sec. 3.1).
//
// Panel p (columns [p*b, p*b+b), rows [p*b+b, n)) is factorised by blocked Householder
// QR (compact-WY form Q_p = I - V T V^T); then the trailing symmetric matrix gets the
// two-sided update A22 <- Q_p^T A22 Q_p = A22 - V W^T - W V^T with
// X = A22 V T and W = X - (1/2) V (T^T (V^T X)).
//
// The panel QR is one cooperative launch (panel.cu); the trailing update is GEMM work.
#include "common.cuh"
#include "kernels.h"

namespace egb {

// ---- W of the two-sided update, fused (three small launches instead of five GEMMs):
//   X = (A22 V) T,  Y = V^T X,  W = X - (1/2) V (T^T Y).
// Row blocks of WRows<T> rows; tiles of 64 columns (bw <= 64, zero padded) in shared memory,
// each of the 256 threads computing R x CJ or CJ x CJ elements of a tile product (CJ = 4, or 2 for
// bw <= 32, where half of every tile is padding). Binary64 has
// two FMAs a clock and SM, so its blocks are 16 rows: four times the CTAs of 64-row blocks
// (two launches of 135 us at any order), and V (T^T Y) is formed as (V T^T) Y, whose work
// shrinks with the rows, where T^T Y costs every block 64^3 FMAs: 27 and 20 us at n = 1531,
// b = 32, and 11 and 13 us with CJ = 2. (From 8176 rows on, more than 512 blocks, five general
// products in their place take as long: full to band of n = 9000 317 and 318 ms, n = 16384 1591 and 1589.)
template <typename T> constexpr int WRows = sizeof(T) == 4 ? kWRows32 : kWRows64;
constexpr int kWLd = 65;

// c[R][CJ] = sum_{k < kmax} A[R ty + i][k] B[k][CJ tx + j] for tiles A, B with leading dimension
// kWLd, ty = tid / 16, tx = tid % 16
template <typename T, int R, int CJ>
__device__ __forceinline__ void tile_mm(const T *A, const T *B, int kmax, T (&c)[R][CJ])
{
    const int tr = (threadIdx.x >> 4) * R, tc = (threadIdx.x & 15) * CJ;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < CJ; ++j) c[i][j] = T(0);
    for (int k = 0; k < kmax; ++k) {
        T a[R], b[CJ];
#pragma unroll
        for (int i = 0; i < R; ++i) a[i] = A[(tr + i) * kWLd + k];
#pragma unroll
        for (int j = 0; j < CJ; ++j) b[j] = B[k * kWLd + tc + j];
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
            for (int j = 0; j < CJ; ++j) c[i][j] = fma(a[i], b[j], c[i][j]);
    }
}

// A ROWS x 64 tile from global memory, element (i, c) = ld(i, c) stored by st(i, c, value); all
// loads of a thread (256 threads) in flight before the first store.
template <typename T, int ROWS, typename Ld, typename St>
__device__ __forceinline__ void tile_in(Ld ld, St st)
{
    constexpr int U = ROWS * 64 / 256;
    T v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int e = threadIdx.x + 256 * u;
        v[u] = ld(e % ROWS, e / ROWS);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int e = threadIdx.x + 256 * u;
        st(e % ROWS, e / ROWS, v[u]);
    }
}

// tile[i][c] = src[(r0 + i) + c * ld] for i < rows, c < bw; zero elsewhere
template <typename T, int ROWS>
__device__ __forceinline__ void load_rows(T *tile, const T *src, int ld, int r0, int rows, int bw)
{
    tile_in<T, ROWS>([&](int i, int c) { return (i < rows && c < bw) ? src[(size_t)(r0 + i) + (size_t)c * ld] : T(0); },
                     [&](int i, int c, T x) { tile[i * kWLd + c] = x; });
}

// X rows = Xa rows T; partial Y (64 x 64 per block, column-major) = V rows^T X rows. *wexp = 0 for
// w_stage3 (binary64: what the two-sided digit product scales W by).
template <typename T, int CJ>
__global__ void __launch_bounds__(256) w_stage1_kernel(int m, int bw, const T *xa, const T *V, int ldv,
                                                       const T *Tm, int ldt, T *X, T *ypart, int *wexp)
{
    if (sizeof(T) == 8 && blockIdx.x == 0 && threadIdx.x == 0) *wexp = 0;
    constexpr int ROWS = WRows<T>, R = ROWS / 16;
    extern __shared__ unsigned char wsm_raw[];
    T *sT = reinterpret_cast<T *>(wsm_raw), *sA = sT + 64 * kWLd, *sX = sA + 64 * kWLd;
    const int r0 = blockIdx.x * ROWS, rows = min(ROWS, m - r0);
    load_rows<T, 64>(sT, Tm, ldt, 0, bw, bw);
    load_rows<T, ROWS>(sA, xa, m, r0, rows, bw);
    __syncthreads();
    T c[R][CJ];
    tile_mm<T, R, CJ>(sA, sT, bw, c);
    const int tr = (threadIdx.x >> 4) * R, tc = (threadIdx.x & 15) * CJ;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < CJ; ++j) {
            sX[(tr + i) * kWLd + tc + j] = c[i][j];
            if (tr + i < rows && tc + j < bw) X[(size_t)(r0 + tr + i) + (size_t)(tc + j) * m] = c[i][j];
        }
    __syncthreads();
    // V rows transposed into sA: sA[a][i] = V[r0 + i][a]
    tile_in<T, ROWS>([&](int i, int a) { return (i < rows && a < bw) ? V[(size_t)(r0 + i) + (size_t)a * ldv] : T(0); },
                     [&](int i, int a, T x) { sA[a * kWLd + i] = x; });
    __syncthreads();
    T y[CJ][CJ];
    tile_mm<T, CJ, CJ>(sA, sX, ROWS, y);
    const int ta = (threadIdx.x >> 4) * CJ;
    T *yp = ypart + (size_t)blockIdx.x * 64 * 64;
    if (ta < bw && tc < bw)
#pragma unroll
        for (int i = 0; i < CJ; ++i)
#pragma unroll
            for (int j = 0; j < CJ; ++j) yp[(ta + i) + (tc + j) * 64] = y[i][j];
}

// Y[e] = sum over blocks g of ypart[g][e] (e < 64 * 64): four threads an element, each over a
// quarter of the blocks in ascending order
template <typename T>
__global__ void __launch_bounds__(256) w_stage2_kernel(int nblk, int bw, const T *ypart, T *Y)
{
    __shared__ T part[4][64];
    const int el = threadIdx.x & 63, q = threadIdx.x >> 6, e = blockIdx.x * 64 + el;
    T s = T(0);
    if (el < bw && (int)blockIdx.x < bw) {
        const int per = (nblk + 3) / 4, g1 = min(nblk, (q + 1) * per);
        int g = q * per;
        for (; g + 8 <= g1; g += 8) {
            T v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = ypart[(size_t)(g + u) * 64 * 64 + e];
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        for (; g < g1; ++g) s += ypart[(size_t)g * 64 * 64 + e];
    }
    part[q][el] = s;
    __syncthreads();
    if (q == 0) Y[e] = (part[0][el] + part[1][el]) + (part[2][el] + part[3][el]);
}

// The exponent field of the largest value of a CTA (256 threads), into *wexp; one atomic a CTA, since
// those of a launch all go to one address
__device__ __forceinline__ void block_exponent(int top, int *wexp)
{
    __shared__ int tops[8];
    top = __reduce_max_sync(0xffffffffu, top & 0x7FF00000);
    if ((threadIdx.x & 31) == 0) tops[threadIdx.x >> 5] = top;
    __syncthreads();
    if (threadIdx.x < 32) {
        top = __reduce_max_sync(0xffffffffu, tops[threadIdx.x & 7]);
        if (threadIdx.x == 0) atomicMax(wexp, top >> 20);
    }
}

// W rows = X rows - (1/2) (V rows T^T) Y
template <typename T, int CJ>
__global__ void __launch_bounds__(256) w_stage3_kernel(int m, int bw, const T *X, const T *V, int ldv,
                                                       const T *Tm, int ldt, const T *Y, T *W, int *wexp)
{
    constexpr int ROWS = WRows<T>, R = ROWS / 16;
    extern __shared__ unsigned char wsm_raw[];
    T *sA = reinterpret_cast<T *>(wsm_raw), *sB = sA + 64 * kWLd, *sZ = sB + 64 * kWLd;
    const int r0 = blockIdx.x * ROWS, rows = min(ROWS, m - r0);
    // sA = T^T (sA[a][k] = T[k][a]), sB = Y, sZ = V rows
    tile_in<T, 64>([&](int i, int c) { return (i < bw && c < bw) ? Tm[(size_t)i + (size_t)c * ldt] : T(0); },
                   [&](int i, int c, T x) { sA[c * kWLd + i] = x; });
    tile_in<T, 64>([&](int i, int c) { return Y[i + c * 64]; }, [&](int i, int c, T x) { sB[i * kWLd + c] = x; });
    load_rows<T, ROWS>(sZ, V, ldv, r0, rows, bw);
    __syncthreads();
    T c[R][CJ];
    tile_mm<T, R, CJ>(sZ, sA, bw, c);
    const int tr = (threadIdx.x >> 4) * R, tc = (threadIdx.x & 15) * CJ;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < CJ; ++j) sZ[(tr + i) * kWLd + tc + j] = c[i][j];
    __syncthreads();
    tile_mm<T, R, CJ>(sZ, sB, bw, c);
    int top = 0;
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < CJ; ++j)
            if (tr + i < rows && tc + j < bw) {
                const size_t q = (size_t)(r0 + tr + i) + (size_t)(tc + j) * m;
                const T v = X[q] - T(0.5) * c[i][j];
                W[q] = v;
                if (sizeof(T) == 8) top = max(top, __double2hiint((double)v) & 0x7FF00000);
            }
    if (sizeof(T) == 8) block_exponent(top, wexp);
}

template <typename T, int CJ>
static cudaError_t form_w(cudaStream_t st, int m, int bw, const T *xa, const T *V, int ldv,
                          const T *Tm, int ldt, T *X, T *Y, T *W, T *ypart, int *wexp)
{
    const int nblk = ceil_div(m, WRows<T>);
    const size_t smem = (size_t)3 * 64 * kWLd * sizeof(T);
    static PerDeviceOnce attr;  // per instantiation
    cudaError_t e = once_per_device(attr, [&] {
        cudaError_t r = cudaFuncSetAttribute(w_stage1_kernel<T, CJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(w_stage3_kernel<T, CJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return r;
    });
    if (e != cudaSuccess) return e;
    EGB_COUNT_LAUNCH();
    w_stage1_kernel<T, CJ><<<nblk, 256, smem, st>>>(m, bw, xa, V, ldv, Tm, ldt, X, ypart, wexp);
    EGB_COUNT_LAUNCH();
    w_stage2_kernel<T><<<64, 256, 0, st>>>(nblk, bw, ypart, Y);
    EGB_COUNT_LAUNCH();
    w_stage3_kernel<T, CJ><<<nblk, 256, smem, st>>>(m, bw, X, V, ldv, Tm, ldt, Y, W, wexp);
    return cudaGetLastError();
}

size_t sy2sb_work_elems(int n, int b)
{
    // X (n x b), W (n x b), scratch of the panel (2 b x b)
    return (size_t)4 * n * b + 4 * (size_t)b * b;
}

template <typename T>
cudaError_t sy2sb(cudaStream_t st, int n, int b, T *a, int lda, T *v1, T *t1, T *work,
                  size_t work_elems, unsigned *sync, int *status, int num_sms)
{
    cudaError_t e;
    if (b > 64 || b < 1) return cudaErrorInvalidValue;
    // sync layout: partials of the W kernels, then the packets of the panel factorisation
    T *ypart = reinterpret_cast<T *>(sync + 64);
    unsigned long long *packets = reinterpret_cast<unsigned long long *>(sync + sync_base_words(n, sizeof(T)));
    const int m_first = n - b;
    if (m_first >= 2 &&
        (e = cudaMemsetAsync(packets, 0, sizeof(unsigned long long) * panel_packet_words(m_first, sizeof(T)), st)) != cudaSuccess)
        return e;
    // V1 explicit and zero outside each panel's reflectors (the back-transformation merges
    // consecutive panels into one block)
    if ((e = cudaMemsetAsync(v1, 0, sizeof(T) * (size_t)n * n, st)) != cudaSuccess) return e;
    for (int c0 = 0; c0 + b <= n - 2; c0 += b) {
        const int r0 = c0 + b;
        const int m = n - r0;
        const int bw = b;
        T *P = a + r0 + (size_t)c0 * lda;
        T *V = v1 + r0 + (size_t)c0 * n;
        T *Tm = t1 + (size_t)c0 * b;
        int ldt = b;
        T *Y = work + (size_t)2 * n * b;  // 2 b x b, for panel_qr
        if ((e = panel_qr<T>(st, m, m_first, bw, P, lda, V, n, Tm, ldt, (unsigned)c0, packets, Y, status, num_sms)) != cudaSuccess)
            return e;

        // ---- two-sided update of A22 = a[r0:, r0:] (full symmetric storage)
        T *A22 = a + r0 + (size_t)r0 * lda;
        T *X = work;                      // m x b
        T *W = work + (size_t)n * b;      // m x b
        // X = A22 V (binary32: the symmetric panel product that streams A22 once)
        bool xdone = false;
        if constexpr (sizeof(T) == 4) {
            float *tw;
            size_t te;
            int *ts;
            if (tc_scratch(&tw, &te, &ts)) {
                e = symm_tall_f32(st, m, bw, (const float *)A22, lda, (const float *)V, n, (float *)W, m,
                                  tw, te, ts);
                if (e != cudaErrorNotSupported) {
                    if (e != cudaSuccess) return e;
                    xdone = true;
                }
            }
        }
        // (A22 is symmetric: transposed, its rows are contiguous for the digit split)
        if (!xdone && (e = gemm<T>(st, 1, 0, m, bw, m, T(1), A22, lda, V, n, T(0), W, m)) != cudaSuccess)
            return e;
        // X = (A22 V) T, W = X - 1/2 V (T^T (V^T X))
        T *ysum = ypart + (size_t)ceil_div(m, WRows<T>) * 64 * 64;
        e = bw <= 32 ? form_w<T, 2>(st, m, bw, W, V, n, Tm, ldt, X, ysum, W, ypart, status + ST_WEXP)
                     : form_w<T, 4>(st, m, bw, W, V, n, Tm, ldt, X, ysum, W, ypart, status + ST_WEXP);
        if (e != cudaSuccess) return e;
        // A22 -= V W^T + W V^T   (lower triangle), then mirror. On the tensor-core path the
        // two products are one GEMM over K = 2 bw: [V W] [W V]^T.
        bool done = false;
        if constexpr (sizeof(T) == 4) {
            float *tw;
            size_t te;
            int *ts;
            if (tc_scratch(&tw, &te, &ts)) {
                TcPart pa[2] = {{(const float *)V, n, 0, bw}, {(const float *)W, m, 0, bw}};
                TcPart pb[2] = {{(const float *)W, m, 1, bw}, {(const float *)V, n, 1, bw}};
                e = tc_gemm_f32_parts(st, m, m, 2, pa, pb, -1.0f, 1.0f, (float *)A22, lda, 1, tw, te, ts);
                if (e != cudaErrorNotSupported) {
                    if (e != cudaSuccess) return e;
                    done = true;
                }
            }
        }
        if constexpr (sizeof(T) == 8) {
            e = gemm_f64_two_sided(st, m, bw, V, n, W, m, A22, lda, status + ST_WEXP);
            if (e != cudaErrorNotSupported) {
                if (e != cudaSuccess) return e;
                done = true;
            }
        }
        if (!done) {
            if ((e = gemm<T>(st, 0, 1, m, m, bw, T(-1), V, n, W, m, T(1), A22, lda, 1)) != cudaSuccess) return e;
            if ((e = gemm<T>(st, 0, 1, m, m, bw, T(-1), W, m, V, n, T(1), A22, lda, 1)) != cudaSuccess) return e;
        }
        if ((e = mirror_lower<T>(st, m, A22, lda)) != cudaSuccess) return e;
    }
    (void)work_elems;
    return cudaSuccess;
}

template cudaError_t sy2sb<double>(cudaStream_t, int, int, double *, int, double *, double *,
                                   double *, size_t, unsigned *, int *, int);
template cudaError_t sy2sb<float>(cudaStream_t, int, int, float *, int, float *, float *,
                                  float *, size_t, unsigned *, int *, int);

}  // namespace egb
