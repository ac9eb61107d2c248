// Back-transformation through Q1 (step (5) of the two-stage method, arXiv:1705.11191 sec. 3.1):
// Z <- Q1 Z, Q1 = Q_0 Q_1 ... Q_{P-1} (panels of the full-to-band reduction, each
// Q_p = I - V_p T_p V_p^T), applied from the last to the first. Groups of up to q1_group(n) consecutive
// panels are applied as one compact-WY block I - V T V^T, V = [V_p ... V_q] (explicit, zero above each
// panel's first row), T merged panel by panel as [[T_a, -T_a (V_a^T V_b) T_b], [0, T_b]]: the passes over
// Z fall by the group size and the products have K = group width.
//
// The T of all groups are formed first, in one launch more than panels in a group: the products V_a^T V_b are a few
// small blocks with a long K, which the general products run on a handful of SMs, one group after the
// other; over all groups there are enough of them to fill the chip without dividing K, and they are
// cheap (b = 64: 0.7 % of the work of Q1).
// Measured against merging each group with general products on the way: n = 512 1.01 -> 0.52 ms, n = 1531
// 4.2 -> 1.8, n = 5000 20.5 -> 9.7 (binary64, b = 32); n = 777 0.59 -> 0.30, n = 4096 7.4 -> 2.3, n = 16384
// 114 -> 62 (binary32, b = 64).
#include "common.cuh"
#include "kernels.h"

namespace egb {
namespace q1 {

constexpr int kCols = 8;  // columns of a merged block per CTA

struct Group {
    int plo, np;  // first panel, panels
    __host__ __device__ __forceinline__ Group(int z, int npan, int group)
    {
        const int phi = npan - 1 - z * group;
        plo = phi - group + 1 < 0 ? 0 : phi - group + 1;
        np = phi - plo + 1;
    }
};

// Block (i, j) of the T of group z (tg, ld gw = group b): V_i^T V_j for i < j, T_i for
// i = j, zero for i > j. Binary32 sums are taken over 64 rows at a time, so that an error grows with the
// number of pieces.
template <typename T, int BT, int TM, int TN>
__global__ void __launch_bounds__((BT / TM) * (BT / TN))
gram_kernel(int n, int b, int npan, int group, const T *__restrict__ v1, const T *__restrict__ t1, T *__restrict__ tg)
{
    constexpr int NT = (BT / TM) * (BT / TN), BK = 16, PER = BT * BK / NT, LD = BT + 16 / (int)sizeof(T);
    __shared__ T As[2][BK][LD], Bs[2][BK][LD];
    const Group g(blockIdx.z, npan, group);
    const int pi = blockIdx.y / group, pj = blockIdx.y % group, nt = (b + BT - 1) / BT, gw = group * b;
    if (pi >= g.np || pj >= g.np) return;
    const int m0 = blockIdx.x % nt * BT, n0 = blockIdx.x / nt * BT, tid = threadIdx.x;
    T *out = tg + (size_t)blockIdx.z * gw * gw + pi * b + (size_t)(pj * b) * gw;
    if (pi >= pj) {
        for (int e = tid; e < BT * BT; e += NT) {
            const int i = m0 + e % BT, j = n0 + e / BT;
            if (i < b && j < b) out[i + (size_t)j * gw] = pi > pj ? T(0) : t1[i + (size_t)((g.plo + pi) * b + j) * b];
        }
        return;
    }
    // rows from the first one of the later panel
    const int r0 = (g.plo + pj + 1) * b, k = n - r0;
    const T *A = v1 + r0 + (size_t)(g.plo + pi) * b * n, *B = v1 + r0 + (size_t)(g.plo + pj) * b * n;
    T av[PER], bv[PER];
    auto load = [&](int k0) {
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int e = tid + r * NT, i = e / BK, kk = k0 + e % BK;
            av[r] = m0 + i < b && kk < k ? A[kk + (size_t)(m0 + i) * n] : T(0);
            bv[r] = n0 + i < b && kk < k ? B[kk + (size_t)(n0 + i) * n] : T(0);
        }
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int r = 0; r < PER; ++r) {
            const int e = tid + r * NT;
            As[buf][e % BK][e / BK] = av[r];
            Bs[buf][e % BK][e / BK] = bv[r];
        }
    };
    const int r = tid % (BT / TM) * TM, q = tid / (BT / TM) * TN;
    T acc[TM][TN], sum[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = sum[i][j] = T(0);
    load(0);
    store(0);
    __syncthreads();
    for (int k0 = 0, buf = 0; k0 < k; k0 += BK, buf ^= 1) {
        if (k0 + BK < k) load(k0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk)
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) acc[i][j] = fma(As[buf][kk][r + i], Bs[buf][kk][q + j], acc[i][j]);
        if (sizeof(T) == 4 && (k0 & 48) == 48) {
#pragma unroll
            for (int i = 0; i < TM; ++i)
#pragma unroll
                for (int j = 0; j < TN; ++j) { sum[i][j] += acc[i][j]; acc[i][j] = T(0); }
        }
        if (k0 + BK < k) store(buf ^ 1);
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < TN; ++j)
#pragma unroll
        for (int i = 0; i < TM; ++i)
            if (m0 + r + i < b && n0 + q + j < b)
                out[m0 + r + i + (size_t)(n0 + q + j) * gw] = sizeof(T) == 4 ? sum[i][j] + acc[i][j] : acc[i][j];
}

constexpr int kRows = 32;

// Blocks (i, p), i < p, of every group: G <- -G T_p. kRows rows per CTA.
template <typename T>
__global__ void __launch_bounds__(256) scale_kernel(int b, int npan, int group, T *tg)
{
    __shared__ T row[64][kRows];
    const int p = blockIdx.y + 1, gw = group * b, i0 = blockIdx.x * kRows, tid = threadIdx.x;
    const Group g(blockIdx.z, npan, group);
    if (p >= g.np || i0 >= p * b) return;
    const int rows = min(kRows, p * b - i0);
    T *blk = tg + (size_t)blockIdx.z * gw * gw + (size_t)(p * b) * gw;
    for (int e = tid; e < b * kRows; e += 256)
        row[e / kRows][e % kRows] = e % kRows < rows ? blk[i0 + e % kRows + (size_t)(e / kRows) * gw] : T(0);
    __syncthreads();
    for (int e = tid; e < b * kRows; e += 256) {
        const int i = e % kRows, c = e / kRows;
        const T *tp = blk + p * b + (size_t)c * gw;  // column c of T_p, upper triangular
        T s = T(0);
#pragma unroll 4
        for (int k = 0; k <= c; ++k) s = fma(row[k][i], tp[k], s);
        if (i < rows) blk[i0 + i + (size_t)c * gw] = -s;
    }
}

// Block column p of every group, after the ones before it: X <- T_a X, T_a the upper triangle merged
// so far. kCols columns per CTA.
template <typename T>
__global__ void __launch_bounds__(256) merge_kernel(int p, int b, int npan, int group, T *tg)
{
    __shared__ T x[kCols][(kQ1MaxGroup - 1) * 64];
    const Group g(blockIdx.y, npan, group);
    if (p >= g.np) return;
    const int gw = group * b, wa = p * b, tid = threadIdx.x;
    T *t = tg + (size_t)blockIdx.y * gw * gw, *blk = t + (size_t)(wa + blockIdx.x * kCols) * gw;
    for (int e = tid; e < wa * kCols; e += 256) x[e / wa][e % wa] = blk[e % wa + (size_t)(e / wa) * gw];
    __syncthreads();
    for (int e = tid; e < wa * kCols; e += 256) {
        const int i = e % wa, c = e / wa;
        T s0 = T(0), s1 = T(0);
        int k = i;
#pragma unroll 2
        for (; k + 1 < wa; k += 2) {
            s0 = fma(t[i + (size_t)k * gw], x[c][k], s0);
            s1 = fma(t[i + (size_t)(k + 1) * gw], x[c][k + 1], s1);
        }
        if (k < wa) s0 = fma(t[i + (size_t)k * gw], x[c][k], s0);
        blk[i + (size_t)c * gw] = s0 + s1;
    }
}

}  // namespace q1

template <typename T>
cudaError_t apply_q1(cudaStream_t st, int n, int b, int k, const T *v1, const T *t1, T *z, int ldz, T *work)
{
    using namespace q1;
    int npan = 0;
    for (int c0 = 0; c0 + b <= n - 2; c0 += b) ++npan;
    if (npan == 0) return cudaSuccess;
    const int group = q1_group(n), gw_max = group * b, ngroups = ceil_div(npan, group);
    T *tg = work;                                        // gw_max x gw_max of every group
    T *Y = tg + (size_t)ngroups * gw_max * gw_max;       // gw_max x k
    T *Y2 = Y + (size_t)gw_max * k;                      // gw_max x k
    T *part = Y2 + (size_t)gw_max * k;                   // split-K partials (what is left)
    const size_t part_elems = (size_t)2 * gw_max * k;
    constexpr int BT = sizeof(T) == 8 ? 16 : 32, TM = sizeof(T) == 8 ? 2 : 4, TN = sizeof(T) == 8 ? 1 : 4;
    const int nt = ceil_div(b, BT);
    EGB_COUNT_LAUNCH();
    gram_kernel<T, BT, TM, TN><<<dim3(nt * nt, group * group, ngroups), (BT / TM) * (BT / TN), 0, st>>>(
        n, b, npan, group, v1, t1, tg);
    if (npan > 1) {
        EGB_COUNT_LAUNCH();
        scale_kernel<T><<<dim3(ceil_div((group - 1) * b, kRows), group - 1, ngroups), 256, 0, st>>>(b, npan, group, tg);
    }
    for (int p = 1; p < group && p < npan; ++p) {
        EGB_COUNT_LAUNCH();
        merge_kernel<T><<<dim3(b / kCols, ngroups), 256, 0, st>>>(p, b, npan, group, tg);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    for (int gi = 0; gi < ngroups; ++gi) {
        const Group g(gi, npan, group);
        const int c0 = g.plo * b, r0 = c0 + b, m = n - r0, gw = g.np * b;
        const T *V = v1 + r0 + (size_t)c0 * n;  // m x gw
        const T *Tg = tg + (size_t)gi * gw_max * gw_max;
        T *Zr = z + r0;
        if ((e = gemm_splitk<T>(st, 1, 0, gw, k, m, T(1), V, n, Zr, ldz, Y, gw, part, part_elems)) != cudaSuccess) return e;
        if ((e = gemm<T>(st, 0, 0, gw, k, gw, T(1), Tg, gw_max, Y, gw, T(0), Y2, gw)) != cudaSuccess) return e;
        if ((e = gemm<T>(st, 0, 0, m, k, gw, T(-1), V, n, Y2, gw, T(1), Zr, ldz)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template cudaError_t apply_q1<double>(cudaStream_t, int, int, int, const double *, const double *,
                                      double *, int, double *);
template cudaError_t apply_q1<float>(cudaStream_t, int, int, int, const float *, const float *,
                                     float *, int, float *);

}  // namespace egb
