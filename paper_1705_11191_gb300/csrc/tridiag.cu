// Symmetric tridiagonal eigensolver (step (3) of the two-stage method, arXiv:1705.11191
// sec. 3.1), restricted to the wanted eigenpairs as the paper describes for KS-DFT.
//
//  * eigenvalues: Sturm-sequence bisection (Givens 1954; Barth, Martin & Wilkinson
//    1967), a few threads per wanted eigenvalue index (multisection);
//  * eigenvectors: one twisted factorisation T - lambda I = N_r D_r N_r^T per
//    eigenvalue (Parlett & Dhillon 1997/2000), which gives the vector with residual
//    O(eps ||T||) in O(n) work;
//  * vectors of eigenvalues closer than 1e-5 ||T|| are re-orthogonalised (two passes of
//    Gram-Schmidt within the cluster, as in inverse-iteration codes), which bounds the
//    loss of orthogonality between close vectors by about eps*1e5. A cluster is worked
//    on in pieces of 64 consecutive vectors and then in the 64-vector seams across piece
//    boundaries, so that a long chain of close eigenvalues (an ill-conditioned overlap
//    puts one huge eigenvalue into ||T|| and with it every gap of the rest of the
//    spectrum below the threshold) costs O(64 n) per vector instead of O(cluster n):
//    vectors more than 32 places apart are left as the twisted factorisation gives them,
//    orthogonal to about eps ||T|| / (32 times the eigenvalue spacing).
// All of this runs in binary64 regardless of the precision of the reduction.
#include <float.h>

#include "common.cuh"
#include "kernels.h"
#include "packets.cuh"

namespace egb {

__device__ __forceinline__ double guard_pivot(double q, double pivmin)
{
    return (fabs(q) < pivmin) ? -pivmin : q;
}

// p and pm times the power of two that brings |p| to [1, 2), or |pm| to 2^500 if it would pass that.
__device__ __forceinline__ void sturm_rescale(double &p, double &pm)
{
    const int ep = (__double2hiint(p) >> 20) & 0x7FF, em = (__double2hiint(pm) >> 20) & 0x7FF;
    const int f = max(min(2046 - max(ep, 1), 2546 - em), 1);
    const double s = __hiloint2double(f << 20, 0);
    p *= s;
    pm *= s;
}

// number of eigenvalues < sigma: the sign changes of the leading principal minors
// p_i = det(T[0:i, 0:i] - sigma I), p_0 = 1, p_{i+1} = (d_i - sigma) p_i - e_{i-1}^2 p_{i-1}
// (Sturm; Givens 1954), e2 = e^2. The ratio q_i = p_{i+1} / p_i is the pivot of the LDL^T
// factorisation of T - sigma I, and a pivot smaller than pivmin in magnitude is replaced
// by -pivmin as in the pivot form. This form needs no division, and everything but the three
// operations of the recurrence is done on the bit patterns: on this chip a warp holds its
// scheduler's binary64 unit for 64 cycles with every addition, product or comparison. Signs
// come from the sign bits; the test for a tiny pivot is made when the exponent of p_{i+1} is
// below that of pivmin 2^460 >= pivmin |p_i| (it always is for a zero; a pivot that this test lets
// through has the sign of its computed value, which is as good). The pair (p_i, p_{i-1}) is
// multiplied by the power of two that puts |p_i| next to 1 (sturm_rescale) when one of the two has
// left [2^-200, 2^200] at the end of eight steps, so that every piece starts there whatever
// ||T|| is: a fixed factor of 2^200 a piece loses to steps of more than 25 bits, and the counts of
// ||T|| below 2^-24 or above 2^26 were wrong. Eight steps of up to 100 bits each stay in range; a
// piece with a value out of range (an infinity or a NaN, or one so small that digits may be lost) is
// done again step by step, rescaled before each.
// A warp issues in order, so eight steps are one straight piece without a branch: the next d and
// e^2 are on their way, the eight d_i - sigma do not wait for the chain, and what has to be done
// again is seen afterwards, from the smallest and the largest exponent.
// Measured against a form with a binary64 product and comparison for the pivot test, sign
// comparisons and e^2 formed on the way (8 such operations a step, eigenvalues by 8 or 2 lanes
// at every count), the bisection: n = 1531, 382 values 8.7 -> 4.1 ms; n = 4096, all 15.2 -> 7.1
// ms; n = 16384, all 111 -> 65 ms; 8 solves of n = 2000 at a time 25 -> 10 ms each; and then
// with the straight pieces 2.2, 4.3, 38 and 7.4 ms.
// e2[i] = e_{i-1}^2, e2[0] = 0.
__device__ int sturm_count(int n, const double *__restrict__ d, const double *__restrict__ e2,
                           double sigma, double pivmin)
{
    constexpr int P = 8;
    const int tiny = (__double2hiint(pivmin) & 0x7FF00000) + (461 << 20);
    double pm = 0.0, p = 1.0;  // p_{i-1}, p_i
    unsigned cnt = 0;
    auto steps = [&](int i0, int i1) {
        for (int i = i0; i < i1; ++i) {
            sturm_rescale(p, pm);
            double pn = fma(d[i] - sigma, p, -e2[i] * pm);
            // pivot q = pn / p below pivmin in magnitude: q = -pivmin
            if (fabs(pn) < pivmin * fabs(p)) pn = -pivmin * p;
            cnt += (unsigned)(__double2hiint(pn) ^ __double2hiint(p)) >> 31;
            pm = p;
            p = pn;
        }
    };
    const int whole = n / P * P;
    double dn[P], en[P];
    if (whole > 0) {
#pragma unroll
        for (int q = 0; q < P; ++q) { dn[q] = d[q]; en[q] = e2[q]; }
    }
    for (int i = 0; i < whole; i += P) {
        double x[P], y[P];
#pragma unroll
        for (int q = 0; q < P; ++q) { x[q] = dn[q] - sigma; y[q] = en[q]; }
        if (i + P < whole) {
#pragma unroll
            for (int q = 0; q < P; ++q) { dn[q] = d[i + P + q]; en[q] = e2[i + P + q]; }
        }
        const double p0 = p, pm0 = pm;
        unsigned c = 0;
        int least = 0x7FF00000, most = 0;
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const double pn = fma(x[q], p, -y[q] * pm);
            least = min(least, __double2hiint(pn) & 0x7FF00000);
            most = max(most, __double2hiint(pn) & 0x7FF00000);
            c += (unsigned)(__double2hiint(pn) ^ __double2hiint(p)) >> 31;
            pm = p;
            p = pn;
        }
        if (least <= tiny || most == 0x7FF00000) {
            p = p0;
            pm = pm0;
            steps(i, i + P);
        } else {
            cnt += c;
        }
        const int ex = __double2hiint(p) & 0x7FF00000, mx = max(ex, __double2hiint(pm) & 0x7FF00000);
        if (mx > ((1023 + 200) << 20) || ex < ((1023 - 200) << 20)) sturm_rescale(p, pm);
    }
    steps(whole, n);
    return (int)cnt;
}

// [0]=gl, [1]=gu, [2]=pivmin, [3]=||T|| bound, [4]=1 if T splits into blocks, else 0
__global__ void gershgorin_kernel(int n, const double *d, const double *e, double *out)
{
    __shared__ double red[32];
    double lo = DBL_MAX, hi = -DBL_MAX, e2max = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double r = 0.0;
        if (i > 0) r += fabs(e[i - 1]);
        if (i + 1 < n) { r += fabs(e[i]); e2max = fmax(e2max, e[i] * e[i]); }
        lo = fmin(lo, d[i] - r);
        hi = fmax(hi, d[i] + r);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        e2max = fmax(e2max, __shfl_xor_sync(0xffffffffu, e2max, o));
    }
    __shared__ double slo[32], shi[32], se[32];
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) { slo[w] = lo; shi[w] = hi; se[w] = e2max; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int q = 1; q < (int)(blockDim.x >> 5); ++q) {
            lo = fmin(lo, slo[q]); hi = fmax(hi, shi[q]); e2max = fmax(e2max, se[q]);
        }
        double tn = fmax(fabs(lo), fabs(hi));
        double pad = 2.0 * DBL_EPSILON * tn * n + DBL_MIN;
        out[0] = lo - pad;
        out[1] = hi + pad;
        out[2] = DBL_MIN * fmax(1.0, e2max);
        out[3] = tn;
        red[0] = tn;
    }
    __syncthreads();
    // [4] = 1 if T splits (an off-diagonal at or below the threshold of split_kernel)
    const double thr = 2.0 * DBL_EPSILON * red[0];
    int split = 0;
    for (int i = threadIdx.x; i < n - 1; i += blockDim.x) split |= (fabs(e[i]) <= thr) ? 1 : 0;
    split = __syncthreads_or(split);
    if (threadIdx.x == 0) out[4] = split ? 1.0 : 0.0;
}

// number of eigenvalues < sigma, binary32 (used only to bracket); d and e^2 rounded once for
// all counts (a conversion is a binary64 operation too)
__device__ int sturm_count32(int n, const float *__restrict__ d, const float *__restrict__ e2,
                             float sigma, float pivmin)
{
    float q = d[0] - sigma;
    if (fabsf(q) < pivmin) q = -pivmin;
    int cnt = q < 0.0f;
    for (int i = 1; i < n; ++i) {
        q = d[i] - sigma - __fdividef(e2[i - 1], q);
        if (fabsf(q) < pivmin) q = -pivmin;
        cnt += q < 0.0f;
    }
    return cnt;
}

// Bisection for eigenvalue index idx = blockIdx.x * (blockDim.x / LANES) + group, with
// LANES threads per eigenvalue evaluating LANES interior points of the current interval
// (multisection: the interval shrinks by LANES + 1 per step).
// Phase 1 (bracket32 != 0): binary32 counts down to a width of 1e-6 ||T|| (a binary32
// Sturm count is exact for a matrix within a few binary32 roundings of T, so its
// eigenvalues move by far less), then the bracket is widened by 2e-6 ||T|| and checked
// with binary64 counts (falling back to the Gershgorin interval if the check fails). Phase 2: binary64 counts down to
// max(tol_rel * ||T||, 2 eps max|lo|,|hi|).
template <int LANES>
__global__ void bisect_kernel(int n, const double *__restrict__ d, const double *__restrict__ e2,
                              const float *__restrict__ d32, const float *__restrict__ e232, int count,
                              const double *bounds, double *w, double tol_rel, int bracket32)
{
    const int group = threadIdx.x / LANES, lane = threadIdx.x % LANES;
    const int idx = blockIdx.x * (blockDim.x / LANES) + group;
    const unsigned gmask = (LANES == 32) ? 0xffffffffu
                                         : (((1u << LANES) - 1u) << ((threadIdx.x & 31) / LANES * LANES));
    const bool active = idx < count;
    const double gl = bounds[0], gu = bounds[1], pivmin = bounds[2], tn = bounds[3];
    double lo = gl, hi = gu;
    if (bracket32 && active) {
        float flo = (float)gl, fhi = (float)gu;
        const float fpiv = fmaxf(1e-30f, (float)pivmin);
        for (int it = 0; it < 64 && (double)(fhi - flo) > 1e-6 * tn; ++it) {
            float sig = flo + (fhi - flo) * (float)(lane + 1) / (float)(LANES + 1);
            int c = sturm_count32(n, d32, e232, sig, fpiv);
            unsigned ok = __ballot_sync(gmask, c <= idx) & gmask;
            int pcount = __popc(ok);
            float nlo = __shfl_sync(gmask, sig, (threadIdx.x & 31) / LANES * LANES + max(pcount - 1, 0));
            float nhi = __shfl_sync(gmask, sig, (threadIdx.x & 31) / LANES * LANES + min(pcount, LANES - 1));
            if (pcount > 0) flo = nlo;
            if (pcount < LANES) fhi = nhi;
        }
        lo = (double)flo - 2e-6 * tn;
        hi = (double)fhi + 2e-6 * tn;
        if (lo < gl) lo = gl;
        if (hi > gu) hi = gu;
        // verify the bracket in binary64: count(lo) <= idx < count(hi)
        int c = sturm_count(n, d, e2, lane == 0 ? lo : hi, pivmin);
        int clo = __shfl_sync(gmask, c, (threadIdx.x & 31) / LANES * LANES);
        int chi = (LANES > 1) ? __shfl_sync(gmask, c, (threadIdx.x & 31) / LANES * LANES + 1)
                              : sturm_count(n, d, e2, hi, pivmin);
        if (!(clo <= idx && idx < chi)) { lo = gl; hi = gu; }
    }
    if (active) {
        for (int it = 0; it < 128; ++it) {
            // tol_rel relative to ||T||, but not looser than 10 tol_rel |lambda| (a single
            // huge eigenvalue of an ill-conditioned overlap must not loosen all others)
            const double scale = fmin(tn, 10.0 * fmax(1.0, fmax(fabs(lo), fabs(hi))));
            double tol = fmax(tol_rel * scale, 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi))) + 4.0 * pivmin;
            if (hi - lo <= tol) break;
            double sig = lo + (hi - lo) * (double)(lane + 1) / (double)(LANES + 1);
            int c = sturm_count(n, d, e2, sig, pivmin);
            unsigned ok = __ballot_sync(gmask, c <= idx) & gmask;
            int pcount = __popc(ok);
            double nlo = __shfl_sync(gmask, sig, (threadIdx.x & 31) / LANES * LANES + max(pcount - 1, 0));
            double nhi = __shfl_sync(gmask, sig, (threadIdx.x & 31) / LANES * LANES + min(pcount, LANES - 1));
            if (pcount > 0) lo = nlo;
            if (pcount < LANES) hi = nhi;
        }
        if (lane == 0) w[idx] = 0.5 * (lo + hi);
    }
}

// Off-diagonals below 2 eps ||T|| are set to zero: T splits into unreduced blocks, which
// changes no eigenvalue by more than 2 eps ||T|| and lets exactly degenerate eigenvalues
// (e.g. those of a complex Hermitian matrix written as a real one) be found in
// different blocks.
// Also the forms of T that the counts read: e^2 (from index 1), and d and e^2 in binary32.
__global__ void split_kernel(int n, const double *d, double *e, const double *bounds, double *e2, float *d32,
                             float *e232)
{
    const double tn = bounds[3];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        d32[i] = (float)d[i];
        if (i < n - 1) {
            double x = e[i];
            if (fabs(x) <= 2.0 * DBL_EPSILON * tn) e[i] = x = 0.0;
            e2[i + 1] = x * x;
            e232[i] = (float)x * (float)x;
        }
        if (i == 0) e2[0] = 0.0;
    }
}

static thread_local int t_concurrent_solves = 1;
void set_concurrent_solves(int solves) { t_concurrent_solves = solves; }

cudaError_t stebz(cudaStream_t st, int n, const double *d, double *e, int count,
                  double *w, int *status, double *scratch, double tol_rel)
{
    (void)status;
    if (n <= 0 || count <= 0) return cudaSuccess;
    // the Gershgorin bounds live right after the count eigenvalues (w has count + 8)
    double *bounds = w + count;
    double *e2 = scratch;
    float *d32 = reinterpret_cast<float *>(scratch + n), *e232 = d32 + n;
    EGB_COUNT_LAUNCH();
    gershgorin_kernel<<<1, 1024, 0, st>>>(n, d, e, bounds);
    EGB_COUNT_LAUNCH();
    split_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, d, e, bounds, e2, d32, e232);
    // Lanes per eigenvalue. A count of L points gains log2(L + 1) bits, so one lane is the best
    // use of a busy binary64 unit and many lanes the shortest chain on idle ones: the most lanes
    // that keep a warp per scheduler (608, divided among the solves that run at the same time).
    // n = 120: 32 lanes; n = 4096 with all eigenvalues: 4; n = 16384: 1.
    const int budget = 608 * 32 / (t_concurrent_solves > 0 ? t_concurrent_solves : 1);
    int lanes = 1;
    while (lanes < 32 && (long long)count * lanes * 2 <= budget) lanes *= 2;
    const int b32 = n > 512;
    const int grid = ceil_div(count, 128 / lanes);
    EGB_COUNT_LAUNCH();
    switch (lanes) {
    case 1: bisect_kernel<1><<<grid, 128, 0, st>>>(n, d, e2, d32, e232, count, bounds, w, tol_rel, b32); break;
    case 2: bisect_kernel<2><<<grid, 128, 0, st>>>(n, d, e2, d32, e232, count, bounds, w, tol_rel, b32); break;
    case 4: bisect_kernel<4><<<grid, 128, 0, st>>>(n, d, e2, d32, e232, count, bounds, w, tol_rel, b32); break;
    case 8: bisect_kernel<8><<<grid, 128, 0, st>>>(n, d, e2, d32, e232, count, bounds, w, tol_rel, b32); break;
    case 16: bisect_kernel<16><<<grid, 128, 0, st>>>(n, d, e2, d32, e232, count, bounds, w, tol_rel, b32); break;
    default: bisect_kernel<32><<<grid, 128, 0, st>>>(n, d, e2, d32, e232, count, bounds, w, tol_rel, b32); break;
    }
    return cudaGetLastError();
}

// The count in the pivot form, from e (rare: only where T splits).
__device__ int sturm_count_e(int n, const double *__restrict__ d, const double *__restrict__ e, double sigma,
                             double pivmin)
{
    double q = guard_pivot(d[0] - sigma, pivmin);
    int cnt = q < 0.0;
    for (int i = 1; i < n; ++i) {
        q = guard_pivot(d[i] - sigma - e[i - 1] * e[i - 1] / q, pivmin);
        cnt += q < 0.0;
    }
    return cnt;
}

// Block of each eigenvalue: with [lo, hi] a small interval around w[l], the eigenvalues of
// T in it are numbered by block order; w[l] is the (l - count(lo))-th of them. blk[2l],
// blk[2l+1] = [start, end) of its block.
__global__ void block_assign_kernel(int n, const double *d, const double *e, int kvec,
                                    const double *w, const double *bounds, int *blk)
{
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= kvec) return;
    if (bounds[4] == 0.0) {  // T is one block
        blk[2 * l] = 0;
        blk[2 * l + 1] = n;
        return;
    }
    const double tn = bounds[3], pivmin = bounds[2];
    const double delta = 8.0 * DBL_EPSILON * fmax(fabs(w[l]), tn) + 4.0 * pivmin;
    const double lo = w[l] - delta, hi = w[l] + delta;
    const int clo = sturm_count_e(n, d, e, lo, pivmin);
    int r = l - clo;  // rank among the eigenvalues in [lo, hi]
    if (r < 0) r = 0;
    double qlo = 1.0, qhi = 1.0;
    int cl = 0, ch = 0, start = 0;
    int bs = 0, be = n;
    for (int i = 0; i < n; ++i) {
        const double ei2 = (i > 0) ? e[i - 1] * e[i - 1] : 0.0;
        if (i == 0 || e[i - 1] == 0.0) {
            qlo = d[i] - lo;
            qhi = d[i] - hi;
        } else {
            qlo = d[i] - lo - ei2 / qlo;
            qhi = d[i] - hi - ei2 / qhi;
        }
        if (fabs(qlo) < pivmin) qlo = -pivmin;
        if (fabs(qhi) < pivmin) qhi = -pivmin;
        cl += qlo < 0.0;
        ch += qhi < 0.0;
        const bool block_end = (i == n - 1) || (e[i] == 0.0);
        if (block_end) {
            if (ch - cl > r) { bs = start; be = i + 1; break; }
            start = i + 1;
        }
    }
    blk[2 * l] = bs;
    blk[2 * l + 1] = be;
}

// |a| < |b| on the bit patterns
__device__ __forceinline__ bool mag_less(double a, double b)
{
    return (__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFll) < (__double_as_longlong(b) & 0x7FFFFFFFFFFFFFFFll);
}

// Twisted factorisation of T_b - lam I on the block [bs, be) of each eigenvalue lam = w[l], in two
// kernels. The first one runs the two recurrences, a thread each: the pivots D+ (dplus) and ratios
// L+ = e / D+ (lplus) of the forward factorisation, the ratios U- = e / D- (uminus) of the
// backward one. Arrays are indexed [i * kvec + l].
//
// What bounds it: the recurrence, seven dependent binary64 operations a row (a reciprocal from the
// hardware's approximation, L+, the pivot), each 64 clocks of a warp's unit; so the two directions go
// to different warps, and everything that is not in the recurrence goes to the second kernel. There
// 32 vectors belong to a CTA of eight warps: the search for the twist index r = argmin |gamma_i|,
// gamma_i = D+_i + D-_i - (d_i - lam), is divided by rows (D- is formed again from U-, the same
// operations); the products z_i = -L+_i z_{i+1} above r and z_{i+1} = -U-_i z_i below it (z_r = 1)
// are two chains for two warps, whose lanes step through the rows together; then all warps scale by
// 1 / ||z|| and transpose through shared memory into whole lines of z.
// Measured against one thread per vector from the forward recurrence to the store of z, with the
// loads of each row waited for: n = 1531, 381 vectors 2.2 -> 0.9 ms; n = 4096, all 9.3 -> 2.8 ms;
// n = 16384, all 47 -> 19 ms.
__global__ void __launch_bounds__(32)
twist_factor_kernel(const double *__restrict__ d, const double *__restrict__ e, int kvec,
                    const double *__restrict__ w, const double *bounds, const int *__restrict__ blk,
                    double *dplus, double *lplus, double *uminus)
{
    const int l = blockIdx.x * 32 + threadIdx.x;
    if (l >= kvec) return;
    const double pivmin = bounds[2], lam = w[l];
    const int bs = blk[2 * l], be = blk[2 * l + 1];  // the eigenvalue's block [bs, be)
    if (blockIdx.y == 0) {
        double dp = guard_pivot(d[bs] - lam, pivmin);
        dplus[(size_t)bs * kvec + l] = dp;
        double en = 0.0, dn = 0.0;  // read one row ahead
        if (bs + 1 < be) { en = e[bs]; dn = d[bs + 1]; }
        for (int i = bs; i < be - 1; ++i) {
            const double ei = en, dl = dn - lam;
            if (i + 2 < be) { en = e[i + 1]; dn = d[i + 2]; }
            const double lp = ei * recip(dp);
            lplus[(size_t)i * kvec + l] = lp;
            dp = fma(-lp, ei, dl);
            if (mag_less(dp, pivmin)) dp = -pivmin;
            dplus[(size_t)(i + 1) * kvec + l] = dp;
        }
    } else {
        double dm = guard_pivot(d[be - 1] - lam, pivmin);
        double en = 0.0, dn = 0.0;
        if (bs + 1 < be) { en = e[be - 2]; dn = d[be - 2]; }
        for (int i = be - 2; i >= bs; --i) {
            const double ei = en, dl = dn - lam;
            if (i > bs) { en = e[i - 1]; dn = d[i - 1]; }
            const double um = ei * recip(dm);
            uminus[(size_t)i * kvec + l] = um;
            dm = fma(-um, ei, dl);
            if (mag_less(dm, pivmin)) dm = -pivmin;
        }
    }
}

constexpr int kTwistWarps = 8, kTwistRows = 16;

// z / ||z|| for each of the first kvec eigenvalues (zero outside its block), from the factors;
// lplus and uminus are overwritten by z. A vector that is lost is zero, and the end of its block negative.
template <typename T>
__global__ void __launch_bounds__(32 * kTwistWarps)
twist_vector_kernel(int n, const double *__restrict__ d, const double *__restrict__ e, int kvec,
                    const double *__restrict__ w, const double *bounds, int *blk,
                    const double *__restrict__ dplus, double *lplus, double *uminus, T *z, int ldz)
{
    __shared__ T tile[kTwistWarps][32][kTwistRows + 1];
    __shared__ double best_w[kTwistWarps][32], nrm_w[2][32];
    __shared__ int r_w[kTwistWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l = blockIdx.x * 32 + lane;
    const bool have = l < kvec;
    const double pivmin = bounds[2], lam = have ? w[l] : 0.0;
    const int bs = have ? blk[2 * l] : 0, be = have ? blk[2 * l + 1] : 0;
    // ---- twist index: the last row of the smallest |gamma|
    double best = __longlong_as_double(0x7FFFFFFFFFFFFFFFll);
    int r = be - 1;
    const int per = (n + kTwistWarps - 1) / kTwistWarps;
    const int lo = min(n, warp * per), hi = min(n, lo + per);
#pragma unroll 4
    for (int i = hi - 1; i >= lo; --i) {
        if (i < bs || i >= be) continue;
        const double dl = d[i] - lam;
        double dm = dl;
        if (i < be - 1) dm = fma(-uminus[(size_t)i * kvec + l], e[i], dl);
        if (mag_less(dm, pivmin)) dm = -pivmin;
        const double g = dplus[(size_t)i * kvec + l] + dm - dl;
        if (mag_less(g, best)) { best = g; r = i; }
    }
    best_w[warp][lane] = best;
    r_w[warp][lane] = r;
    __syncthreads();
    best = best_w[kTwistWarps - 1][lane];
    r = r_w[kTwistWarps - 1][lane];
#pragma unroll
    for (int q = kTwistWarps - 2; q >= 0; --q)
        if (mag_less(best_w[q][lane], best)) { best = best_w[q][lane]; r = r_w[q][lane]; }
    // ---- the two chains of products
    constexpr int P = 8;
    if (warp == 0) {
        const int top = __reduce_max_sync(0xffffffffu, r), bot = __reduce_min_sync(0xffffffffu, have ? bs : n);
        double zi = 1.0, s = 0.0;
        for (int i0 = top - 1; i0 >= bot; i0 -= P) {
            double f[P];
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int i = i0 - q;
                f[q] = i >= bs && i < r ? lplus[(size_t)i * kvec + l] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int i = i0 - q;
                if (i >= bs && i < r) {
                    zi = -f[q] * zi;
                    s = fma(zi, zi, s);
                    lplus[(size_t)i * kvec + l] = zi;
                }
            }
        }
        nrm_w[0][lane] = s;
    } else if (warp == 1) {
        const int first = __reduce_min_sync(0xffffffffu, have ? r : n), last = __reduce_max_sync(0xffffffffu, be);
        double zi = 1.0, s = 0.0;
        for (int i0 = first; i0 < last - 1; i0 += P) {
            double f[P];
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int i = i0 + q;
                f[q] = i >= r && i < be - 1 ? uminus[(size_t)i * kvec + l] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < P; ++q) {
                const int i = i0 + q;
                if (i >= r && i < be - 1) {
                    zi = -f[q] * zi;
                    s = fma(zi, zi, s);
                    uminus[(size_t)i * kvec + l] = zi;
                }
            }
        }
        nrm_w[1][lane] = s;
    }
    __syncthreads();
    const double nrm2 = 1.0 + nrm_w[0][lane] + nrm_w[1][lane];
    // No eigenvector: a product out of range, next to pivots of zero in a group of coinciding eigenvalues,
    // or a residual |gamma| / ||z|| far above the accuracy of the eigenvalue (at most sqrt(n) times
    // 2e-9 ||T||, or 1e-15): a block that does not hold it, where a group is spread over several. The
    // vector is left to cluster_orth_kernel.
    const bool lost = !(nrm2 < DBL_MAX) || !(fabs(best) <= ((sizeof(T) == 8 ? 1e-8 : 1e-4) * bounds[3] + 8.0 * pivmin) * sqrt(nrm2));
    if (warp == 0 && have && lost) blk[2 * l + 1] = -be;
    const double s = lost ? 0.0 : 1.0 / sqrt(nrm2);
    // ---- scaled into the columns of z
    for (int i0 = warp * kTwistRows; i0 < n; i0 += kTwistWarps * kTwistRows) {
#pragma unroll
        for (int q = 0; q < kTwistRows; ++q) {
            const int i = i0 + q;
            double x = 0.0;
            if (i >= bs && i < be)
                x = i < r ? lplus[(size_t)i * kvec + l] : i > r ? uminus[(size_t)(i - 1) * kvec + l] : 1.0;
            tile[warp][lane][q] = lost ? T(0) : (T)(x * s);
        }
        __syncwarp();
        const int q = lane % kTwistRows;
#pragma unroll
        for (int c = lane / kTwistRows; c < 32; c += 32 / kTwistRows)
            if (blockIdx.x * 32 + c < kvec && i0 + q < n)
                z[(size_t)(blockIdx.x * 32 + c) * ldz + i0 + q] = tile[warp][c][q];
        __syncwarp();
    }
}

// Sums and updates of the Gram-Schmidt step with at least the precision of binary64 arithmetic
// rounded to T. A binary32 product and a sum are kept as two binary32 numbers (products split by
// an FMA, Knuth's two-sum: Ogita, Rump & Oishi 2005), a dozen operations of a unit that has 64
// times the rate of the binary64 one; a conversion and an FMA there hold it for 128 clocks. What is
// stored is rounded to binary32 once, so the sums' 48 bits leave what binary64 sums would: of 64
// vectors the largest |z_u . z_v| is 5.2e-9 at n = 500 and 2.8e-9 at n = 2000 with either, against 1.3e-8
// and 7.9e-9 with binary64 sums and a rounded update for every pair.
template <typename T> struct Wide;
template <> struct Wide<double> {
    double v;
    __device__ __forceinline__ explicit Wide(double x = 0.0) : v(x) {}
    __device__ __forceinline__ void fma_(double a, double b) { v = fma(a, b, v); }
    __device__ __forceinline__ void fms(double2 c, double b) { v = fma(-c.x, b, v); }
    __device__ __forceinline__ double rounded() const { return v; }
    __device__ __forceinline__ double value() const { return v; }
    __device__ __forceinline__ static double2 coef(double s) { return make_double2(s, 0.0); }
    using Coef = double2;
};
template <> struct Wide<float> {
    float h, l;
    __device__ __forceinline__ explicit Wide(float x = 0.f) : h(x), l(0.f) {}
    __device__ __forceinline__ void add(float p, float e)
    {
        const float s = h + p, b = s - h;
        l += ((h - (s - b)) + (p - b)) + e;
        h = s;
    }
    __device__ __forceinline__ void fma_(float a, float b)
    {
        const float p = __fmul_rn(a, b);  // not contracted with the sum
        add(p, fmaf(a, b, -p));
    }
    __device__ __forceinline__ void fms(float2 c, float b)  // minus (c.x + c.y) b
    {
        const float p = __fmul_rn(-c.x, b);
        add(p, fmaf(-c.y, b, fmaf(-c.x, b, -p)));
    }
    __device__ __forceinline__ float rounded() const { return h + l; }
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
    __device__ __forceinline__ static float2 coef(double s)
    {
        const float h = (float)s;
        return make_float2(h, (float)(s - (double)h));
    }
    using Coef = float2;
};

// Gram-Schmidt of vector zv against the cluster vectors i0 .. v-1 (two passes, each with all
// products first: Giraud et al. 2005); returns the squared norm left. What bounds it: the rows of
// the cluster, read from L2 twice a pass; a warp per product, so a pass has two barriers, where one
// product and one update at a time by the whole CTA had three per vector.
// Measured together with inverse_iteration below, both phases: n = 16384 39 -> 3.6 ms, eight solves of
// n = 2000 at a time 49 -> 5.3 ms in all (of which this form 2 and 1).
constexpr int kOrthPiece = 64;  // vectors orthogonalised together (pieces and seams)
constexpr int kOrthRun = 1024;  // and of a run of coinciding eigenvalues

template <typename T>
__device__ double cluster_project(int n, int i0, int v, T *z, int ldz, double *red)
{
    using W = Wide<T>;
    __shared__ typename W::Coef coef[kOrthPiece];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    T *zv = z + (size_t)v * ldz;
    for (int pass = 0; pass < 2; ++pass)
        for (int u0 = i0; u0 < v; u0 += kOrthPiece) {  // (once but for the long runs of phase 2)
            const int u1 = min(v, u0 + kOrthPiece);
            for (int u = u0 + warp; u < u1; u += nw) {
                const T *zu = z + (size_t)u * ldz;
                W a, b;
                int i = lane;
                for (; i + 32 < n; i += 64) {
                    a.fma_(zu[i], zv[i]);
                    b.fma_(zu[i + 32], zv[i + 32]);
                }
                if (i < n) a.fma_(zu[i], zv[i]);
                double s = a.value() + b.value();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) coef[u - u0] = W::coef(s);
            }
            __syncthreads();
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                W x(zv[i]);
                const T *zu = z + (size_t)u0 * ldz + i;
#pragma unroll 4
                for (int u = 0; u < u1 - u0; ++u) x.fms(coef[u], zu[(size_t)u * ldz]);
                zv[i] = x.rounded();
            }
            __syncthreads();
        }
    W s;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s.fma_(zv[i], zv[i]);
    return block_sum(s.value(), red);
}

__device__ __forceinline__ double hash_unit(unsigned a, unsigned b)
{
    unsigned h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
    h ^= h >> 15; h *= 0x2C1B3C6Du; h ^= h >> 12; h *= 0x297A2D39u; h ^= h >> 15;
    return (double)h * (2.0 / 4294967296.0) - 1.0;
}

// cstart[i] = first index of the cluster of i (chains of eigenvalues closer than
// tol_rel * ||T||). One CTA: each thread scans a contiguous segment, then the segment
// results are combined in order.
__global__ void cluster_start_kernel(int kvec, const double *w, const double *bounds, double tol_rel,
                                     int *cstart)
{
    __shared__ int last[1024];
    const double tol = tol_rel * fmax(bounds[3], DBL_MIN);
    const int nt = blockDim.x, t = threadIdx.x;
    const int seg = (kvec + nt - 1) / nt;
    const int a = t * seg, b = min(kvec, a + seg);
    int cur = -1;  // start of the current cluster inside the segment (-1: continues from left)
    for (int i = a; i < b; ++i) {
        if (i == 0 || !(w[i] - w[i - 1] < tol)) cur = i;
        cstart[i] = cur;
    }
    last[t] = cur;
    __syncthreads();
    if (t == 0)
        for (int q = 1; q < nt; ++q)
            if (last[q] < 0) last[q] = last[q - 1];
    __syncthreads();
    if (a < b && t > 0) {
        const int carry = last[t - 1];
        for (int i = a; i < b && cstart[i] < 0; ++i) cstart[i] = carry;
    }
}

// zv <- x / max |x|, x = (T_b - lambda I)^{-1} zv on the block [bs, be) from the factors L+ D+ L+^T of
// vector v (dplus; L+ = e / D+): forward L+ y = b, backward L+^T x = D+^{-1} y. Entries are rescaled
// (all at once) whenever one exceeds 2^500. work: x[i * kvec], the vector's spent U- column. By the
// whole CTA (kOrthThreads threads): a chunk of rows is loaded and divided in parallel, one thread runs the
// recurrence over it in shared memory, an FMA a row.
// Measured against one thread that loaded and divided row by row (1.1 us a row): n = 16384 18.5 -> 1.8 ms
// a phase.
constexpr int kOrthThreads = 256;
template <typename T>
__device__ void inverse_iteration(int n, int bs, int be, int kvec, int v, const double *__restrict__ e,
                                  const double *__restrict__ dplus, double *work, T *zv, double *red)
{
    __shared__ double sr[kOrthThreads], sb[kOrthThreads], sy[kOrthThreads];
    __shared__ int scales;  // rescalings in this chunk
    constexpr int C = kOrthThreads, kBig = (1023 + 500) << 20;
    const double shrink = 0x1p-500;
    const int tid = threadIdx.x;
    double *x = work + v;
    // the recurrence over rows first, first + dir, .. of the chunk: val = sb - sr val
    auto chain = [&](int first, int dir, int cnt, double val) {
        int times = 0;
        for (int j0 = 0; j0 < cnt; j0 += 4) {
            double r[4], c[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int j = first + dir * min(j0 + q, cnt - 1);
                r[q] = sr[j];
                c[q] = sb[j];
            }
            const int at = times;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (j0 + q >= cnt) break;
                const int j = first + dir * (j0 + q);
                for (int s = at; s < times; ++s)
                    if (dir < 0) c[q] *= shrink;  // right-hand sides loaded before a rescaling
                val = fma(-r[q], val, c[q]);
                if ((__double2hiint(val) & 0x7FFFFFFF) >= kBig) {
                    for (int i = 0; i < j0 + q; ++i) sy[first + dir * i] *= shrink;
                    if (dir < 0)  // the rows that are still to come are y of the forward pass
                        for (int i = j0 + 4; i < cnt; ++i) sb[first + dir * i] *= shrink;
                    val *= shrink;
                    ++times;
                }
                sy[j] = val;
            }
        }
        scales = times;
        return val;
    };
    double val = 0.0;  // (thread 0) last value of the recurrence
    for (int r0 = bs; r0 < be; r0 += C) {
        const int i = r0 + tid, cnt = min(C, be - r0);
        if (i < be) {
            sb[tid] = (double)zv[i];
            sr[tid] = i > bs ? e[i - 1] / dplus[(size_t)(i - 1) * kvec + v] : 0.0;
        }
        __syncthreads();
        if (tid == 0) val = chain(0, 1, cnt, val);
        __syncthreads();
        for (int s = 0; s < scales; ++s)
            for (int j = bs + tid; j < r0; j += C) x[(size_t)j * kvec] *= shrink;
        if (i < be) x[(size_t)i * kvec] = sy[tid];
        __syncthreads();
    }
    val = 0.0;
    int times = 0;  // rescalings so far, which rows not yet loaded still need
    for (int r0 = bs + (be - bs - 1) / C * C; r0 >= bs; r0 -= C) {
        const int i = r0 + tid, cnt = min(C, be - r0);
        if (i < be) {
            double y = x[(size_t)i * kvec];
            for (int s = 0; s < times; ++s) y *= shrink;
            const double d = dplus[(size_t)i * kvec + v];
            sb[tid] = y / d;
            sr[tid] = i < be - 1 ? e[i] / d : 0.0;
        }
        __syncthreads();
        if (tid == 0) val = chain(cnt - 1, -1, cnt, val);
        __syncthreads();
        times += scales;
        for (int s = 0; s < scales; ++s)
            for (int j = r0 + C + tid; j < be; j += C) x[(size_t)j * kvec] *= shrink;
        if (i < be) x[(size_t)i * kvec] = sy[tid];
        __syncthreads();
    }
    double mx = 0.0;
    for (int i = bs + tid; i < be; i += C) mx = fmax(mx, fabs(x[(size_t)i * kvec]));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((tid & 31) == 0) red[tid >> 5] = mx;
    __syncthreads();
    for (int q = 0; q < C / 32; ++q) mx = fmax(mx, red[q]);
    const double sc = (mx > 0.0 && mx <= DBL_MAX) ? 1.0 / mx : 0.0;
    for (int i = tid; i < n; i += C) zv[i] = (i >= bs && i < be) ? (T)(x[(size_t)i * kvec] * sc) : T(0);
}

// D+ of vector v for another shift, by the whole CTA: one thread runs the recurrence over chunks of
// rows in shared memory (rare: a second attempt below).
__device__ void shifted_factor(int bs, int be, int kvec, int v, const double *__restrict__ d,
                               const double *__restrict__ e, double lam, double pivmin, double *dplus)
{
    __shared__ double sd[kOrthThreads], se[kOrthThreads];
    const int tid = threadIdx.x;
    double dp = 0.0;
    for (int r0 = bs; r0 < be; r0 += kOrthThreads) {
        const int i = r0 + tid, cnt = min(kOrthThreads, be - r0);
        if (i < be) {
            sd[tid] = d[i] - lam;
            se[tid] = i > bs ? e[i - 1] : 0.0;
        }
        __syncthreads();
        if (tid == 0)
            for (int j = 0; j < cnt; ++j) {
                dp = r0 + j == bs ? sd[j] : fma(-(se[j] / dp), se[j], sd[j]);
                dp = guard_pivot(dp, pivmin);
                sd[j] = dp;
            }
        __syncthreads();
        if (i < be) dplus[(size_t)i * kvec + v] = sd[tid];
        __syncthreads();
    }
}

// |(T - lam I) z|^2
template <typename T>
__device__ double residual2(int n, const double *__restrict__ d, const double *__restrict__ e, double lam, const T *zv,
                            double *red)
{
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double r = (d[i] - lam) * (double)zv[i];
        if (i > 0) r = fma(e[i - 1], (double)zv[i - 1], r);
        if (i + 1 < n) r = fma(e[i], (double)zv[i + 1], r);
        s = fma(r, r, s);
    }
    return block_sum(s, red);
}

// Gram-Schmidt (two passes) within clusters of eigenvalues closer than tol_rel * ||T||,
// on ranges of at most kOrthPiece vectors: phase 0 takes the pieces [s + 64p, s + 64p + 64)
// of a cluster starting at s, phase 1 the seams [s + 64p + 32, s + 64p + 96) that cross a
// piece boundary; one CTA per range start. Eigenvalues that coincide to working accuracy have vectors
// that are anything in their space, not orthogonal to eps ||T|| / spacing beyond a seam: phase 2 takes
// every run of more than 32 of them whole, up to kOrthRun (binary64; one CTA, so time
// grows with the square of the run: 64-fold at n = 600 10 ms). A vector that the projection nearly annihilates (its
// eigenvalue coincides with an earlier one to working accuracy, as for the pairs of the
// real form of a complex Hermitian matrix) is replaced by one step of inverse iteration
// on its block, x = (T_b - lambda I)^{-1} b for a pseudo-random b orthogonal to the
// cluster's vectors, using the L+ D+ L+^T factors that the twisted factorisation left in
// dplus (the vector's spent U- column holds the intermediate values), and is then
// projected and normalised again. When lambda sits much closer to an accepted vector's
// eigenvalue than to its own, that vector dominates x; what is left after the projection
// is still accurate as long as it is far above the rounding level. In a group of many eigenvalues
// that coincide to working accuracy lambda can be one of them to the last bit, and then x is that
// one vector whatever b is; and where T splits, two of the group can have been given the same place
// in the same block. So further attempts shift lambda by some roundings of ||T||, from where the
// members of the group look alike (residuals stay at that size), and take all of T.
template <typename T>
__global__ void cluster_orth_kernel(int n, int kvec, const int *cstart, int phase, const double *d, const double *e,
                                    const double *w, const double *bounds, int *blk, double *dplus, double *work,
                                    T *z, int ldz, int *status)
{
    __shared__ double red[32];
    const int i0 = blockIdx.x;
    int cend = i0 + 1;  // end of the range
    if (phase < 2) {
        const int s = cstart[i0];
        const int off = phase == 0 ? 0 : kOrthPiece / 2;
        if ((i0 - s) % kOrthPiece != off) return;  // not a range start
        while (cend < kvec && cend < i0 + kOrthPiece && cstart[cend] == s) ++cend;
        if (phase == 1 && cend <= i0 + kOrthPiece / 2) return;  // no piece boundary inside
    } else {
        // (some hundred roundings; with one huge eigenvalue more would take in the rest of the spectrum)
        const double same = 1e-13 * bounds[3];
        if (i0 > 0 && w[i0] - w[i0 - 1] <= same) return;
        while (cend < kvec && cend < i0 + kOrthRun && w[cend] - w[cend - 1] <= same) ++cend;
        if (cend - i0 <= kOrthPiece / 2) return;
    }
    const int i1 = cend;
    for (int v = i0; v < i1; ++v) {
        const bool lost = blk[2 * v + 1] < 0;  // no vector from the twisted factorisation
        if (v == i0 && !lost) continue;
        T *zv = z + (size_t)v * ldz;
        double s = lost ? 0.0 : cluster_project(n, i0, v, z, ldz, red);
        // a regenerated vector is accepted when its part orthogonal to the cluster is far above the
        // rounding level of T (its direction error is then eps / sqrt(s)). In binary64, before the last
        // attempt, when that is a good part of it: what is wrong with the vectors before it enters
        // with the factor 1 / sqrt(s), and adds up over a large group. (Binary32 vectors are refined.)
        constexpr int kAttempts = 5;
        double accept = 1e-4;
        for (int attempt = lost ? 1 : 0; attempt < kAttempts && !(s >= accept); ++attempt) {
            accept = sizeof(T) == 4 ? 1e-8 : attempt + 1 < kAttempts ? 1e-3 : 1e-16;
            const int bs = attempt == 0 ? blk[2 * v] : 0, be = attempt == 0 ? blk[2 * v + 1] : n;
            if (attempt > 0) {
                const double roundings = attempt == 1 ? 8.0 : attempt == 2 ? -8.0 : attempt == 3 ? 32.0 : -128.0;
                // in units of the eigenvalues' accuracy (2e-9 ||T|| at most in the binary32 route)
                const double unit = (sizeof(T) == 8 ? DBL_EPSILON : 1e-9) * bounds[3];
                shifted_factor(bs, be, kvec, v, d, e, w[v] + roundings * unit, bounds[2], dplus);
            }
            // start b: pseudo-random on the block, orthogonal to the cluster's vectors
            for (int i = threadIdx.x; i < n; i += blockDim.x)
                zv[i] = (i >= bs && i < be) ? (T)hash_unit((unsigned)(v * 7919 + attempt), (unsigned)i) : T(0);
            __syncthreads();
            cluster_project(n, i0, v, z, ldz, red);
            inverse_iteration(n, bs, be, kvec, v, e, dplus, work, zv, red);
            __syncthreads();
            double nr = 0.0;
            for (int i = threadIdx.x; i < n; i += blockDim.x) nr += (double)zv[i] * (double)zv[i];
            nr = block_sum(nr, red);
            const double inv = (nr > 0.0) ? 1.0 / sqrt(nr) : 0.0;
            for (int i = threadIdx.x; i < n; i += blockDim.x) zv[i] = (T)((double)zv[i] * inv);
            __syncthreads();
            s = cluster_project(n, i0, v, z, ldz, red);
            // with every vector of the group in this block taken, x is of other eigenvalues (binary64; 1e-14:
            // the rounding of the projection)
            if (sizeof(T) == 8) {
                const double tol = (1e-10 * sqrt(s) + 1e-14) * bounds[3] + 8.0 * bounds[2];
                if (!(residual2(n, d, e, w[v], zv, red) <= tol * tol)) s = 0.0;
            }
        }
        if (!(s >= accept)) {
            if (threadIdx.x == 0) report_error(status, ELSI_ERR_NO_CONVERGENCE, v);
            return;
        }
        const double inv = 1.0 / sqrt(s);
        for (int i = threadIdx.x; i < n; i += blockDim.x) zv[i] = (T)((double)zv[i] * inv);
        if (lost && threadIdx.x == 0) blk[2 * v + 1] = -blk[2 * v + 1];
        __syncthreads();
    }
}

template <typename T>
cudaError_t stein(cudaStream_t st, int n, const double *d, const double *e, int kvec,
                  const double *w, T *z, int ldz, double *scratch, int *status)
{
    if (n <= 0 || kvec <= 0) return cudaSuccess;
    // scratch: D+ (n x kvec), U- (n x kvec), bounds (8), blk (2 kvec ints), L+ (n x kvec)
    double *dplus = scratch, *uminus = scratch + (size_t)n * kvec;
    double *bounds = scratch + (size_t)2 * n * kvec;
    int *blk = reinterpret_cast<int *>(bounds + 8);
    double *lplus = bounds + 16 + kvec;
    EGB_COUNT_LAUNCH();
    gershgorin_kernel<<<1, 1024, 0, st>>>(n, d, e, bounds);
    EGB_COUNT_LAUNCH();
    block_assign_kernel<<<ceil_div(kvec, 64), 64, 0, st>>>(n, d, e, kvec, w, bounds, blk);
    EGB_COUNT_LAUNCH();
    twist_factor_kernel<<<dim3(ceil_div(kvec, 32), 2), 32, 0, st>>>(d, e, kvec, w, bounds, blk, dplus, lplus, uminus);
    EGB_COUNT_LAUNCH();
    twist_vector_kernel<T><<<ceil_div(kvec, 32), 32 * kTwistWarps, 0, st>>>(n, d, e, kvec, w, bounds, blk, dplus, lplus,
                                                                           uminus, z, ldz);
    // cluster starts (in the L+ scratch, no longer needed), then pieces and seams
    int *cstart = reinterpret_cast<int *>(lplus);
    EGB_COUNT_LAUNCH();
    cluster_start_kernel<<<1, 1024, 0, st>>>(kvec, w, bounds, 1e-5, cstart);
    for (int phase = 0; phase < (sizeof(T) == 8 && kvec > kOrthPiece / 2 ? 3 : 2); ++phase) {
        EGB_COUNT_LAUNCH();
        cluster_orth_kernel<T><<<kvec, kOrthThreads, 0, st>>>(n, kvec, cstart, phase, d, e, w, bounds, blk, dplus, uminus,
                                                              z, ldz, status);
    }
    return cudaGetLastError();
}

template cudaError_t stein<double>(cudaStream_t, int, const double *, const double *, int,
                                   const double *, double *, int, double *, int *);
template cudaError_t stein<float>(cudaStream_t, int, const double *, const double *, int,
                                  const double *, float *, int, double *, int *);

}  // namespace egb
