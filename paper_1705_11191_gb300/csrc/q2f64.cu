// Back-transformation through Q2 (step (4) of the two-stage method, arXiv:1705.11191 sec. 3.1)
// in binary64: Z <- Q2 Z, Q2 = prod over sweep blocks J (64 sweeps, ascending) of prod over
// steps t (descending) of H(J,t) H(J+1,t) ... H(J+63,t); so the blocks are applied from the
// last to the first, t ascending, and inside a group the later sweep first.
//
// What bounds it: binary64 FMAs, two a clock and SM (4 b k n^2 / (2 b) of them), and the order
// of the reflectors, which is one chain per column of Z. One warp works on four columns, eight
// lanes a column: a reflector is b / 8 FMAs a lane for the dot product, three shuffled
// additions, and b / 8 FMAs for the update. A CTA of one warp per four columns leaves most of
// the chip's FMA units without a warp (k = 668 columns: 167 warps for 608 schedulers), so the
// sweep blocks themselves are pipelined: eight warps of a CTA work on the same four columns,
// warp w on the w-th block of a round, one step behind warp w - 1. Their windows do not
// overlap, since step t of block J ends below row J + 65 + (t + 1) b, where block J + 64 starts
// step t + 1. The rows between the first and the last warp's windows are in a ring in shared
// memory: the first warp brings rows in, the last one stores them.
//
// The b rows under a reflector stay in registers: row g is in slot g mod b (lane slot mod 8,
// register slot / 8), and from one reflector to the next one row leaves to the ring and one
// enters in its slot. The reflector is read from L2 in the rotated order, one ahead.
//
// Measured against one warp per four columns with its rows in shared memory: n = 512, k = 512
// 2.9 -> 0.9 ms, n = 1531, k = 381 25 -> 5.7 ms, n = 5000, k = 668 264 -> 97 ms (b = 32; 167 CTAs
// on 152 SMs, so that some SMs do twice the work of the others).
#include "common.cuh"
#include "kernels.h"
#include "packets.cuh"

namespace egb {
namespace q2d {

constexpr int kM = 64;       // sweeps per block
constexpr int kP = 8;        // warps: blocks in the pipeline
constexpr int kCols = 4;     // columns of Z per CTA
constexpr int kRing = 2048;  // ring rows: kP * 64 + (kLead + 3) * b of them in use at most
constexpr int kLead = 12;    // steps the first warp may be ahead of the last
constexpr int kLd = kRing + 4;
constexpr int kSmem = kCols * kLd * (int)sizeof(double);
static_assert(kP * kM + (kLead + 3) * 64 + 64 <= kRing, "ring");

struct Args {
    int n, S, k, ldz;
    const double *v2, *tau2;
    double *z;
    int *status;
    long long spin_limit;
};

__device__ __forceinline__ void cp_async8(double *dst, const double *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src));
}

template <int B>
__global__ void __launch_bounds__(32 * kP) q2_f64_kernel(const Args a)
{
    constexpr int RPT = B / 8;  // rows of a lane
    extern __shared__ __align__(16) double ring[];  // [column][row mod kRing]
    __shared__ volatile int progress[kP];
    __shared__ volatile int failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int sub = lane & 7, col = lane >> 3;
    const int n = a.n, S = a.S;
    const int c0 = blockIdx.x * kCols, ncol = min(kCols, a.k - c0);
    const int nsweep = n - 2, nblk = (nsweep + kM - 1) / kM;
    double *my = ring + col * kLd;
    auto at = [&](int row) -> double & { return my[row & (kRing - 1)]; };
    // rows [r0, r1) of the CTA's columns into the ring (zeros past n and past the columns)
    auto fetch = [&](int r0, int r1, int first, int step) {
        for (int e = first; e < (r1 - r0) * kCols; e += step) {
            const int r = r0 + e % (r1 - r0), c = e / (r1 - r0);
            double *d = ring + c * kLd + (r & (kRing - 1));
            if (r < n && c < ncol) cp_async8(d, a.z + (size_t)r + (size_t)(c0 + c) * a.ldz);
            else *d = 0.0;
        }
        asm volatile("cp.async.commit_group;\n" ::);
    };
    if (tid == 0) failed = 0;
    __syncthreads();

    for (int top = nblk - 1; top >= 0; top -= kP) {
        const int act = min(kP, top + 1);  // blocks of this round: top, top - 1, .., top - act + 1
        const int Jlead = top * kM, Jlast = (top - act + 1) * kM;
        const int lead_end = Jlead + kM + B;  // rows below this are needed by step 0 of the first block
        fetch(Jlast + 1, lead_end, tid, 32 * kP);
        asm volatile("cp.async.wait_group 0;\n" ::);
        if (tid < kP) progress[tid] = 0;
        __syncthreads();
        if (warp < act) {
            const int J = (top - warp) * kM, Jend = min(nsweep, J + kM);
            const int SJ = (n - 2 - J) / B + 1;
            const int Sprev = warp > 0 ? (n - 2 - (J + kM)) / B + 1 : 0;
            const int Slast = (n - 2 - Jlast) / B + 1;
            int stored = Jlast + 1;  // last block: rows below are back in z
            bool ok = true;
            for (int t = 0; t < SJ; ++t) {
                // ---- wait: the block ahead has finished step t; the first block must not run away
                {
                    const int w = warp > 0 ? warp - 1 : act - 1;
                    const int need = warp > 0 ? min(t + 1, Sprev) : min(t - kLead, Slast);
                    long long it = 0;
                    while (progress[w] < need && act > 1) {
                        if (failed) { ok = false; break; }
                        if (++it > a.spin_limit) {
                            if (lane == 0) report_error(a.status, ELSI_ERR_TIMEOUT, t);
                            failed = 1;
                            ok = false;
                            break;
                        }
                    }
                    ok = __all_sync(0xffffffffu, ok);
                    if (!ok) break;
                    __threadfence_block();
                }
                if (warp == 0) {
                    asm volatile("cp.async.wait_group 0;\n" ::);
                    __syncwarp();
                    // rows of the next step
                    const int r0 = lead_end + t * B;
                    if (r0 < n + B + kM) fetch(r0, r0 + B, lane, 32);
                }
                // ---- the group's reflectors, later sweep first
                const int jtop = min(Jend - 1, n - 2 - t * B);  // sweeps above have no step t
                if (jtop >= J) {
                    double z[RPT], v[RPT], vn[RPT];
                    int rs;  // slot of the reflector's first row
                    auto load_v = [&](int j, double (&d)[RPT]) {
                        const int r = (j + 1 + t * B) % B;
                        const double *p = a.v2 + ((size_t)j * S + t) * B;
#pragma unroll
                        for (int q = 0; q < RPT; ++q) {
                            const int i = sub + 8 * q - r;
                            d[q] = __ldg(p + (i < 0 ? i + B : i));
                        }
                    };
                    int r0 = jtop + 1 + t * B;
                    rs = r0 % B;
                    double taun = __ldg(a.tau2 + (size_t)jtop * S + t);
                    load_v(jtop, vn);
#pragma unroll
                    for (int q = 0; q < RPT; ++q) {
                        const int i = sub + 8 * q - rs;
                        z[q] = at(r0 + (i < 0 ? i + B : i));
                    }
                    for (int j = jtop; j >= J; --j) {
                        const double tau = taun;
#pragma unroll
                        for (int q = 0; q < RPT; ++q) v[q] = vn[q];
                        double zin = 0.0;
                        if (j > J) {  // the next reflector, and the row that comes with it
                            taun = __ldg(a.tau2 + (size_t)(j - 1) * S + t);
                            load_v(j - 1, vn);
                            zin = at(r0 - 1);
                        }
                        if (tau != 0.0) {
                            double s0 = 0.0, s1 = 0.0;
#pragma unroll
                            for (int q = 0; q < RPT; q += 2) {
                                s0 = fma(v[q], z[q], s0);
                                if (q + 1 < RPT) s1 = fma(v[q + 1], z[q + 1], s1);
                            }
                            double s = RPT > 1 ? s0 + s1 : s0;
                            s += __shfl_xor_sync(0xffffffffu, s, 4);
                            s += __shfl_xor_sync(0xffffffffu, s, 2);
                            s += __shfl_xor_sync(0xffffffffu, s, 1);
                            s *= -tau;
#pragma unroll
                            for (int q = 0; q < RPT; ++q) z[q] = fma(s, v[q], z[q]);
                        }
                        if (j > J) {
                            // row r0 + B - 1 leaves, row r0 - 1 takes its slot
                            const int sl = rs == 0 ? B - 1 : rs - 1;
                            if (sub == (sl & 7)) {
                                at(r0 + B - 1) = pick(z, sl >> 3);
#pragma unroll
                                for (int q = 0; q < RPT; ++q) move_if(z[q], zin, sl >> 3, q);
                            }
                            rs = sl;
                            --r0;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < RPT; ++q) {
                        const int i = sub + 8 * q - rs;
                        at(r0 + (i < 0 ? i + B : i)) = z[q];
                    }
                }
                __syncwarp();
                // ---- the last block's finished rows go back to z
                if (warp == act - 1) {
                    const int upto = t + 1 == SJ ? n : min(n, J + 1 + (t + 1) * B);
                    const int nr = upto - stored;
                    for (int e = lane; e < nr * kCols; e += 32) {
                        const int r = stored + e % nr, c = e / nr;
                        if (c < ncol) a.z[(size_t)r + (size_t)(c0 + c) * a.ldz] = ring[c * kLd + (r & (kRing - 1))];
                    }
                    stored = upto > stored ? upto : stored;
                }
                __threadfence_block();
                __syncwarp();
                if (lane == 0) progress[warp] = t + 1;
            }
        }
        asm volatile("cp.async.wait_group 0;\n" ::);
        __syncthreads();  // the next round starts from the rows this one stored
        if (failed) return;
    }
}

template <int B>
cudaError_t launch(cudaStream_t st, const Args &a)
{
    static PerDeviceOnce attr;
    cudaError_t e = once_per_device(attr, [] {
        return cudaFuncSetAttribute(q2_f64_kernel<B>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    });
    if (e != cudaSuccess) return e;
    EGB_COUNT_LAUNCH();
    q2_f64_kernel<B><<<ceil_div(a.k, kCols), 32 * kP, kSmem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace q2d

cudaError_t apply_q2_f64(cudaStream_t st, int n, int b, const double *v2, const double *tau2, int k, double *z,
                         int ldz, int *status)
{
    if (n < 3 || k <= 0) return cudaSuccess;
    q2d::Args a;
    a.n = n; a.S = sb2st_steps(n, b); a.k = k; a.ldz = ldz; a.v2 = v2; a.tau2 = tau2; a.z = z;
    a.status = status; a.spin_limit = spin_limit();
    switch (b) {
    case 8: return q2d::launch<8>(st, a);
    case 16: return q2d::launch<16>(st, a);
    case 24: return q2d::launch<24>(st, a);
    case 32: return q2d::launch<32>(st, a);
    case 40: return q2d::launch<40>(st, a);
    case 48: return q2d::launch<48>(st, a);
    case 56: return q2d::launch<56>(st, a);
    case 64: return q2d::launch<64>(st, a);
    }
    return cudaErrorInvalidValue;
}

}  // namespace egb
