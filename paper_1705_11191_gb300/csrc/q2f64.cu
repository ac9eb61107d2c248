// Back-transformation through Q2 (step (4) of the two-stage method, arXiv:1705.11191 sec. 3.1)
// in binary64: Z <- Q2 Z, Q2 = prod over sweep blocks J (16 sweeps, ascending) of prod over
// steps t (descending) of H(J,t) H(J+1,t) ... H(J+15,t); so the blocks are applied from the
// last to the first, t ascending, and inside a group the later sweep first.
//
// What bounds it: binary64 operations, a warp's instruction every 64 clocks on each of the 608
// schedulers, and the order of the reflectors, which is one chain per column of Z. LPC lanes
// work on a column: a reflector is b / LPC operations a lane for the dot product, log2(LPC) + 2
// to add it up and scale it, b / LPC for the update. Few lanes per column waste less on the sum
// (b = 32: 67 of 64 operations with one lane, 12 of 8 with eight), many make the chain shorter and
// give more warps. The rule of lanes_per_column() weighs the two.
//
// Pipeline over the blocks. There are too few columns to fill the chip, so the unit of work of a
// warp is (block, 32 / LPC columns): step t of block J ends above the rows of step t + 1 of block
// J + 16, so block J runs one step behind block J + 16, in whatever warp that is. The rows go
// through L2 (a step takes 7 us or more, a hand-over about one); a progress word per unit says
// how many steps are stored. Units are handed out by a counter in the order of the blocks, so a
// unit waits only for one that was handed out before it, whatever the number of warps that run.
//
// The b rows under a reflector stay in registers: row g is in slot g mod b, and from one reflector
// to the next one row leaves and one enters in its slot, both loaded and stored in L2 directly.
// The reflector is in shared memory in the order of the slots, loaded one ahead by the lanes together.
//
// Measured against eight lanes per column and a pipeline of eight blocks of 64 sweeps inside a CTA, its
// rows in a ring in shared memory (b = 32): n = 5000, k = 668 97 -> 36 ms (two lanes; the 390 000
// reflectors are 30 ms of the binary64 units); n = 1531, k = 381 5.7 -> 3.4 ms (four); n = 1000 2.7 ->
// 1.6 ms and n = k = 512 0.91 -> 0.80 ms (eight). Blocks of 32 sweeps: 39, 4.1, 2.0 and 0.99 ms.
#include "common.cuh"
#include "kernels.h"
#include "packets.cuh"

namespace egb {
namespace q2d {

constexpr int kM = 16;      // sweeps per block
constexpr int kWarps = 4;   // warps per CTA, each with its own units

// sync words: units handed out, a warp gave up, steps stored by each unit
constexpr int kSyncNext = 0, kSyncStop = 1, kSyncHead = 2;

struct Args {
    int n, S, k, ldz;
    const double *v2, *tau2;
    double *z;
    int *status;
    unsigned *sync;
    long long spin_limit;
};

template <int B, int LPC>
__global__ void __launch_bounds__(32 * kWarps) q2_f64_kernel(const Args a)
{
    constexpr int RPT = B / LPC;       // rows of a lane
    constexpr int NCOL = 32 / LPC;     // columns of a warp
    constexpr int VPL = (B + 31) / 32; // entries of a reflector that a lane loads
    static_assert(RPT % 2 == 0, "pairs of slots");
    // slot s belongs to lane part s % (2 LPC) / 2, in register s / (2 LPC) * 2 + s % 2
    __shared__ __align__(16) double sv[kWarps][2][B];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int part = lane % LPC;
    const int n = a.n, S = a.S, nsweep = n - 2;
    const int ncg = (a.k + NCOL - 1) / NCOL, nblk = (nsweep + kM - 1) / kM;
    const long long units = (long long)ncg * nblk;
    double(*const sw)[B] = sv[warp];

    for (;;) {
        unsigned u = 0;
        if (lane == 0) u = atomicAdd(a.sync + kSyncNext, 1u);
        u = __shfl_sync(0xffffffffu, u, 0);
        if (u >= units) return;
        const int rank = u / ncg, J = (nblk - 1 - rank) * kM;
        const int col = (u % ncg) * NCOL + lane / LPC;
        const bool colok = col < a.k;
        double *zc = a.z + (size_t)(colok ? col : 0) * a.ldz;
        const int SJ = (n - 2 - J) / B + 1;
        const int Sabove = rank > 0 ? (n - 2 - (J + kM)) / B + 1 : 0;
        const unsigned *above = a.sync + kSyncHead + u - ncg;
        int seen = 0;
        auto row = [&](int r, bool mine) { return mine && colok && r < n ? __ldcg(zc + r) : 0.0; };
        for (int t = 0; t < SJ; ++t) {
            // ---- the block above must have stored its step t
            const int need = min(t + 1, Sabove);
            for (long long it = 0; seen < need; ++it) {
                unsigned v, stop = 0;
                asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(above) : "memory");
                seen = (int)v;
                if (seen >= need) break;
                if ((it & 63) == 63)
                    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(stop) : "l"(a.sync + kSyncStop));
                if (stop || it > a.spin_limit) { seen = -1; break; }
            }
            if (!__all_sync(0xffffffffu, seen >= need)) {
                if (lane == 0) {
                    report_error(a.status, ELSI_ERR_TIMEOUT, t);
                    atomicExch(a.sync + kSyncStop, 1u);
                }
                return;
            }
            // ---- the group's reflectors, later sweep first
            const int jtop = min(min(nsweep, J + kM) - 1, n - 2 - t * B);  // sweeps above have no step t
            if (jtop >= J) {
                double z[RPT], vn[VPL], taun;
                // entry e of reflector j belongs to row j + 1 + t B + e: the lanes load it by slot
                auto load_v = [&](int j) {
                    const int r = (j + 1 + t * B) % B;
                    const double *p = a.v2 + ((size_t)j * S + t) * B;
#pragma unroll
                    for (int q = 0; q < VPL; ++q) {
                        const int s = lane + 32 * q, i = s - r;
                        if (s < B) vn[q] = __ldg(p + (i < 0 ? i + B : i));
                    }
                    taun = __ldg(a.tau2 + (size_t)j * S + t);
                };
                auto store_v = [&](int j) {
#pragma unroll
                    for (int q = 0; q < VPL; ++q)
                        if (lane + 32 * q < B) sw[j & 1][lane + 32 * q] = vn[q];
                };
                int r0 = jtop + 1 + t * B, rs = r0 % B;  // the reflector's first row and its slot
                load_v(jtop);
#pragma unroll
                for (int q = 0; q < RPT; ++q) {
                    const int i = (q >> 1) * 2 * LPC + 2 * part + (q & 1) - rs;
                    z[q] = row(r0 + (i < 0 ? i + B : i), true);
                }
                store_v(jtop);
                double tau = taun;
                __syncwarp();
                for (int j = jtop; j >= J; --j) {
                    const int sl = rs == 0 ? B - 1 : rs - 1;  // row r0 + B - 1 leaves it, row r0 - 1 enters
                    const bool mine = part == (sl % (2 * LPC)) / 2;
                    double zin = 0.0;
                    if (j > J) {  // the next reflector, and the row that comes with it
                        load_v(j - 1);
                        zin = row(r0 - 1, mine);
                    }
                    if (tau != 0.0) {
                        const double2 *v = reinterpret_cast<const double2 *>(sw[j & 1]) + part;
                        double s0 = 0.0, s1 = 0.0;
#pragma unroll
                        for (int q = 0; q < RPT; q += 2) {
                            const double2 x = v[(q >> 1) * LPC];
                            s0 = fma(x.x, z[q], s0);
                            s1 = fma(x.y, z[q + 1], s1);
                        }
                        double s = s0 + s1;
#pragma unroll
                        for (int d = LPC / 2; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
                        s *= -tau;
#pragma unroll
                        for (int q = 0; q < RPT; q += 2) {
                            const double2 x = v[(q >> 1) * LPC];
                            z[q] = fma(s, x.x, z[q]);
                            z[q + 1] = fma(s, x.y, z[q + 1]);
                        }
                    }
                    if (j > J) {
                        const int q0 = sl / (2 * LPC) * 2 + (sl & 1);
                        if (mine) {
                            if (colok && r0 + B - 1 < n) __stcg(zc + r0 + B - 1, pick(z, q0));
#pragma unroll
                            for (int q = 0; q < RPT; ++q) move_if(z[q], zin, q0, q);
                        }
                        store_v(j - 1);
                        tau = taun;
                        rs = sl;
                        --r0;
                        __syncwarp();
                    }
                }
#pragma unroll
                for (int q = 0; q < RPT; ++q) {
                    const int i = (q >> 1) * 2 * LPC + 2 * part + (q & 1) - rs;
                    const int r = r0 + (i < 0 ? i + B : i);
                    if (colok && r < n) __stcg(zc + r, z[q]);
                }
            }
            __syncwarp();
            if (lane == 0)
                asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(a.sync + kSyncHead + u), "r"((unsigned)(t + 1))
                             : "memory");
        }
    }
}

template <int B, int LPC>
cudaError_t launch(cudaStream_t st, const Args &a, int num_sms)
{
    const long long units = (long long)ceil_div(a.k, 32 / LPC) * ceil_div(a.n - 2, kM);
    cudaError_t e = cudaMemsetAsync(a.sync, 0, (size_t)(kSyncHead + units) * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    const long long ctas = (units + kWarps - 1) / kWarps;
    EGB_COUNT_LAUNCH();
    q2_f64_kernel<B, LPC><<<(int)(ctas < 2 * num_sms ? ctas : 2 * num_sms), 32 * kWarps, 0, st>>>(a);
    return cudaGetLastError();
}

// Lanes per column, by the longer of two times in units of a warp instruction on one scheduler: all
// reflectors of all columns over the 608 schedulers, and the chain through the blocks (n / 16
// blocks, a step apart, and the n / b steps of the last one).
inline double cost(int n, int b, int k, int lpc)
{
    const double op = 2.0 * b / lpc + 2 + (lpc > 1) + (lpc > 2) + (lpc > 4), steps = 0.5 * n / kM * (n / b + 1.0);
    const double work = steps * ceil_div(k, 32 / lpc) / 608.0, chain = (double)n / kM + (double)n / b;
    return op * (work > chain ? work : chain);
}

inline size_t words(int n, int k, int lpc) { return kSyncHead + (size_t)ceil_div(k, 32 / lpc) * ceil_div(n - 2, kM); }

}  // namespace q2d

size_t q2_f64_sync_words(int n) { return n < 3 ? 1 : q2d::words(n, n, 4); }

cudaError_t apply_q2_f64(cudaStream_t st, int n, int b, const double *v2, const double *tau2, int k, double *z,
                         int ldz, int *status, unsigned *sync, size_t sync_words)
{
    if (n < 3 || k <= 0) return cudaSuccess;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int lpc = 4;
    if (b == 32 || b == 64)
        for (int l = 2; l <= 8; l *= 4)
            if (q2d::cost(n, b, k, l) < q2d::cost(n, b, k, lpc) && q2d::words(n, k, l) <= sync_words) lpc = l;
    if (q2d::words(n, k, lpc) > sync_words) return cudaErrorInvalidValue;
    q2d::Args a;
    a.n = n; a.S = sb2st_steps(n, b); a.k = k; a.ldz = ldz; a.v2 = v2; a.tau2 = tau2; a.z = z;
    a.status = status; a.sync = sync; a.spin_limit = spin_limit();
    switch (b) {
    case 8: return q2d::launch<8, 4>(st, a, sms);
    case 16: return q2d::launch<16, 4>(st, a, sms);
    case 24: return q2d::launch<24, 4>(st, a, sms);
    case 32: return lpc == 2 ? q2d::launch<32, 2>(st, a, sms) : lpc == 4 ? q2d::launch<32, 4>(st, a, sms) : q2d::launch<32, 8>(st, a, sms);
    case 40: return q2d::launch<40, 4>(st, a, sms);
    case 48: return q2d::launch<48, 4>(st, a, sms);
    case 56: return q2d::launch<56, 4>(st, a, sms);
    case 64: return lpc == 2 ? q2d::launch<64, 2>(st, a, sms) : lpc == 4 ? q2d::launch<64, 4>(st, a, sms) : q2d::launch<64, 8>(st, a, sms);
    }
    return cudaErrorInvalidValue;
}

}  // namespace egb
