// Band -> tridiagonal bulge chase with the band held on chip (arXiv:1705.11191 Eq. 11,
// second line; the same reflectors and the same order as chase_kernel in sb2st.cu).
//
// What bounds it: the chase is one chain. Step t of sweep j + 1 needs step t + 1 of sweep
// j, which needs step t of sweep j, so n sweeps cost n times (two steps + two hand-overs),
// whatever the number of SMs. With a CTA per sweep every step loads a 2b x b window of the
// band from L2, stores it again and hands over through a fence and a flag: 7.4 us a step
// in binary32 and 17 us in binary64 (b = 64).
//
// Layout: a CTA per step position t instead. Its window (X = A[r .. r+b-1, r-b .. r-1] and
// D = A[r .. r+b-1]^2, r = j + 1 + t b) moves by one row and column per sweep; row and column
// g of the matrix live in slot g mod b, so a sweep replaces one slot and moves nothing:
// thread (row slot i, column slots c0 ..) keeps its elements of X and D in registers for
// the whole reduction, and the column that leaves D enters X inside the same thread. What
// two positions exchange per sweep is a reflector (t -> t + 1: b + 1 values) and one row
// (t + 1 -> t: b + 1 values), as packets of value and sweep number in one 64-bit word: the
// reader polls the data itself, so a hand-over is one store and one load through L2 with
// no fence and no separate flag. A position's first step after its reflector is known
// sends it on before updating its own D.
//
// Per step, with v_p, tau_p the previous position's reflector (X0 before the step):
//   y = tau_p X0 v_p, x = X0[:, first] - y, v = house(x), p = tau v^T (X0 - y v_p^T),
//   q = tau D v, w = q - (1/2) tau (v.q) v,
//   X = X0 - y v_p^T - v p^T,  D = D - v w^T - w v^T.
// The column sums x^T X0 and D x are taken with the unscaled x (x_first apart). A sweep's share of
// the chain is one step from its reflector's arrival to the row it sends back and one from a row's
// arrival to the reflector it sends on, so each step sends as early as it can: the reflector
// before the sums x^T X0 and D x, the row before the update of D (in binary64, where an
// operation holds a warp's unit 64 clocks, 57 -> 40 and 121 -> 101 operations).
//
// Measured against the kernel of sb2st.cu: binary32, b = 64, n = 777 10.6 -> 2.7 ms, n = 4096
// 60.3 -> 16.0 ms, n = 16384 245 -> 70 ms (14.7 -> 3.5 - 4.3 us a sweep, two L2 hand-overs and
// two steps' arithmetic); binary64, b = 64, n = 512 15.2 -> 11.0 ms, n = 1531 51.3 -> 35.7 ms (a
// step's 28 000 FMAs at two a clock bound it), and with b = 32 4.5 and 14.0 ms, 3.8 and 11.9 with
// the early messages (3.9, 12.3) and the shorter reciprocals of packets.cuh. As one cluster, up to 16
// positions: n = 512 3.8 -> 3.5 ms, binary32 n = 777 2.65 -> 2.27 ms.
#include "common.cuh"
#include "kernels.h"
#include "packets.cuh"

namespace egb {
namespace sys {

using namespace pkt;

struct Args {
    int n, ldb, S;      // S positions = grid size; also the stride of the reflector slots
    u64 *vmsg, *rmsg;   // reflector / row packets, one record of kWords<T> * (B + 2) words each
    int *status;
    long long spin_limit;
};

// A value that what follows cannot be computed before this point
__device__ __forceinline__ void pin(double &x) { asm volatile("" : "+d"(x)); }
__device__ __forceinline__ void pin(float &x) { asm volatile("" : "+f"(x)); }

template <typename T, int B, bool CL>
__global__ void __launch_bounds__(4 * B, 512 / (4 * B))
chase_resident_kernel(const T *__restrict__ band, T *v2, T *tau2, double *dout, double *eout, const Args a)
{
    constexpr int CPT = B / 4;       // columns of a row per thread (four threads per row)
    constexpr int NW = 4 * B / 32;   // warps
    constexpr int PH = CPT / 8;      // columns per lane after the in-warp column sums
    // binary32: the column sums cost less than the barrier that taking them later needs
    constexpr bool EARLY = sizeof(T) == 4;
    __shared__ __align__(16) T vps[2][B];      // v_p by slot (double buffered: see the end)
    __shared__ __align__(16) T rows_[2][B];    // row message by slot
    __shared__ T msc[2][2];                    // tau_p, d of the row message
    __shared__ __align__(16) T xs[B], xrow[B], ps[B], qs[B], vs[B];
    __shared__ __align__(16) T upart[NW][B];
    __shared__ T red[3][NW], ysl[2];           // partial sums; x and y at the first row
    __shared__ int failed;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int i = tid >> 2, part = tid & 3, c0 = part * CPT, quad = lane & ~3;
    const int t = blockIdx.x, n = a.n, ldb = a.ldb;
    const int nsweep = n - 2;
    constexpr int REC = kWords<T> * (B + 2);
    u64 *vin = a.vmsg + (size_t)(t > 0 ? t - 1 : 0) * REC, *vout = a.vmsg + (size_t)t * REC;
    u64 *rin = a.rmsg + (size_t)t * REC, *rout = a.rmsg + (size_t)(t > 0 ? t - 1 : 0) * REC;
    // CL: the positions are one cluster (and some idle CTAs), messages go to the reader's shared memory
    __shared__ u64 vbox[CL ? REC : 1], rbox[CL ? REC : 1];
    unsigned vto = 0, rto = 0;
    if (CL) {
        for (int q = tid; q < REC; q += 4 * B) vbox[CL ? q : 0] = rbox[CL ? q : 0] = 0;
        vto = cluster_addr(vbox, min(t + 1, (int)gridDim.x - 1));
        rto = cluster_addr(rbox, max(t - 1, 0));
        __syncwarp();
        cluster_sync();
    }
    auto put_v = [&](int q, T x, unsigned seq) {
        if (CL) put_cluster(vto + 8 * kWords<T> * q, x, seq); else put(vout + q * kWords<T>, x, seq);
    };
    auto put_r = [&](int q, T x, unsigned seq) {
        if (CL) put_cluster(rto + 8 * kWords<T> * q, x, seq); else put(rout + q * kWords<T>, x, seq);
    };
    auto get_v = [&](int q, unsigned seq, T &x) {
        return CL ? get_own(vbox + q * kWords<T>, seq, x, a.spin_limit, a.status) : get(vin + q * kWords<T>, seq, x, a.spin_limit, a.status);
    };
    auto get_r = [&](int q, unsigned seq, T &x) {
        return CL ? get_own(rbox + q * kWords<T>, seq, x, a.spin_limit, a.status) : get(rin + q * kWords<T>, seq, x, a.spin_limit, a.status);
    };

    if (t == 0)  // defined values should a wait run out below
        for (int q = tid; q < n; q += 4 * B) {
            dout[q] = (q == 0) ? (double)band[0] : 0.0;
            if (q + 1 < n) eout[q] = 0.0;
        }
    if (tid == 0) failed = *(volatile int *)(a.status + ST_CODE) != 0;

    // ---- windows of sweep 0
    T X[CPT], D[CPT], x0 = T(0);
    {
        const int r = 1 + t * B, rs = r % B;
        const int gi = r + (i - rs + B) % B;
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int c = c0 + q, gj = r + (c - rs + B) % B, gc = gj - B;
            const int lo = min(gi, gj), hi = max(gi, gj);
            D[q] = (hi < n) ? band[(size_t)(hi - lo) + (size_t)lo * ldb] : T(0);
            X[q] = (t > 0 && gi < n) ? band[(size_t)(gi - gc) + (size_t)gc * ldb] : T(0);
        }
        if (t == 0 && gi < n) x0 = band[gi];  // column 0, rows 1 .. B
    }
    __syncthreads();
    const bool off = failed || t >= a.S;

    int rs = 1 % B;      // slot of the first row (and, for t > 0, of the first column of X)
    for (int j = 0; j < nsweep && !off; ++j) {
        const int r = j + 1 + t * B;
        if (r > n - 1) break;
        const int par = j & 1;
        const int pr = rs == 0 ? B - 1 : rs - 1;           // slot that leaves / enters
        const bool have_row = j > 0 && r - 1 + B <= n - 1;  // position t + 1 had a step in sweep j - 1
        const bool have_next = r + B <= n - 1;              // position t + 1 has one in this sweep
        // ---- the window moves, the part that needs no message: the column that leaves D enters X
        if (j > 0) {
            if (t == 0) x0 = __shfl_sync(0xffffffffu, pick(D, pr % CPT), quad | (pr / CPT));
            if (i != pr && part == pr / CPT)
#pragma unroll
                for (int q = 0; q < CPT; ++q) move_if(X[q], D[q], pr % CPT, q);
        }
        // ---- what this step waits for
        {
            bool ok = true;
            if (tid < B) {
                T v = T(0);
                if (t > 0) ok = get_v(tid, (unsigned)j + 1, v);
                vps[par][tid] = v;
            } else if (tid < 2 * B) {
                const int c = tid - B;
                T v = T(0);
                if (have_row) ok = get_r(c, (unsigned)j, v);
                rows_[par][c] = v;
            } else if (tid == 2 * B) {
                T v = T(0);
                if (t > 0) ok = get_v(B, (unsigned)j + 1, v);
                msc[par][0] = v;
            } else if (tid == 2 * B + 32) {
                T v = T(0);
                if (have_row) ok = get_r(B, (unsigned)j, v);
                msc[par][1] = v;
            }
            if (!ok) failed = 1;
        }
        __syncthreads();
        if (failed) break;
        // ---- slot pr takes the new row and column
        if (j > 0) {
            if (i == pr) {
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
                    const int c = c0 + q;
                    X[q] = (c == pr) ? rows_[par][c] : T(0);
                    D[q] = (c == pr) ? msc[par][1] : rows_[par][c];
                }
                x0 = rows_[par][pr];
            } else if (part == pr / CPT) {
                const T ri = rows_[par][i];
#pragma unroll
                for (int q = 0; q < CPT; ++q) move_if(D[q], ri, pr % CPT, q);
            }
        }
        // ---- y, x and the partial sums over rows
        const bool first = i == rs;
        T y = T(0), x = x0;
        if (t > 0) {
            T y1 = T(0);
#pragma unroll
            for (int q = 0; q < CPT; q += 2) {
                y = fma(X[q], vps[par][c0 + q], y);
                y1 = fma(X[q + 1], vps[par][c0 + q + 1], y1);
            }
            y += y1;
            y += __shfl_xor_sync(0xffffffffu, y, 1);
            y += __shfl_xor_sync(0xffffffffu, y, 2);
            y *= msc[par][0];
            x = __shfl_sync(0xffffffffu, pick(X, rs % CPT), quad | (rs / CPT)) - y;
        }
        const T xz = first ? T(0) : x;
        if (part == 0) {
            xs[i] = xz;
            if (first) { ysl[0] = x; ysl[1] = y; }
        }
        auto column_sums = [&]() {
            T xp = xz;
            if (!EARLY) pin(xp);  // after the reflector is on its way
            // column sums of xz X0 over the warp's eight rows: exchange halves so that each
            // lane ends with PH columns
            T u[CPT];
#pragma unroll
            for (int q = 0; q < CPT; ++q) u[q] = xp * X[q];
            if (first)
#pragma unroll
                for (int q = 0; q < CPT; ++q) xrow[c0 + q] = X[q];
            int base = 0;
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const int o = 16 >> s;
                const int half = CPT >> (s + 1);
                const bool up = (lane & o) != 0;
#pragma unroll
                for (int q = 0; q < half; ++q) {
                    const T keep = up ? u[q + half] : u[q], give = up ? u[q] : u[q + half];
                    u[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                }
                base += up ? half : 0;
            }
#pragma unroll
            for (int q = 0; q < PH; ++q) upart[warp][c0 + base + q] = u[q];
        };
        if (t > 0 && EARLY) column_sums();
        {
            const T ss = xz * xz, xy = xz * y;
            // |xz|^2 in the lanes of the lower half, xz . y in the upper half
            const T keep = (lane & 16) ? xy : ss, give = (lane & 16) ? ss : xy;
            T r2 = keep + __shfl_xor_sync(0xffffffffu, give, 16);
            r2 += __shfl_xor_sync(0xffffffffu, r2, 8);
            r2 += __shfl_xor_sync(0xffffffffu, r2, 4);
            if ((lane & 15) == 0) red[lane >> 4][warp] = r2;
        }
        __syncthreads();
        // ---- the reflector (every thread computes the same scalars) and q = tau D v
        const T alpha = ysl[0];
        T ss = red[0][0], xy = red[1][0];
#pragma unroll
        for (int w = 1; w < NW; ++w) { ss += red[0][w]; xy += red[1][w]; }
        T beta, tau, scl;
        reflector<T>(alpha, ss, beta, tau, scl);
        const T v = first ? T(1) : xz * scl;
        if (part == 0) {
            if (have_next) put_v(i, v, (unsigned)j + 1);
            if (i == 0 && have_next) put_v(B, tau, (unsigned)j + 1);
            vs[i] = v;
        } else if (part == 1) {
            const size_t slot = (size_t)j * a.S + t;
            v2[slot * B + (i >= rs ? i - rs : i - rs + B)] = v;
            if (i == 0) tau2[slot] = tau;
        }
        auto form_p = [&]() {
            if (tid < B) {
                T s = upart[0][tid];
#pragma unroll
                for (int w = 1; w < NW; ++w) s += upart[w][tid];
                ps[tid] = tau * (fma(scl, s, xrow[tid]) - fma(scl, xy, ysl[1]) * vps[par][tid]);
            }
        };
        if (t > 0 && !EARLY) column_sums();
        T qd;
        {
            T g = T(0), g1 = T(0);
#pragma unroll
            for (int q = 0; q < CPT; q += 2) {
                g = fma(D[q], xs[c0 + q], g);
                g1 = fma(D[q + 1], xs[c0 + q + 1], g1);
            }
            g += g1;
            g += __shfl_xor_sync(0xffffffffu, g, 1);
            g += __shfl_xor_sync(0xffffffffu, g, 2);
            const T dc = __shfl_sync(0xffffffffu, pick(D, rs % CPT), quad | (rs / CPT));
            qd = tau * fma(scl, g, dc);
        }
        if (t > 0 && EARLY) form_p();
        if (part == 0) qs[i] = qd;
        {
            T kp = v * qd;
#pragma unroll
            for (int o = 16; o >= 4; o >>= 1) kp += __shfl_xor_sync(0xffffffffu, kp, o);
            if (lane == 0) red[2][warp] = kp;
        }
        __syncthreads();
        T K = red[2][0];
#pragma unroll
        for (int w = 1; w < NW; ++w) K += red[2][w];
        // D - v w^T - w v^T with w = q - K v / 2, as D - v q^T - (q - K v) v^T
        T vd = v, w2 = fma(-K * tau, v, qd);
        if (t > 0) {
            if (!EARLY) {
                form_p();
                __syncthreads();
            }
            // ---- updates: X first, and the row that position t - 1 takes in at its next sweep
#pragma unroll
            for (int q = 0; q < CPT; ++q) {
                const int c = c0 + q;
                X[q] = fma(-v, ps[c], fma(-y, vps[par][c], X[q]));
            }
            if (first) {
#pragma unroll
                for (int q = 0; q < CPT; ++q) {
                    const int c = c0 + q;
                    put_r(c, c == rs ? beta : X[q], (unsigned)j + 1);
                }
                if (part == rs / CPT)
                    put_r(B, fma(-v, qs[rs], fma(-w2, vs[rs], pick(D, rs % CPT))), (unsigned)j + 1);
            }
            pin(vd);
            pin(w2);  // D after the row is on its way
        }
#pragma unroll
        for (int q = 0; q < CPT; ++q) {
            const int c = c0 + q;
            D[q] = fma(-vd, qs[c], fma(-w2, vs[c], D[q]));
        }
        if (t == 0) {
            if (first && part == rs / CPT) {
                dout[j + 1] = (double)pick(D, rs % CPT);
                eout[j] = (double)beta;
            }
            if (j == nsweep - 1 && i == (n - 1) % B) {
                if (part == i / CPT) dout[n - 1] = (double)pick(D, i % CPT);
                if (part == rs / CPT) eout[n - 2] = (double)pick(D, rs % CPT);
            }
        }
        // The next step's packets go to the other buffer of vps, rows_ and msc while slower
        // threads still read this one; every other shared array is written again only after
        // the next step's first barrier.
        rs = rs + 1 == B ? 0 : rs + 1;
    }
    if (CL) {
        __syncwarp();
        cluster_sync();  // nobody stores to the shared memory of a CTA that has ended
    }
}

template <typename T, int B>
cudaError_t launch(cudaStream_t st, int n, const T *band, int ldb, double *d, double *e, T *v2, T *tau2,
                   int *status, unsigned *sync, size_t sync_words, int num_sms)
{
    const int S = sb2st_steps(n, B);
    Args a;
    a.n = n; a.ldb = ldb; a.S = S; a.status = status; a.spin_limit = spin_limit();
    a.vmsg = reinterpret_cast<u64 *>(sync + 64);
    a.rmsg = a.vmsg;
    void *args[] = {&band, &v2, &tau2, &d, &e, &a};
    cudaError_t err;
    // Up to 16 positions (the largest cluster): every hand-over is a store to another SM's shared memory
    // instead of a store to and a load from L2. One pair that goes through L2 would set the pace of all.
    if (S <= 16) {
        auto *kernel = chase_resident_kernel<T, B, true>;
        static PerDeviceOnce attr;  // per instantiation
        err = once_per_device(attr, [&] {
            return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        });
        if (err != cudaSuccess) return err;
        unsigned size = 1;
        while ((int)size < S) size *= 2;
        cudaLaunchAttribute dim[1];
        dim[0].id = cudaLaunchAttributeClusterDimension;
        dim[0].val.clusterDim.x = size;
        dim[0].val.clusterDim.y = dim[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(size);
        cfg.blockDim = dim3(4 * B);
        cfg.stream = st;
        cfg.attrs = dim;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0) {
            EGB_COUNT_LAUNCH();
            return cudaLaunchKernelExC(&cfg, (void *)kernel, args);
        }
        cudaGetLastError();
    }
    int per_sm = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, chase_resident_kernel<T, B, false>, 4 * B, 0);
    if (err != cudaSuccess) return err;
    const size_t words = (size_t)S * kWords<T> * (B + 2);
    if (S > per_sm * num_sms || 64 + 4 * words > sync_words) return cudaErrorNotSupported;
    a.rmsg = a.vmsg + words;
    if ((err = cudaMemsetAsync(a.vmsg, 0, 2 * words * sizeof(u64), st)) != cudaSuccess) return err;
    EGB_COUNT_LAUNCH();
    return cudaLaunchCooperativeKernel((void *)chase_resident_kernel<T, B, false>, dim3(S), dim3(4 * B), args, 0, st);
}

}  // namespace sys

template <typename T>
cudaError_t chase_resident(cudaStream_t st, int n, int b, const T *band, int ldb, double *d, double *e,
                           T *v2, T *tau2, int *status, unsigned *sync, size_t sync_words, int num_sms)
{
    if (n < 3) return cudaErrorNotSupported;
    if (b == 64) return sys::launch<T, 64>(st, n, band, ldb, d, e, v2, tau2, status, sync, sync_words, num_sms);
    if (b == 32) return sys::launch<T, 32>(st, n, band, ldb, d, e, v2, tau2, status, sync, sync_words, num_sms);
    return cudaErrorNotSupported;
}
template cudaError_t chase_resident<double>(cudaStream_t, int, int, const double *, int, double *, double *,
                                            double *, double *, int *, unsigned *, size_t, int);
template cudaError_t chase_resident<float>(cudaStream_t, int, int, const float *, int, double *, double *,
                                           float *, float *, int *, unsigned *, size_t, int);

}  // namespace egb
