// QR factorisation of one panel (m x bw, bw <= 64) of the full -> band reduction: Householder
// reflectors column by column and the compact-WY factor T (Q = I - V T V^T).
//
// What bounds it: bw columns one after the other, each with a sum over all rows between the
// column and the update, so the time is bw times the latency of one all-to-all exchange plus
// the arithmetic of the CTA with the most rows. With the panel in shared memory, a grid
// barrier per column and the partial sums read after it, a column took 12.5 us in binary32
// and 18 us in binary64.
//
// Layout: lane l of warp w holds columns l and l + 32 of RW consecutive rows in registers for
// the whole factorisation, so the column sums and the rank-1 update need no exchange between
// lanes; the current column reaches the other lanes through one broadcast from shared memory.
// A CTA publishes its 64 column sums as packets (packets.cuh) and every CTA polls the packets
// of all others directly: one store and one load through L2 per column, no barrier between
// CTAs. The sums x_j . P_c over the rows below j serve three uses at once: c = j is the
// column's squared norm, c > j gives the update and c < j, where the storage already holds
// the reflectors, the Gram column for T. T itself is formed by one extra CTA that reads the
// same packets and is never waited for.
//
// Sums over CTAs are kept to more than the panel's precision: binary32 partial sums are added
// with their rounding errors (Knuth's two-sum), since binary64 additions are scarce here, and
// stay a pair of binary32 numbers up to the one rounding of the update's factors; T is formed from
// the pairs in binary64.
//
// T is off the row CTAs' path only while its CTA keeps up: with a Gram entry converted to binary64
// for every row of T it was the slower one (full to band of n = 16384 173 ms, 164 with one conversion
// an entry and column; whole solves of n = 4096 76.3 -> 72.6 ms).
//
// Measured per 64-column panel, before -> now: binary32 n = 777 0.73 -> 0.21 ms, n = 4096 0.82
// -> 0.24 ms, n = 16384 0.85 -> 0.29 ms; binary64 n = 512 1.09 -> 0.40 ms, n = 5000 1.24 ->
// 0.51 ms; per 32-column panel, binary64 n = 512 0.152 -> 0.133 ms, n = 5000 0.192 -> 0.169 ms with
// the late scale, the row fetched with the sums and the shorter reciprocals of packets.cuh. What is left is one L2 exchange a column (about 1.5 us) and, in binary64, the
// 2 x 64 x 64 FMAs of a CTA's rows at two a clock.
#include "common.cuh"
#include "kernels.h"
#include "packets.cuh"

namespace egb {
namespace pan {

using namespace pkt;

struct Args {
    int m, bw, lda, ldv, G, gs;  // G row CTAs (one more forms T); gs >= G the packet stride
    unsigned seq0;               // the packets of column j carry seq0 + j + 1
    u64 *dpk;                    // [64][gs][64][2]: column sums
    u64 *rpk;                    // [64][64][2]: row j of the panel
    int *status;
    long long spin_limit;
};

// A sum with at least the precision of binary64 accumulation of binary32 terms, or a plain
// binary64 one; two packet words either way.
template <typename T> struct Sum;
template <> struct Sum<double> {
    double v = 0.0;
    __device__ __forceinline__ void add(double x) { v += x; }
    __device__ __forceinline__ void add(const Sum &o) { v += o.v; }
    __device__ __forceinline__ double value() const { return v; }
    __device__ __forceinline__ double low() const { return 0.0; }
    __device__ __forceinline__ unsigned w0() const { return (unsigned)__double2loint(v); }
    __device__ __forceinline__ unsigned w1() const { return (unsigned)__double2hiint(v); }
    __device__ __forceinline__ static Sum from(unsigned a, unsigned b) { Sum s; s.v = __hiloint2double((int)b, (int)a); return s; }
    __device__ __forceinline__ Sum other(int o) const { Sum s; s.v = __shfl_xor_sync(0xffffffffu, v, o); return s; }
};
template <> struct Sum<float> {
    float h = 0.f, l = 0.f;
    __device__ __forceinline__ void add(float x)
    {
        const float s = h + x, b = s - h;
        l += (h - (s - b)) + (x - b);
        h = s;
    }
    __device__ __forceinline__ void add(const Sum &o) { add(o.h); l += o.l; }
    __device__ __forceinline__ float value() const { return h + l; }
    __device__ __forceinline__ float low() const { return l - ((h + l) - h); }  // of value() + low()
    __device__ __forceinline__ unsigned w0() const { return __float_as_uint(h); }
    __device__ __forceinline__ unsigned w1() const { return __float_as_uint(l); }
    __device__ __forceinline__ static Sum from(unsigned a, unsigned b) { Sum s; s.h = __uint_as_float(a); s.l = __uint_as_float(b); return s; }
    __device__ __forceinline__ Sum other(int o) const
    {
        Sum s;
        s.h = __shfl_xor_sync(0xffffffffu, h, o);
        s.l = __shfl_xor_sync(0xffffffffu, l, o);
        return s;
    }
};

// tau (row + scl (d + dl)), rounded once: the products split by an FMA, the sum by two-sum
__device__ __forceinline__ float update_factor(float tau, float scl, float row, float d, float dl)
{
    const float p = __fmul_rn(scl, d), s = __fadd_rn(row, p), b = __fadd_rn(s, -row);
    const float t = __fadd_rn(__fadd_rn(row, -__fadd_rn(s, -b)), __fadd_rn(p, -b));
    const float low = fmaf(scl, dl, t + fmaf(scl, d, -p));
    const float h = __fadd_rn(s, low), l = __fadd_rn(low, -__fadd_rn(h, -s));
    const float q = __fmul_rn(tau, h);
    return q + fmaf(tau, l, fmaf(tau, h, -q));
}
__device__ __forceinline__ double update_factor(double tau, double scl, double row, double d, double)
{
    return tau * fma(scl, d, row);
}

__device__ __forceinline__ void ld2_relaxed(const u64 *p, u64 &a, u64 &b)
{
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// RW rows per warp, CPL columns per lane (bw <= 32 CPL), NW warps.
template <typename T, int RW, int CPL, int NW>
constexpr size_t smem_bytes()
{
    const size_t tile = (size_t)NW * 32 * CPL * (RW + 1) * sizeof(T);
    const size_t tm = (size_t)64 * 65 * sizeof(double);
    return tile > tm ? tile : tm;
}

template <typename T, int RW, int CPL, int NW>
__global__ void __launch_bounds__(32 * NW, 512 / (32 * NW))
panel_kernel(T *P, T *V, T *Tm, int ldt, const Args a)
{
    constexpr int NC = 32 * CPL;       // columns held (zero beyond bw)
    constexpr int LPC = 32 * NW / NC;  // threads per column in the exchange
    constexpr int RPL = 32 / RW;       // columns of a warp's rows moved by one access
    constexpr int FLY = 8;             // packets of a thread in flight
    // binary64: the storage holds x, scaled to the reflector at the end (binary32 would lose sums of
    // two columns of 1e-16 and less)
    constexpr bool LATE = sizeof(T) == 8;
    static_assert(LPC >= 4 && LPC <= 16 && NW % LPC == 0 && RW <= 32 && RW * NW >= NC, "layout");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(16) T xbuf[NW][RW];
    __shared__ T partw[NW][NC];
    __shared__ T rowown[NC], dsum[NC], dlow[sizeof(T) == 4 ? NC : 1], rowj[NC], scal[3], scls[NC];  // scls: 1 / x scale of column c's reflector
    __shared__ double gram[NC];  // CTA G: v_c . v_j
    __shared__ int failed;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = blockIdx.x, G = a.G, bw = a.bw;
    const int row0 = (g * NW + warp) * RW;  // first row of the warp
    T *tile = reinterpret_cast<T *>(smem_raw) + (size_t)warp * NC * (RW + 1);
    double(*Ts)[65] = reinterpret_cast<double(*)[65]>(smem_raw);  // CTA G
    const int nref = min(bw, a.m);
    const int rl = lane % RW, cl = lane / RW;  // row and column of a lane in the copies

    T p[CPL][RW];
    if (tid == 0) failed = 0;
    if (g < G) {
#pragma unroll 8
        for (int c = cl; c < NC; c += RPL)
            tile[c * (RW + 1) + rl] =
                (row0 + rl < a.m && c < bw) ? P[(size_t)(row0 + rl) + (size_t)c * a.lda] : T(0);
        __syncwarp();
#pragma unroll
        for (int h = 0; h < CPL; ++h)
#pragma unroll
            for (int i = 0; i < RW; ++i) p[h][i] = tile[(h * 32 + lane) * (RW + 1) + i];
    } else {
        for (int e = tid; e < 64 * 65; e += 32 * NW) Ts[0][e] = 0.0;
    }
    __syncthreads();

    const int xc = tid / LPC, xg = tid % LPC;  // column and share of this thread in the exchange
    for (int j = 0; j < nref; ++j) {
        const unsigned seq = a.seq0 + (unsigned)j + 1;
        Sum<T> tot;
        if (g < G) {
            // ---- column sums of x P over the rows below j
            __syncwarp();
#pragma unroll
            for (int i = 0; i < RW; ++i) {
                T x = p[0][i];
                if (CPL == 2 && j >= 32) x = p[CPL - 1][i];
                if (lane == (j & 31)) xbuf[warp][i] = (row0 + i > j) ? x : T(0);
            }
            __syncwarp();
            T s[CPL][2] = {};
#pragma unroll
            for (int i = 0; i < RW; i += 2)
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    s[c][0] = fma(xbuf[warp][i], p[c][i], s[c][0]);
                    s[c][1] = fma(xbuf[warp][i + 1], p[c][i + 1], s[c][1]);
                }
#pragma unroll
            for (int c = 0; c < CPL; ++c) partw[warp][c * 32 + lane] = s[c][0] + s[c][1];
            if (g == 0 && warp == j / RW)
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    const T x = pick(p[c], j % RW);
                    rowown[c * 32 + lane] = x;
                    put(a.rpk + (size_t)(j * 64 + c * 32 + lane) * 2, x, seq);
                }
            __syncthreads();
            Sum<T> sm;
#pragma unroll
            for (int w = 0; w < NW / LPC; ++w) sm.add(partw[xg * (NW / LPC) + w][xc]);
#pragma unroll
            for (int o = 1; o < LPC; o <<= 1) sm.add(sm.other(o));
            if (xg == 0) {
                u64 *d = a.dpk + ((size_t)(j * a.gs + g) * 64 + xc) * 2;
                st_relaxed(d, word(sm.w0(), seq));
                st_relaxed(d + 1, word(sm.w1(), seq));
            }
            tot = sm;
        }
        // ---- the sums of all CTAs, and row j
        bool ok = true;
        T row = T(0);
        if (G > 1 || g == G) {
            tot = Sum<T>();
            // row j comes with the first of them (the loads are in flight together)
            bool have_row = g == 0 || xg != 0;
            for (int q0 = xg; q0 < G && ok; q0 += LPC * FLY) {
                u64 w0[FLY], w1[FLY], wr[2];
                long long it = 0;
                for (;;) {
                    bool ready = true;
                    const u64 *rp = a.rpk + (size_t)(j * 64 + xc) * 2;
                    if (!have_row) {
                        wr[0] = ld_relaxed(rp);
                        if (sizeof(T) == 8) wr[1] = ld_relaxed(rp + 1);
                    }
#pragma unroll
                    for (int u = 0; u < FLY; ++u) {
                        const int q = q0 + LPC * u;
                        if (q < G) ld2_relaxed(a.dpk + ((size_t)(j * a.gs + q) * 64 + xc) * 2, w0[u], w1[u]);
                    }
#pragma unroll
                    for (int u = 0; u < FLY; ++u)
                        if (q0 + LPC * u < G) ready = ready && seq_of(w0[u]) == seq && seq_of(w1[u]) == seq;
                    if (!have_row) {
                        have_row = seq_of(wr[0]) == seq && (sizeof(T) == 4 || seq_of(wr[1]) == seq);
                        if (sizeof(T) == 4) row = (T)__uint_as_float((unsigned)wr[0]);
                        else row = (T)__hiloint2double((int)(unsigned)wr[1], (int)(unsigned)wr[0]);
                    }
                    if (ready && have_row) break;
                    if (!poll_again(it, a.spin_limit, a.status, j)) { ok = false; break; }
                }
#pragma unroll
                for (int u = 0; u < FLY; ++u)
                    if (ok && q0 + LPC * u < G) tot.add(Sum<T>::from((unsigned)w0[u], (unsigned)w1[u]));
            }
            __syncwarp();
#pragma unroll
            for (int o = 1; o < LPC; o <<= 1) tot.add(tot.other(o));
        }
        if (xg == 0) {
            if (g == 0) row = rowown[xc];
            const T d = tot.value();
            dsum[xc] = d;
            if (sizeof(T) == 4) dlow[sizeof(T) == 4 ? xc : 0] = tot.low();
            rowj[xc] = row;
            if (xc == j) {
                T beta, tau, scl;
                reflector<T>(row, d, beta, tau, scl);
                scal[0] = beta; scal[1] = tau; scal[2] = scls[j] = scl;
            }
        }
        if (!ok) failed = 1;
        __syncthreads();
        if (failed) return;
        const T beta = scal[0], tau = scal[1], scl = scal[2];
        if (g < G) {
            // ---- P_c -= v (tau v . P_c), c > j, v = scl x; column j becomes the reflector (binary64: at
            //      the end, LATE; the scale would be as many operations as the products)
            T wv[CPL];
#pragma unroll
            for (int c = 0; c < CPL; ++c) {
                const int col = c * 32 + lane;
                wv[c] = col > j ? update_factor(tau, scl, rowj[col], dsum[col], dlow[sizeof(T) == 4 ? col : 0]) : T(0);
            }
            T wx[CPL];
#pragma unroll
            for (int c = 0; c < CPL; ++c) wx[c] = LATE ? scl * wv[c] : wv[c];
#pragma unroll
            for (int i = 0; i < RW; ++i) {
                const T v = LATE ? xbuf[warp][i] : xbuf[warp][i] * scl;
#pragma unroll
                for (int c = 0; c < CPL; ++c) {
                    p[c][i] = fma(-v, wx[c], p[c][i]);
                    if (!LATE && c * 32 + lane == j && row0 + i > j) p[c][i] = v;
                }
            }
            if (g == 0 && warp == j / RW) {
#pragma unroll
                for (int i = 0; i < RW; ++i)
#pragma unroll
                    for (int c = 0; c < CPL; ++c)
                        move_if(p[c][i], c * 32 + lane == j ? beta : p[c][i] - wv[c], j % RW, i);
            }
        } else {
            // ---- T[0:j, j] = -tau T[0:j, 0:j] (v_c . v_j), forward recurrence
            if (xg == 0) {
                double d = (double)dsum[xc];
                if (sizeof(T) == 4) d += (double)dlow[sizeof(T) == 4 ? xc : 0];
                gram[xc] = ((double)scl * d + (double)rowj[xc]) * (LATE && xc < j ? (double)scls[xc] : 1.0);
            }
            __syncthreads();
            double acc = 0.0;
            if (xc < j)
                for (int q = xc + xg; q < j; q += LPC) acc += Ts[xc][q] * gram[q];
            __syncwarp();
#pragma unroll
            for (int o = 1; o < LPC; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (xg == 0 && xc <= j) Ts[xc][j] = xc < j ? -(double)tau * acc : (double)tau;
            __syncthreads();
        }
    }
    __syncthreads();
    if (g == G) {
        for (int e = tid; e < bw * bw; e += 32 * NW) {
            const int r = e % bw, c = e / bw;
            Tm[(size_t)r + (size_t)c * ldt] = (T)Ts[r][c];
        }
        return;
    }
    // ---- the panel (R on and above the diagonal, reflector tails below) and the explicit V
    //      (unit diagonal, zero above) for the products of the update
#pragma unroll
    for (int h = 0; h < CPL; ++h)
#pragma unroll
        for (int i = 0; i < RW; ++i) tile[(h * 32 + lane) * (RW + 1) + i] = p[h][i];
    __syncwarp();
    const int gi = row0 + rl;
    if (gi < a.m)
#pragma unroll 4
        for (int c = cl; c < bw; c += RPL) {
            T pv = tile[c * (RW + 1) + rl];
            if (LATE && gi > c && c < nref) pv *= scls[c];
            P[(size_t)gi + (size_t)c * a.lda] = pv;
            V[(size_t)gi + (size_t)c * a.ldv] = (c >= nref || gi < c) ? T(0) : (gi == c ? T(1) : pv);
        }
}

template <typename T, int RW, int CPL, int NW>
cudaError_t launch(cudaStream_t st, T *P, T *V, T *Tm, int ldt, Args a, int num_sms, bool *fits)
{
    constexpr size_t smem = smem_bytes<T, RW, CPL, NW>();
    static PerDeviceOnce attr;  // per instantiation
    cudaError_t e = once_per_device(attr, [] {
        return cudaFuncSetAttribute(panel_kernel<T, RW, CPL, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e != cudaSuccess) return e;
    a.G = ceil_div(a.m, RW * NW);
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, panel_kernel<T, RW, CPL, NW>, 32 * NW, smem);
    if (e != cudaSuccess) return e;
    *fits = a.G + 1 <= per_sm * num_sms && a.G <= a.gs;
    if (!*fits) return cudaSuccess;
    void *args[] = {&P, &V, &Tm, &ldt, &a};
    EGB_COUNT_LAUNCH();
    return cudaLaunchCooperativeKernel((void *)panel_kernel<T, RW, CPL, NW>, dim3(a.G + 1), dim3(32 * NW), args, smem, st);
}

template <typename T, int CPL>
cudaError_t choose(cudaStream_t st, T *P, T *V, T *Tm, int ldt, const Args &a, int num_sms)
{
    // Rows per CTA: few while the packets of a column still come in one round (64 / CPL CTAs: the
    // threads of a column with 8 in flight each), since a column is the latency of a warp's
    // instructions over its rows and of one exchange, which more CTAs hardly lengthen up to there.
    // Binary32 128 rows against 256: n = 777 210 -> 190 us a panel, n = 4096 234 -> 224 us; above,
    // 256, and 512 once that gives more than 32 CTAs (n = 16384: 321 us, 335 with 128). Binary64 32
    // rows against 64: n = 1531 141 -> 131 us; n = 5000 188 us against 169 with 64.
    constexpr int kFew = sizeof(T) == 4 ? 128 : 32 * CPL;  // the rows j < bw are all in the first CTA
    bool fits = false;
    cudaError_t e = cudaSuccess;
    if (ceil_div(a.m, kFew) <= 64 / CPL) e = launch<T, kFew / 8, CPL, 8>(st, P, V, Tm, ldt, a, num_sms, &fits);
    if constexpr (sizeof(T) == 4) {
        if (e == cudaSuccess && !fits && a.m <= 32 * 256) e = launch<T, 32, CPL, 8>(st, P, V, Tm, ldt, a, num_sms, &fits);
        if (e == cudaSuccess && !fits) e = launch<T, 32, CPL, 16>(st, P, V, Tm, ldt, a, num_sms, &fits);
    } else {
        if (e == cudaSuccess && !fits) e = launch<T, 8, CPL, 8>(st, P, V, Tm, ldt, a, num_sms, &fits);
        if (e == cudaSuccess && !fits) e = launch<T, 16, CPL, 16>(st, P, V, Tm, ldt, a, num_sms, &fits);
        // one column a lane leaves registers for 512 rows a CTA: 77 312 rows
        if constexpr (CPL == 1)
            if (e == cudaSuccess && !fits) e = launch<T, 32, 1, 16>(st, P, V, Tm, ldt, a, num_sms, &fits);
    }
    if (e != cudaSuccess) return e;
    return fits ? cudaSuccess : cudaErrorInvalidConfiguration;
}

// A panel with more rows than fit with two columns a lane (binary64: 38 656), as two panels of one
// column a lane, the reflectors of the first applied to the columns of the second between them.
// work: 2 x 32 x 32 values.
template <typename T>
cudaError_t in_two(cudaStream_t st, T *P, T *V, int ldv, T *Tm, int ldt, const Args &a, T *work, int num_sms)
{
    constexpr int b1 = 32;
    const int m = a.m, b2 = a.bw - b1, lda = a.lda;
    T *C = P + (size_t)b1 * lda, *V2 = V + (size_t)b1 * ldv, *T2 = Tm + b1 + (size_t)b1 * ldt;
    T *Y = work, *Z = work + b1 * b1;
    cudaError_t e;
    Args s = a;
    s.bw = b1;
    if ((e = choose<T, 1>(st, P, V, Tm, ldt, s, num_sms)) != cudaSuccess) return e;
    // C -= V1 T1^T (V1^T C)
    if ((e = gemm<T>(st, 1, 0, b1, b2, m, T(1), V, ldv, C, lda, T(0), Y, b1)) != cudaSuccess) return e;
    if ((e = gemm<T>(st, 1, 0, b1, b2, b1, T(1), Tm, ldt, Y, b1, T(0), Z, b1)) != cudaSuccess) return e;
    if ((e = gemm<T>(st, 0, 0, m, b2, b1, T(-1), V, ldv, Z, b1, T(1), C, lda)) != cudaSuccess) return e;
    if ((e = cudaMemset2DAsync(V2, sizeof(T) * ldv, 0, sizeof(T) * b1, b2, st)) != cudaSuccess) return e;
    s = a;
    s.m = m - b1;
    s.bw = b2;
    s.seq0 = a.seq0 + b1;
    if ((e = choose<T, 1>(st, C + b1, V2 + b1, T2, ldt, s, num_sms)) != cudaSuccess) return e;
    // T = [T1, -T1 (V1^T V2) T2; 0, T2]
    if ((e = gemm<T>(st, 1, 0, b1, b2, m - b1, T(1), V + b1, ldv, V2 + b1, ldv, T(0), Y, b1)) != cudaSuccess) return e;
    if ((e = gemm<T>(st, 0, 0, b1, b2, b2, T(1), Y, b1, T2, ldt, T(0), Z, b1)) != cudaSuccess) return e;
    if ((e = gemm<T>(st, 0, 0, b1, b2, b1, T(-1), Tm, ldt, Z, b1, T(0), Tm + (size_t)b1 * ldt, ldt)) != cudaSuccess) return e;
    return cudaMemset2DAsync(Tm + b1, sizeof(T) * ldt, 0, sizeof(T) * b2, b1, st);
}

}  // namespace pan

// CTAs of a panel with at most m rows, at most: see choose()
static int max_ctas(int m, int elem)
{
    const int most = ceil_div(m, elem == 4 ? 256 : 64), few = ceil_div(m, elem == 4 ? 128 : 32);
    return few < 64 ? few : (most > 64 ? most : 64);
}

size_t panel_packet_words(int m, int elem) { return (size_t)64 * 64 * 2 * (max_ctas(m, elem) + 1); }

template <typename T>
cudaError_t panel_qr(cudaStream_t st, int m, int m_first, int bw, T *P, int lda, T *V, int ldv, T *Tm, int ldt,
                     unsigned seq0, unsigned long long *packets, T *work, int *status, int num_sms)
{
    if (bw < 1 || bw > 64) return cudaErrorInvalidValue;
    pan::Args a;
    a.m = m; a.bw = bw; a.lda = lda; a.ldv = ldv; a.G = 0;
    a.gs = max_ctas(m_first, sizeof(T));
    a.seq0 = seq0; a.rpk = packets; a.dpk = packets + 64 * 64 * 2;
    a.status = status; a.spin_limit = spin_limit();
    if (bw <= 32) return pan::choose<T, 1>(st, P, V, Tm, ldt, a, num_sms);
    const cudaError_t e = pan::choose<T, 2>(st, P, V, Tm, ldt, a, num_sms);
    return e == cudaErrorInvalidConfiguration && m > 64 ? pan::in_two<T>(st, P, V, ldv, Tm, ldt, a, work, num_sms) : e;
}
template cudaError_t panel_qr<double>(cudaStream_t, int, int, int, double *, int, double *, int, double *, int,
                                      unsigned, unsigned long long *, double *, int *, int);
template cudaError_t panel_qr<float>(cudaStream_t, int, int, int, float *, int, float *, int, float *, int,
                                     unsigned, unsigned long long *, float *, int *, int);

}  // namespace egb

namespace egb {

// Packets, then the 2 x 32 x 32 values of work
template <typename T>
static size_t entry_words(int m) { return panel_packet_words(m, sizeof(T)) + 2 * 32 * 32; }

template <typename T>
static int panel_entry(int m, int b, T *P, int lda, T *V, int ldv, T *Tm, int ldt, int num_sms, void *work,
                       size_t work_words, int *status, void *stream)
{
    if (m < 1 || b < 1 || b > 64 || !P || !V || !Tm || !work || !status || lda < m || ldv < m || ldt < b || num_sms < 1 ||
        (size_t)work % 16 != 0 || work_words < entry_words<T>(m))
        return ELSI_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    unsigned long long *packets = reinterpret_cast<unsigned long long *>(work);
    const size_t words = panel_packet_words(m, sizeof(T));
    cudaError_t e = cudaMemsetAsync(packets, 0, sizeof(unsigned long long) * words, st);
    if (e == cudaSuccess)
        e = panel_qr<T>(st, m, m, b, P, lda, V, ldv, Tm, ldt, 0, packets, reinterpret_cast<T *>(packets + words), status,
                        num_sms < sms ? num_sms : sms);
    return e == cudaSuccess ? ELSI_OK : ELSI_ERR_CUDA;
}

}  // namespace egb

extern "C" size_t elsi_gb_panel_qr_f64_work(int m) { return m < 1 ? 0 : egb::entry_words<double>(m); }
extern "C" size_t elsi_gb_panel_qr_f32_work(int m) { return m < 1 ? 0 : egb::entry_words<float>(m); }

extern "C" int elsi_gb_panel_qr_f64(int m, int b, double *P, int lda, double *V, int ldv, double *T, int ldt,
                                    int num_sms, void *work, size_t work_words, int *status, void *stream)
{
    return egb::panel_entry<double>(m, b, P, lda, V, ldv, T, ldt, num_sms, work, work_words, status, stream);
}

extern "C" int elsi_gb_panel_qr_f32(int m, int b, float *P, int lda, float *V, int ldv, float *T, int ldt,
                                    int num_sms, void *work, size_t work_words, int *status, void *stream)
{
    return egb::panel_entry<float>(m, b, P, lda, V, ldv, T, ldt, num_sms, work, work_words, status, stream);
}

namespace egb {
template <typename T>
__global__ void recip_rsq_kernel(int n, const T *x, T *r, T *s)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = recip(x[i]);
    s[i] = rsq(x[i]);
}
}  // namespace egb

extern "C" int elsi_gb_recip_rsq(int n, int binary64, const void *x, void *r, void *s, void *stream)
{
    if (n < 1 || !x || !r || !s) return ELSI_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    const int grid = egb::ceil_div(n, 256);
    if (binary64) egb::recip_rsq_kernel<double><<<grid, 256, 0, st>>>(n, (const double *)x, (double *)r, (double *)s);
    else egb::recip_rsq_kernel<float><<<grid, 256, 0, st>>>(n, (const float *)x, (float *)r, (float *)s);
    return cudaGetLastError() == cudaSuccess ? ELSI_OK : ELSI_ERR_CUDA;
}
