// Values handed from one CTA to another of the same launch through global memory (L2): each
// 64-bit word carries 32 bits of a value and, above them, a sequence number that is never 0
// and is used once per word and launch. The reader polls the word itself, so a hand-over is
// one store and one load: no fence, no separate flag. A binary64 value (or a pair of
// binary32 values) is two words. The words are zeroed before they are used.
#pragma once

#include "common.cuh"

namespace egb {
namespace pkt {

typedef unsigned long long u64;

template <typename T> constexpr int kWords = (int)(sizeof(T) / 4);  // words per value

__device__ __forceinline__ void st_relaxed(u64 *p, u64 v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ u64 ld_relaxed(const u64 *p)
{
    u64 v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ u64 word(unsigned v, unsigned seq) { return ((u64)seq << 32) | v; }
__device__ __forceinline__ unsigned seq_of(u64 w) { return (unsigned)(w >> 32); }

__device__ __forceinline__ void put(u64 *p, float v, unsigned seq) { st_relaxed(p, word(__float_as_uint(v), seq)); }
__device__ __forceinline__ void put(u64 *p, double v, unsigned seq)
{
    st_relaxed(p, word((unsigned)__double2loint(v), seq));
    st_relaxed(p + 1, word((unsigned)__double2hiint(v), seq));
}
__device__ __forceinline__ bool try_get(const u64 *p, unsigned seq, float &v)
{
    const u64 a = ld_relaxed(p);
    v = __uint_as_float((unsigned)a);
    return seq_of(a) == seq;
}
__device__ __forceinline__ bool try_get(const u64 *p, unsigned seq, double &v)
{
    const u64 a = ld_relaxed(p), b = ld_relaxed(p + 1);
    v = __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
    return seq_of(a) == seq && seq_of(b) == seq;
}

// One failed poll: counts it, false when the wait has to be given up (the limit is reached,
// which is recorded, or another CTA has recorded an error).
__device__ __forceinline__ bool poll_again(long long &it, long long limit, int *status, int aux)
{
    if (++it > limit) {
        report_error(status, ELSI_ERR_TIMEOUT, aux);
        return false;
    }
    return (it & 255) != 0 || *(volatile int *)(status + ST_CODE) == 0;
}

// Bounded wait for a value.
template <typename T>
__device__ __forceinline__ bool get(const u64 *p, unsigned seq, T &v, long long limit, int *status)
{
    long long it = 0;
    while (!try_get(p, seq, v))
        if (!poll_again(it, limit, status, (int)seq)) return false;
    return true;
}

// The same between the CTAs of a cluster: the words are in the reader's shared memory, the writer
// stores to them there (cluster_addr: a shared-memory address of the CTA with this rank).
__device__ __forceinline__ unsigned cluster_addr(const void *p, int rank)
{
    unsigned r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_cluster(unsigned p, u64 v)
{
    asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(p), "l"(v) : "memory");
}
__device__ __forceinline__ u64 ld_own(const u64 *p)
{
    u64 v;
    asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"((unsigned)__cvta_generic_to_shared(p)) : "memory");
    return v;
}
__device__ __forceinline__ void put_cluster(unsigned p, float v, unsigned seq) { st_cluster(p, word(__float_as_uint(v), seq)); }
__device__ __forceinline__ void put_cluster(unsigned p, double v, unsigned seq)
{
    st_cluster(p, word((unsigned)__double2loint(v), seq));
    st_cluster(p + 8, word((unsigned)__double2hiint(v), seq));
}
__device__ __forceinline__ bool try_get_own(const u64 *p, unsigned seq, float &v)
{
    const u64 a = ld_own(p);
    v = __uint_as_float((unsigned)a);
    return seq_of(a) == seq;
}
__device__ __forceinline__ bool try_get_own(const u64 *p, unsigned seq, double &v)
{
    const u64 a = ld_own(p), b = ld_own(p + 1);
    v = __hiloint2double((int)(unsigned)b, (int)(unsigned)a);
    return seq_of(a) == seq && seq_of(b) == seq;
}
template <typename T>
__device__ __forceinline__ bool get_own(const u64 *p, unsigned seq, T &v, long long limit, int *status)
{
    long long it = 0;
    while (!try_get_own(p, seq, v))
        if (!poll_again(it, limit, status, (int)seq)) return false;
    return true;
}

}  // namespace pkt

// 1 / x and 1 / sqrt(x), within 1 and 1.25 ulp: the hardware's approximation r (about 2^-20 in
// binary64) and one of Householder's iterations (A. S. Householder, The Numerical Treatment of
// a Single Nonlinear Equation, 1970), that of third order in binary64 (two of second order are
// a longer chain), Newton's in binary32. With h = 1 - x r the value is r / (1 - h) = r (1 + h + h^2 +
// ..), with h = 1 - x r^2 it is r (1 - h)^(-1/2) = r (1 + h / 2 + 3 h^2 / 8 + ..), cut after h^2. A
// library division or square root is two to three times as long a chain, and in binary64 two
// to three times as many operations of the chip's few binary64 units. Arguments whose result
// or whose approximation would be subnormal or overflow take the library's path, or in binary32
// square roots a scaled argument.
__device__ __forceinline__ double recip(double x)
{
    const int ex = __double2hiint(x) & 0x7FF00000;
    if (ex >= (2044 << 20) || ex == 0) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double h = fma(-x, r, 1.0);  // r (1 + h + h^2): a relative error of h^3
    return fma(r, fma(h, h, h), r);
}
__device__ __forceinline__ float recip(float x)
{
    const float a = fabsf(x);
    if (!(a > 1e-36f && a < 1e36f)) return 1.0f / x;
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(fmaf(-x, r, 1.0f), r, r);
}
__device__ __forceinline__ double rsq(double x)
{
    const int ex = __double2hiint(x) & 0x7FF00000;
    if (ex >= (2000 << 20) || ex <= (40 << 20)) return rsqrt(x);
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    const double h = fma(-x * r, r, 1.0);  // r (1 + h / 2 + 3 h^2 / 8): a relative error of 5 h^3 / 16
    return fma(h * r, fma(0.375, h, 0.5), r);
}
__device__ __forceinline__ float rsq_step(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return fmaf(0.5f * r, fmaf(-x * r, r, 1.0f), r);
}
__device__ __forceinline__ float rsq(float x)
{
    if (x > 1e-36f && x < 1e36f) return rsq_step(x);
    // (a square root and a division are two roundings, up to 1.5 ulp)
    if (x > 0.0f && x <= 1e-36f) return 0x1p32f * rsq_step(0x1p64f * x);
    if (x >= 1e36f && x < INFINITY) return 0x1p-32f * rsq_step(0x1p-64f * x);
    return 1.0f / sqrtf(x);
}

// Householder scalars of x = (alpha, tail) with |tail|^2 = ss: v = (1, scl tail), H = I - tau
// v v^T, H x = beta e_1.
template <typename T>
__device__ __forceinline__ void reflector(T alpha, T ss, T &beta, T &tau, T &scl)
{
    beta = alpha;
    tau = scl = T(0);
    if (ss != T(0)) {
        const T s2 = fma(alpha, alpha, ss), rn = rsq(s2), nrm = s2 * rn;
        beta = (alpha >= T(0)) ? -nrm : nrm;
        tau = fma(fabs(alpha), rn, T(1));  // (beta - alpha) / beta
        scl = recip(alpha - beta);
    }
}

// v = a where q == k: a predicated move that the compiler cannot turn into an indexed access
// (which would put the array that a comes from into local memory).
__device__ __forceinline__ void move_if(float &v, float a, int q, int k)
{
    asm("{\n .reg .pred p;\n setp.eq.s32 p, %2, %3;\n @p mov.b32 %0, %1;\n}\n" : "+f"(v) : "f"(a), "r"(q), "r"(k));
}
__device__ __forceinline__ void move_if(double &v, double a, int q, int k)
{
    asm("{\n .reg .pred p;\n setp.eq.s32 p, %2, %3;\n @p mov.b64 %0, %1;\n}\n" : "+d"(v) : "d"(a), "r"(q), "r"(k));
}

// a[q] for a run-time q without indexing registers
template <typename T, int N>
__device__ __forceinline__ T pick(const T (&a)[N], int q)
{
    T v = a[0];
#pragma unroll
    for (int k = 1; k < N; ++k) move_if(v, a[k], q, k);
    return v;
}

}  // namespace egb
