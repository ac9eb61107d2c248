// Binary64-accurate matrix products on the bf16 tensor cores (Ozaki et al.,
// "Error-free transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59 (2012); the
// integer-digit form).
//
// Every row of A (and column of B) is scaled by a power of two 2^e so that its entries
// lie in [-1/2, 1/2], then cut into D signed 9-bit integer digits:
//     x = 2^e sum_{s=1..D} d_s 2^{-9s} (+ a remainder of at most 2^{-9D-1}),  |d_s| <= 256,
// each digit exactly representable in bf16 (whose significand has 8 bits: every integer up
// to 256). Then
//     (A B)_ij = 2^{e_i + f_j} sum_L 2^{-9L} sum_{s+t=L} (D_s^A D_t^B)_ij
// and every digit product is an exact integer. Levels L = 2..D+1 are kept: D (D + 1) / 2
// products. (Seven-bit digits, which leave the tensor cores more terms before a sum passes
// 2^24, need 7 digits and 28 products for 49 bits; 6 nine-bit digits hold 53 in 21.)
//
// Two forms:
//  * refinement (D <= 6, 128 x 128 tiles): the corrections of the binary32 route, P and W. With
//    D = 6 the dropped part is about 2^-54 of max|A_i.| max|B_.j| per term.
//  * binary64 route (D = 8, 128 x 64 tiles, 128-bit sums): 71 bits below the largest entry and
//    a dropped part of 2^-72. A binary64 FMA chain rounds relative to each product, not to
//    the row's largest entry; on graded operands (the standard form of an ill-conditioned
//    overlap) the 2^-54 form lost four digits of P at lambda_min(S) = 1e-6, this one none.
//
// Exactness. The tensor cores add in binary32, exact below 2^24: a sum over 64 of K and L - 1
// digit pairs stays below 64 (L - 1) 2^16, so levels up to 5 are exact and one of the levels
// 6 to 8 can pass 2^24 only if nearly all its digits are extreme, when it is rounded to a
// multiple of 2 of its own unit. Such sums are drained every 64 terms into integers in
// registers. The last level, and in the refinement form level 6 as well, whose units are
// 2^-45 of the level-2 unit and below, are summed in binary32 over all of K.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace egb {

constexpr int kOzBits = 9;       // bits per digit
constexpr int kOzBM = 128, kOzBN = 128, kOzBK = 16;  // plane padding: rows, K
constexpr int kOzSegK = 32768;  // K per kernel launch (64-bit integer sums: see the shift)

// ------------------------------------------------------------------ splitting
// x is rounded (half to even) to the integer N = x 2^{9D - e}, |N| < 2^{9D-1}, in two's complement, and
// N plus 256 in every digit but the first is read nine bits at a time: a field u is the digit
// u - 256, the first digit is what remains. All on the bit pattern, with one shift of the whole
// number and a few 32-bit operations a digit (binary64 arithmetic is scarce on this chip, and
// rounding the number anew for every digit took 64-bit shifts that cost twice the memory traffic).
// A prefix of the digits is within (1/2 + 1/511) of its last unit of x. All splits
// along memory, n = 1531 1.18 -> 0.86 ms, n = 5000 (the trailing blocks) 26 -> 14 ms, refinement of
// n = 16384 11.6 -> 7.3 ms.

// M / 2^k rounded to nearest, ties to even (M < 2^53, k >= 0).
__device__ __forceinline__ unsigned long long rne_shift(unsigned long long M, int k)
{
    if (k == 0) return M;
    if (k > 63) return 0ull;  // M < 2^53 < 2^(k-1): below one half
    unsigned long long q = M >> k;
    const unsigned long long rem = M & ((1ull << k) - 1ull), half = 1ull << (k - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
    return q;
}

__device__ __forceinline__ unsigned long long magnitude(double x)
{
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// The row exponent from the largest magnitude bit pattern: max |x| = m 2^e, m in [0.25, 0.5). A
// vector with an infinity or a NaN has kOzNonFinite, and all its digits are zero: the product forms
// its row or column from the operands instead (see direct_sum).
constexpr int kOzNonFinite = 1 << 28;
__device__ __forceinline__ int row_exponent(unsigned long long mb)
{
    if (mb == 0ull) return 0;
    // (the field alone: the compiler may take the magnitude by arithmetic, which makes a NaN negative)
    if (((mb >> 52) & 0x7FFull) == 0x7FFull) return kOzNonFinite;
    const int xf = (int)(mb >> 52);
    return 1 + (xf ? xf - 1022 : (64 - __clzll((long long)(mb & 0xFFFFFFFFFFFFFull))) - 1074);
}

// d[s - 1] = the binary32 bits of digit s of x under the row exponent e, s = 1..ND (exact, and
// exact in their upper half, bf16)
template <int ND>
__device__ __forceinline__ void digits_of(double x, int e, unsigned (&d)[ND])
{
    constexpr int P = kOzBits * ND;
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int xf = (int)((u >> 52) & 0x7FF);
    const unsigned long long M = xf ? ((u & 0xFFFFFFFFFFFFFull) | (1ull << 52)) : (u & 0xFFFFFFFFFFFFFull);
    const int sh = P - e + (xf ? xf - 1075 : -1074);  // N = x 2^(P - e) = M 2^sh, at most P - 1 bits
    unsigned long long lo, hi = 0ull;
    if (sh <= 0) {
        lo = rne_shift(M, -sh);
    } else if (sh < 64) {
        lo = M << sh;
        hi = M >> (64 - sh);
    } else {  // a row of subnormal numbers
        lo = 0ull;
        hi = M << (sh - 64);
    }
    if (u >> 63) {
        lo = 0ull - lo;
        hi = ~hi + (lo == 0ull ? 1ull : 0ull);
    }
    unsigned long long bias = 0ull;  // 256 in the digits 2 .. ND: below bit 64
#pragma unroll
    for (int j = 0; j < ND - 1; ++j) bias |= 256ull << (kOzBits * j);
    lo += bias;
    hi += lo < bias ? 1ull : 0ull;
    const unsigned w[4] = {(unsigned)lo, (unsigned)(lo >> 32), (unsigned)hi, (unsigned)(hi >> 32)};
#pragma unroll
    for (int s = 1; s <= ND; ++s) {
        constexpr int B = kOzBits;
        const int bit = B * (ND - s), k = bit / 32;
        const unsigned f = __funnelshift_r(w[k], w[k + 1], bit % 32);
        // 2^23 + the field (1.5 2^23 + the signed first digit) as a binary32 number
        d[s - 1] = s > 1 ? __float_as_uint(__uint_as_float(0x4B000000u | (f & 511u)) - 8388864.0f)
                         : __float_as_uint(__uint_as_float(0x4B400000u + f) - 12582912.0f);
    }
}

__device__ __forceinline__ unsigned bf16_pair(unsigned a, unsigned b) { return __byte_perm(a, b, 0x7632); }

// Vector v (0 <= v < V) has elements x(v, q) = src.at(v, q), q < K. The first nd of its digit
// planes go to out[s * plane + v * ldo + q] (bf16, q < Kpad, zero padded), its exponent to
// exps[v]. Vectors V <= v < Vpad get zero digits.
//
// One matrix, with optional per-element factors scale[q], scale2[q] (diagonal matrices multiplied
// in before splitting)
struct SplitSrc {
    const double *src, *scale, *scale2;
    long long sv, sq;
    __device__ __forceinline__ int prepare() { return 0; }  // what exps[v] is raised by
    __device__ __forceinline__ double at(int v, int q) const
    {
        double x = src[(size_t)v * sv + (size_t)q * sq];
        if (scale) x *= scale[q];
        if (scale2) x *= scale2[q];
        return x;
    }
};

// Two matrices side by side along q, rows consecutive in memory: V and W / 2^e in either order, 2^e
// the size of W by its exponent field *wexp (e = 0 within 2^+-8, where 64 bits and more are left
// of either half). A type of its own: the test of every element in SplitSrc took 2 % of a binary64
// solve of n = 5000.
struct SplitHalves {
    const double *src, *src2;
    long long sq, sq2;
    int k1;
    const int *wexp;
    bool scaled_first;  // src is W: the vectors' exponents take the 2^e
    double f1, f2;
    __device__ __forceinline__ int prepare()
    {
        const int xf = *wexp;
        int e = xf == 0 || xf == 2047 ? 0 : xf - 1022;
        e = abs(e) <= 8 ? 0 : max(-1000, min(e, 1000));
        const double f = __hiloint2double((1023 - e) << 20, 0);
        f1 = scaled_first ? f : 1.0;
        f2 = scaled_first ? 1.0 : f;
        return scaled_first ? e : 0;
    }
    __device__ __forceinline__ double at(int v, int q) const
    {
        return q < k1 ? f1 * src[v + (size_t)q * sq] : f2 * src2[v + (size_t)(q - k1) * sq2];
    }
};

// Vectors along memory (sq = 1): one CTA per vector.
template <int ND, class Src>
__global__ void __launch_bounds__(256) ozaki_split_kernel(int V, int K, int Kpad, Src s, int nd,
                                                          __nv_bfloat16 *__restrict__ out, int ldo, size_t plane,
                                                          int *__restrict__ exps)
{
    __shared__ unsigned long long red[8];
    const int v = blockIdx.x, raise = s.prepare();
    unsigned long long mb = 0ull;
    if (v < V)
        for (int q = threadIdx.x; q < K; q += 256) {
            const unsigned long long b = magnitude(s.at(v, q));
            mb = b > mb ? b : mb;
        }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, mb, o);
        mb = t > mb ? t : mb;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mb;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) mb = red[w] > mb ? red[w] : mb;
    const int e = row_exponent(mb);
    if (threadIdx.x == 0) exps[v] = e == kOzNonFinite ? e : e + raise;
    unsigned *o = reinterpret_cast<unsigned *>(out + (size_t)v * ldo);
    for (int q = 2 * threadIdx.x; q < Kpad; q += 512) {
        unsigned a[ND], b[ND];
        digits_of<ND>((v < V && q < K) ? s.at(v, q) : 0.0, e, a);
        digits_of<ND>((v < V && q + 1 < K) ? s.at(v, q + 1) : 0.0, e, b);
#pragma unroll
        for (int d = 0; d < ND; ++d)
            if (d < nd) o[(d * plane + q) >> 1] = bf16_pair(a[d], b[d]);
    }
}

// Vectors across memory (sv = 1): 8 vectors per CTA, read along the vectors' index (64 bytes of
// each line) and transposed through shared memory; one CTA per vector would read one 8-byte
// element per 32-byte sector. Up to 256 elements of a vector are read once and kept in
// registers; longer ones are read twice. (32 vectors per CTA read whole lines but left two
// thirds of the SMs idle at n = 1531: 34 us at K = 256.)
template <int ND, class Src>
__global__ void __launch_bounds__(256) ozaki_split_t_kernel(int V, int K, int Kpad, Src s, int nd,
                                                            __nv_bfloat16 *__restrict__ out, int ldo, size_t plane,
                                                            int *__restrict__ exps)
{
    constexpr int R = 8, C = 256;  // vectors, elements of a tile
    __shared__ unsigned long long red[8][R];
    __shared__ double tile[R][C + 2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tx = tid & (R - 1), ty = tid / R;  // vector; elements ty, ty + 32, ..
    const int v0 = blockIdx.x * R, v = v0 + tx, raise = s.prepare();
    unsigned long long mb = 0ull;
    double x[C / 32];
    for (int q0 = 0; q0 < K; q0 += C) {
#pragma unroll
        for (int u = 0; u < C / 32; ++u) {
            const int q = q0 + ty + 32 * u;
            x[u] = (v < V && q < K) ? s.at(v, q) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < C / 32; ++u) {
            const unsigned long long b = magnitude(x[u]);
            mb = b > mb ? b : mb;
        }
    }
#pragma unroll
    for (int o = 16; o >= R; o >>= 1) {
        const unsigned long long t = __shfl_xor_sync(0xffffffffu, mb, o);
        mb = t > mb ? t : mb;
    }
    if (lane < R) red[warp][lane] = mb;
    __syncthreads();
    // warp w cuts vector v0 + w
    mb = 0ull;
#pragma unroll
    for (int w = 0; w < 8; ++w) mb = red[w][warp] > mb ? red[w][warp] : mb;
    const int e = row_exponent(mb);
    if (lane == 0) exps[v0 + warp] = e == kOzNonFinite ? e : e + raise;
    unsigned *o = reinterpret_cast<unsigned *>(out + (size_t)(v0 + warp) * ldo);
    for (int q0 = 0; q0 < Kpad; q0 += C) {
        if (K > C) {
#pragma unroll
            for (int u = 0; u < C / 32; ++u) {
                const int q = q0 + ty + 32 * u;
                x[u] = (v < V && q < K) ? s.at(v, q) : 0.0;
            }
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < C / 32; ++u) tile[tx][ty + 32 * u] = x[u];
        __syncthreads();
        for (int c = 2 * lane; c < C && q0 + c < Kpad; c += 64) {
            unsigned a[ND], b[ND];
            digits_of<ND>(tile[warp][c], e, a);
            digits_of<ND>(tile[warp][c + 1], e, b);
#pragma unroll
            for (int d = 0; d < ND; ++d)
                if (d < nd) o[(d * plane + q0 + c) >> 1] = bf16_pair(a[d], b[d]);
        }
    }
}

// ------------------------------------------------------------------ GEMM (tcgen05)
// One CTA per 128 x BN tile of C (and K range), 320 threads:
//   warp 0, one lane: TMA producer: for each k-tile (64 of K, 128 bytes with the 128-byte
//                     swizzle) the digit tiles A_1, B_1, A_2, B_2, .. A_D, B_D into two rings;
//   warp 1, one lane: MMA issuer, tcgen05.mma kind::f16 (bf16 x bf16 -> fp32), M = 128,
//                     N = BN, K = 16 per instruction;
//   warps 2..9:       epilogue, warp w owns tensor-memory lanes (rows) 32 (w mod 4) .. + 31
//                     and the tile columns h BN / 2 .. , h = (w - 2) / 4.
// Every digit tile is loaded once per k-tile and used by all its products (level by level:
// level L needs the digits up to L - 1, so the first products start when two tiles are there;
// in the last level each tile is used once and its slot given back). Loading a pair of tiles
// for each product instead costs as much shared-memory bandwidth in writes as the MMAs read.
//
// The epilogue converts each drained sum to an integer (exact) and adds it, shifted, to
// integers in registers. Refinement form: 64 bits, units of 2^(e - 9 (D + 1)) with e the
// smallest shift that cannot overflow them (D = 6: e = 7 at K = 256, one more for each
// doubling of K; 0 for D <= 4). Wide form: levels 2..5 and 6..9 in two 64-bit integers (units
// of level 5 and of level 9), put together to 128 bits at the end. The sums become binary64
// values by integer operations and are written as C = alpha (...) + beta C. (A binary64
// conversion and addition per level and element, at two a clock, took longer than the MMAs of
// a product with K <= 2048.)
//
// Measured (8192 x 2304 x 8192): D = 6 6.3 ms, 1.03 PFLOP/s of digit products (0.54 of the
// measured bf16 rate; 5.5 ms without loads and drains, what is left are the hand-overs of a
// ring that holds little more than one k-tile); n = 16384 solve, all refinement products 385
// -> 257 ms. Binary64 route, products of a solve against the SIMT kernel: n = 1531 67 -> 13 ms,
// n = 5000 758 -> 93 ms.
namespace oztc {
constexpr int BM = 128, BK = 64;
constexpr int A_BYTES = BM * BK * 2;  // 16 KB
constexpr int EPI_WARPS = 8;
constexpr int THREADS = 32 * (2 + EPI_WARPS);

template <bool WIDE> struct Cfg {
    static constexpr int BN = WIDE ? 64 : 128;
    static constexpr int RING = WIDE ? 9 : 7;  // slots of each operand's ring (> D)
    static constexpr int NBUF = WIDE ? 3 : 2;  // accumulators of the drained levels
    static constexpr int EXACT = WIDE ? 8 : 5; // levels above are summed in binary32 over K
    static constexpr int NBACK = 16;           // barriers of the give-back events (> events in flight)
    static constexpr int B_BYTES = BN * BK * 2;
    static constexpr int SMEM_BYTES = RING * (A_BYTES + B_BYTES) + 1024 + 512;
    static constexpr int TMEM_COLS = 4 * BN;   // NBUF accumulators, then the binary32 levels
    static constexpr int CW = BN / 2;          // columns per epilogue warp
};

struct Maps {
    CUtensorMap a, b;  // planes as (D * Mpad) x Kpad and (D * Npad) x Kpad bf16 matrices
};

struct Args {
    int m_real, n_real, mpad, npad, uplo, ldc;
    int kt0, nkt, ktz;  // first k-tile and number of them in this launch; k-tiles per blockIdx.z
    int digits;         // D digit planes per operand (levels 2 .. D + 1)
    int order[9];       // the levels in the order of their products
    int eshift;         // refinement form: units of the integer sums 2^(eshift - 9 (D + 1))
    const int *ea, *eb;
    double alpha, beta;
    int alpha_exp;      // alpha = +-2^alpha_exp, or kNotPow2
    double *C;
    size_t cstride;     // C of blockIdx.z: C + z cstride
    int *status;
    OzOperands src;     // for rows and columns that are not finite
    int k_real;
};
constexpr int kNotPow2 = 1 << 20;
}  // namespace oztc

// x 2^e where the result may not be a normal number (out of line: it is hardly ever taken)
__device__ __noinline__ double scale_slow(double x, int e) { return ldexp(x, e); }

// a 2^e rounded to nearest even, with integer operations where the result is a normal number
__device__ __forceinline__ double pack_double(unsigned long long nrm, bool sticky, bool neg, int biased)
{
    unsigned long long mant = nrm >> 11;  // 53 bits
    const unsigned rem = (unsigned)nrm & 0x7FFu;
    mant += (rem > 0x400u || (rem == 0x400u && (sticky || (mant & 1ull)))) ? 1ull : 0ull;
    const unsigned long long bits = ((unsigned long long)(biased - 1) << 52) + mant;  // mant has bit 52
    return __longlong_as_double((long long)(bits | (neg ? 0x8000000000000000ull : 0ull)));
}

__device__ __forceinline__ double fixed_to_double(long long a, int e)
{
    if (a == 0) return 0.0;
    const unsigned long long u = a < 0 ? 0ull - (unsigned long long)a : (unsigned long long)a;
    const int lz = __clzll((long long)u);
    const int biased = 1086 - lz + e;  // exponent field of 2^63 2^(e - lz)
    if (biased < 1 || biased > 2045) return scale_slow((double)a, e);
    return pack_double(u << lz, false, a < 0, biased);
}

// (hi 2^36 + lo) 2^e
__device__ __forceinline__ double fixed_to_double(long long hi, long long lo, int e)
{
    const __int128 t = ((__int128)hi << 36) + (__int128)lo;
    const bool neg = t < 0;
    const unsigned __int128 u = neg ? (unsigned __int128)(-t) : (unsigned __int128)t;
    const unsigned long long uh = (unsigned long long)(u >> 64), ul = (unsigned long long)u;
    if (uh == 0ull) {
        if (ul == 0ull) return 0.0;
        const int lz = __clzll((long long)ul), biased = 1086 - lz + e;
        if (biased >= 1 && biased <= 2045) return pack_double(ul << lz, false, neg, biased);
        const double v = scale_slow((double)ul, e);
        return neg ? -v : v;
    }
    const int lz = __clzll((long long)uh), biased = 1150 - lz + e;
    const unsigned long long nrm = lz ? (uh << lz) | (ul >> (64 - lz)) : uh;
    const bool sticky = (lz ? ul << lz : ul) != 0ull;
    if (biased >= 1 && biased <= 2045) return pack_double(nrm, sticky, neg, biased);
    const double v = scale_slow((double)(nrm | (sticky ? 1ull : 0ull)), e + 64 - lz);
    return neg ? -v : v;
}

// An element whose row or column holds an infinity or a NaN: the sum over q0 <= q < q1 of the
// operands themselves, which has the infinities and NaNs of binary64 arithmetic; a NaN where the
// operands are not known. Out of line: only input that is not finite gets here.
__device__ __noinline__ double direct_sum(const OzOperands &o, int row, int col, int q0, int q1)
{
    if (!o.a) return __longlong_as_double(0x7FF8000000000000ll);
    const double *pa = o.a + (size_t)row * o.av, *pb = o.b + (size_t)col * o.bv;
    double s = 0.0;
    for (int q = q0; q < q1 && s == s; ++q) s = fma(pa[(size_t)q * o.aq], pb[(size_t)q * o.bq], s);
    return s;
}

template <bool WIDE>
__global__ void __launch_bounds__(oztc::THREADS, 1)
ozaki_gemm_tc_kernel(const __grid_constant__ oztc::Maps maps, const __grid_constant__ oztc::Args a)
{
    using namespace oztc;
    using namespace tc5;
    using F = Cfg<WIDE>;
    constexpr int BN = F::BN, RING = F::RING, NBUF = F::NBUF, CW = F::CW, NBACK = F::NBACK;
    extern __shared__ unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((size_t)smem_raw + 1023) & ~(size_t)1023);
    unsigned long long *bars = (unsigned long long *)(smem + RING * (A_BYTES + F::B_BYTES));
    __shared__ unsigned tmem_slot;
    __shared__ int aborted;
    __shared__ int ebs[BN];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
    if (m0 >= a.m_real || n0 >= a.n_real) return;
    if (a.uplo && m0 + BM - 1 < n0) return;  // tile strictly above the diagonal
    const int kz = blockIdx.z * a.ktz;       // k-tiles [kz, kz + nkt) of this launch's range
    const int nkt = min(a.ktz, a.nkt - kz);
    const int D = a.digits, X = min(D, F::EXACT);  // levels 2..X are drained
    // barriers: digits loaded (one per ring slot), slots given back (events, see below),
    // accumulators full, empty; the end
    const unsigned bar0 = smem_u32(bars);
    const unsigned full0 = bar0, back0 = bar0 + 8 * RING;
    const unsigned accf0 = back0 + 8 * NBACK, acce0 = accf0 + 8 * NBUF, done = acce0 + 8 * NBUF;
    // Slots are given back two digits at a time: event u (u = 0, 1, ..) of a k-tile follows the
    // products (u + 1, D - u) and (D - u, u + 1) of the last level, the last uses of these two
    // digits (one commit for both: a commit holds the tensor pipe up for about 90 cycles).
    const int EV = (D + 1) / 2;  // events per k-tile
    const unsigned sA = smem_u32(smem), sB = sA + RING * A_BYTES;

    if (tid == 0) {
        for (int q = 0; q < RING + NBACK + NBUF; ++q) mbar_init(bar0 + 8 * q, 1);
        for (int q = 0; q < NBUF; ++q) mbar_init(acce0 + 8 * q, EPI_WARPS);
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        aborted = 0;
    }
    if (tid >= 64 && tid < 64 + BN) ebs[tid - 64] = n0 + tid - 64 < a.n_real ? a.eb[n0 + tid - 64] : 0;
    if (warp == 2) tmem_alloc(smem_u32(&tmem_slot), F::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = tmem_slot;
    auto give_up = [&](int where) {
        report_error(a.status, ELSI_ERR_TIMEOUT, where);
        atomicExch(&aborted, 1);
    };

    int armed = 0;  // digits loaded
    if (warp == 0) {
        if (lane == 0) {
            int it = 0, seen = 0;  // digits; give-back events waited for
            bool stop = false;
            for (int kt = 0; kt < nkt && !stop; ++kt) {
                const int kx = (a.kt0 + kz + kt) * BK;
                for (int q = 0; q < D; ++q, ++it) {
                    const int sl = it % RING;
                    if (it >= RING) {  // the event that gave back the slot's digit q0 (0-based)
                        const int old = it - RING, q0 = old % D;
                        const int need = old / D * EV + min(q0, D - 1 - q0);
                        for (; seen <= need && !stop; ++seen)
                            if (!mbar_wait_hot(back0 + 8 * (seen % NBACK), (seen / NBACK) & 1)) {
                                give_up(11);
                                stop = true;
                            }
                    }
                    if (stop || *(volatile int *)&aborted) { stop = true; break; }
                    mbar_expect_tx(full0 + 8 * sl, A_BYTES + F::B_BYTES);
                    tma_load_2d(sA + sl * A_BYTES, &maps.a, full0 + 8 * sl, kx, q * a.mpad + m0);
                    tma_load_2d(sB + sl * F::B_BYTES, &maps.b, full0 + 8 * sl, kx, q * a.npad + n0);
                    armed = it + 1;
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const unsigned idesc = idesc_f32acc(1, BM, BN);
            const unsigned long long dA = sdesc(sA), dB = sdesc(sB);
            int g = 0, ev = 0, base = 0;  // drained sums, events; ring slot of digit 1 of the k-tile
            unsigned phase = 0;   // parity of the full barriers at slot 'base'
            bool stop = false;
            for (int kt = 0; kt < nkt && !stop; ++kt) {
                int have = 0;  // digits of this k-tile that have arrived
                for (int o = 0; o < D && !stop; ++o) {
                    const int L = a.order[o];
                    for (; have < min(L - 1, D); ++have) {
                        const int sl = base + have >= RING ? base + have - RING : base + have;
                        const unsigned ph = base + have >= RING ? phase ^ 1u : phase;
                        if (!mbar_wait_hot(full0 + 8 * sl, ph)) {
                            give_up(13);
                            stop = true;
                            break;
                        }
                    }
                    if (stop) break;
                    unsigned d, acc;
                    const int buf = g % NBUF;
                    if (L <= X) {
                        if (g >= NBUF && !mbar_wait_hot(acce0 + 8 * buf, ((g / NBUF) & 1) ^ 1)) {
                            give_up(12);
                            stop = true;
                            break;
                        }
                        d = tmem + buf * BN;
                        acc = 0;
                    } else {
                        d = tmem + (NBUF + L - X - 1) * BN;
                        acc = kt > 0 ? 1u : 0u;
                    }
                    tc_fence_after();
                    // pairs (s, t), s + t = L, 1 <= s, t <= D; in the last level in the order
                    // (1, D), (D, 1), (2, D - 1), .. that gives the slots back as they are refilled
                    const bool last = L == D + 1;
                    for (int u = 0; u < L - 1; ++u) {
                        const int s = last ? ((u & 1) ? D - (u >> 1) : 1 + (u >> 1)) : 1 + u, t = L - s;
                        int la = base + s - 1, lb = base + t - 1;
                        la = la >= RING ? la - RING : la;
                        lb = lb >= RING ? lb - RING : lb;
                        const unsigned long long da = dA + (unsigned)(la * (A_BYTES >> 4));
                        const unsigned long long db = dB + (unsigned)(lb * (F::B_BYTES >> 4));
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk) {
                            mma_bf16(d, da + 2 * kk, db + 2 * kk, idesc, acc);
                            acc = 1;
                        }
                        if (last && ((u & 1) || u == D - 1)) {
                            mma_commit(back0 + 8 * (ev % NBACK));
                            ++ev;
                        }
                    }
                    if (L <= X) {
                        mma_commit(accf0 + 8 * buf);
                        ++g;
                    }
                }
                base += D;
                if (base >= RING) { base -= RING; phase ^= 1u; }
            }
            mma_commit(done);
            if (stop) mbar_wait(done, 0);  // nothing in flight when the tensor memory is freed
        }
    } else {
        // tensor-memory loads are warp-collective: every lane runs them (rows past m only skip
        // their global-memory accesses) and the wait results are made uniform
        const int quarter = warp & 3, c0 = ((warp - 2) >> 2) * CW;  // rows, first column
        const int row = m0 + quarter * 32 + lane;
        const bool row_in = row < a.m_real;
        const unsigned tlane = tmem + ((unsigned)(quarter * 32) << 16) + c0;
        long long acc[CW], low[WIDE ? CW : 1];
#pragma unroll
        for (int j = 0; j < CW; ++j) acc[j] = 0;
#pragma unroll
        for (int j = 0; j < (WIDE ? CW : 1); ++j) low[j] = 0;
        bool ok = true;
        int g = 0;
        for (int kt = 0; kt < nkt && ok; ++kt)
            for (int L = 2; L <= X; ++L, ++g) {
                const int buf = g % NBUF;
                ok = __all_sync(0xffffffffu, mbar_wait_hot(accf0 + 8 * buf, (g / NBUF) & 1));
                if (!ok) {
                    if (lane == 0) give_up(14);
                    break;
                }
                tc_fence_after();
                const int sh = WIDE ? kOzBits * (L <= 5 ? 5 - L : 9 - L) : kOzBits * (D + 1 - L) - a.eshift;
#pragma unroll
                for (int q = 0; q < CW / 16; ++q) {
                    float v[16];
                    tmem_ld16(tlane + buf * BN + q * 16, v);
                    if (WIDE) {
                        const int mul = 1 << sh;  // sh <= 27
                        if (L <= 5) {
#pragma unroll
                            for (int j = 0; j < 16; ++j) acc[q * 16 + j] += (long long)__float2int_rn(v[j]) * mul;
                        } else {
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                low[WIDE ? q * 16 + j : 0] += (long long)__float2int_rn(v[j]) * mul;
                        }
                    } else if (sh >= 32) {
                        const int up = sh - 32;
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            acc[q * 16 + j] += (long long)((unsigned long long)((unsigned)__float2int_rn(v[j]) << up) << 32);
                    } else if (sh >= 0) {
                        const int mul = 1 << sh;  // sh <= 30: see oz_shift()
#pragma unroll
                        for (int j = 0; j < 16; ++j) acc[q * 16 + j] += (long long)__float2int_rn(v[j]) * mul;
                    } else {
                        const int half = 1 << (-sh - 1);
#pragma unroll
                        for (int j = 0; j < 16; ++j) acc[q * 16 + j] += (__float2int_rn(v[j]) + half) >> -sh;
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acce0 + 8 * buf);
            }
        if (ok) {
            ok = __all_sync(0xffffffffu, mbar_wait(done, 0));
            if (!ok && lane == 0) give_up(15);
        }
        if (ok) {
            tc_fence_after();
            // the levels summed in binary32, in the units of the integers
            for (int L = X + 1; L <= D + 1; ++L) {
                const int sh = WIDE ? 0 : kOzBits * (D + 1 - L) - a.eshift;
                const float sc = __int_as_float((127 + sh) << 23);
#pragma unroll
                for (int q = 0; q < CW / 16; ++q) {
                    float v[16];
                    tmem_ld16(tlane + (NBUF + L - X - 1) * BN + q * 16, v);
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (WIDE) low[WIDE ? q * 16 + j : 0] += __float2ll_rn(v[j]);
                        else acc[q * 16 + j] += __float2ll_rn(v[j] * sc);
                    }
                }
            }
            const bool pow2 = a.alpha_exp != kNotPow2;
            const bool neg = pow2 && a.alpha < 0.0;
            const int er = (row_in ? a.ea[row] : 0) - kOzBits * (WIDE ? 9 : D + 1) + (WIDE ? 0 : a.eshift) +
                           (pow2 ? a.alpha_exp : 0);
            const bool row_bad = row_in && a.ea[row] == kOzNonFinite;
            double *crow = a.C + blockIdx.z * a.cstride + (size_t)row;
            // C = beta C + sum, 4 columns at a time (the loads of C first). The sums go through
            // shared memory (the rings are done), each thread reading back its own: a loop over
            // registers would have to be unrolled, and that much straight-line code, run once,
            // waits for instructions (12 us of a tile's 34).
            long long *stage = reinterpret_cast<long long *>(smem) + (tid - 64);
            constexpr int ET = 32 * EPI_WARPS;
#pragma unroll
            for (int j = 0; j < CW; ++j) {
                stage[j * ET] = acc[j];
                if (WIDE) stage[(CW + j) * ET] = low[WIDE ? j : 0];
            }
#pragma unroll 1
            for (int q = 0; q < CW; q += 4) {
                double cv[4];
                bool in[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int col = n0 + c0 + q + j;
                    in[j] = row_in && col < a.n_real && (!a.uplo || row >= col);
                    cv[j] = (in[j] && a.beta != 0.0) ? crow[(size_t)col * a.ldc] : 0.0;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int cl = c0 + q + j, col = n0 + cl;
                    double val;
                    if (WIDE) val = fixed_to_double(stage[(q + j) * ET], stage[(CW + q + j) * ET], er + ebs[cl]);
                    else val = fixed_to_double(stage[(q + j) * ET], er + ebs[cl]);
                    if (in[j] && (row_bad || ebs[cl] == kOzNonFinite)) {
                        const int q0 = (a.kt0 + kz) * BK;
                        val = direct_sum(a.src, row, col, q0, min(a.k_real, q0 + nkt * BK));
                        if (pow2) val *= fabs(a.alpha);
                    }
                    if (neg) val = -val;
                    if (!pow2) val *= a.alpha;
                    if (a.beta == 1.0) val += cv[j];
                    else if (a.beta != 0.0) val = fma(a.beta, cv[j], val);
                    if (in[j]) crow[(size_t)col * a.ldc] = val;
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (aborted && warp == 0 && lane == 0) {
        for (int it = (armed > RING ? armed - RING : 0); it < armed; ++it)
            mbar_wait(full0 + 8 * (it % RING), (it / RING) & 1);
    }
    __syncthreads();
    if (warp == 2) tmem_free(tmem, F::TMEM_COLS);
}

// C = beta C + sum of the K ranges' partial products (ascending, m x n each)
__global__ void ozaki_reduce_kernel(int m, int n, int parts, const double *__restrict__ part, double beta,
                                    double *C, int ldc)
{
    const size_t total = (size_t)m * n;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int z = 0; z < parts; ++z) s += part[(size_t)z * total + e];
        double *c = C + (e % m) + (e / m) * (size_t)ldc;
        *c = beta != 0.0 ? fma(beta, *c, s) : s;
    }
}

size_t ozaki_plane_elems(int V, int K)
{
    return (size_t)ceil_div(V, kOzBM) * kOzBM * (size_t)(ceil_div(K, kOzBK) * kOzBK);
}

size_t ozaki_split_elems(int V, int K, int digits) { return ozaki_plane_elems(V, K) * digits; }

cudaError_t ozaki_split(cudaStream_t st, int V, int K, const double *src, long long sv,
                        long long sq, const double *scale, const double *scale2,
                        __nv_bfloat16 *planes, int *exps, int digits)
{
    if (digits < 1 || (digits > kOzDigits && digits != kOzWide)) return cudaErrorInvalidValue;
    const int Vpad = ceil_div(V, kOzBM) * kOzBM;
    const int Kpad = ceil_div(K, kOzBK) * kOzBK;
    const size_t plane = ozaki_plane_elems(V, K);
    SplitSrc s;
    s.src = src; s.scale = scale; s.scale2 = scale2; s.sv = sv; s.sq = sq;
    const bool across = sv == 1 && sq != 1;
    EGB_COUNT_LAUNCH();
    if (digits == kOzWide) {
        if (across) ozaki_split_t_kernel<kOzWide><<<Vpad / 8, 256, 0, st>>>(V, K, Kpad, s, digits, planes, Kpad, plane, exps);
        else ozaki_split_kernel<kOzWide><<<Vpad, 256, 0, st>>>(V, K, Kpad, s, digits, planes, Kpad, plane, exps);
    } else {
        if (across) ozaki_split_t_kernel<kOzDigits><<<Vpad / 8, 256, 0, st>>>(V, K, Kpad, s, digits, planes, Kpad, plane, exps);
        else ozaki_split_kernel<kOzDigits><<<Vpad, 256, 0, st>>>(V, K, Kpad, s, digits, planes, Kpad, plane, exps);
    }
    return cudaGetLastError();
}

cudaError_t ozaki_split_halves(cudaStream_t st, int V, int k1, const double *src, long long sq, const double *src2,
                               long long sq2, const int *wexp, bool scaled_first, __nv_bfloat16 *planes, int *exps)
{
    const int K = 2 * k1, Vpad = ceil_div(V, kOzBM) * kOzBM, Kpad = ceil_div(K, kOzBK) * kOzBK;
    SplitHalves s = {};
    s.src = src; s.src2 = src2; s.sq = sq; s.sq2 = sq2; s.k1 = k1; s.wexp = wexp; s.scaled_first = scaled_first;
    EGB_COUNT_LAUNCH();
    ozaki_split_t_kernel<kOzWide><<<Vpad / 8, 256, 0, st>>>(V, K, Kpad, s, kOzWide, planes, Kpad,
                                                            ozaki_plane_elems(V, K), exps);
    return cudaGetLastError();
}

// Units of the integer sums of the refinement form for K terms: level 2 adds up to
// K 2^16 2^(9 (D - 1) - e), which has to stay below 2^62; a shift of exactly 31 is avoided (the
// multiplication by 2^31 does not fit a signed 32-bit factor).
static int oz_shift(int k, int digits)
{
    int lg = 0;
    while ((1ll << lg) < k) ++lg;
    int e = lg + 16 + kOzBits * (digits - 1) - 62;
    if (e < 0) e = 0;
    for (bool again = true; again;) {
        again = false;
        for (int L = 2; L <= digits; ++L)
            if (kOzBits * (digits + 1 - L) - e == 31) again = true;
        if (again) ++e;
    }
    return e;
}

template <bool WIDE>
static cudaError_t oz_launch(cudaStream_t st, dim3 grid, const oztc::Maps &maps, const oztc::Args &a)
{
    static PerDeviceOnce attr;
    cudaError_t e = once_per_device(attr, [] {
        return cudaFuncSetAttribute(ozaki_gemm_tc_kernel<WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    oztc::Cfg<WIDE>::SMEM_BYTES);
    });
    if (e != cudaSuccess) return e;
    EGB_COUNT_LAUNCH();
    ozaki_gemm_tc_kernel<WIDE><<<grid, oztc::THREADS, oztc::Cfg<WIDE>::SMEM_BYTES, st>>>(maps, a);
    return cudaGetLastError();
}

cudaError_t ozaki_gemm(cudaStream_t st, int m, int n, int k, double alpha,
                       const __nv_bfloat16 *Ad, const int *ea, const __nv_bfloat16 *Bd,
                       const int *eb, double beta, double *C, int ldc, int uplo, int digits,
                       double *part, size_t part_elems, const OzOperands &src)
{
    const bool wide = digits == kOzWide;
    if (digits < 1 || (digits > kOzDigits && !wide)) return cudaErrorInvalidValue;
    using namespace oztc;
    if (m <= 0 || n <= 0) return cudaSuccess;
    const int mpad = ceil_div(m, kOzBM) * kOzBM, npad = ceil_div(n, kOzBN) * kOzBN;
    const int kpad = ceil_div(k, kOzBK) * kOzBK;
    const int bn = wide ? Cfg<true>::BN : Cfg<false>::BN;
    Maps maps;
    if (!tc5::make_map_2d(&maps.a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Ad, (long long)digits * mpad, kpad,
                          kpad, BK, BM) ||
        !tc5::make_map_2d(&maps.b, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Bd, (long long)digits * npad, kpad,
                          kpad, BK, bn))
        return cudaErrorNotSupported;
    Args a;
    a.m_real = m; a.n_real = n; a.mpad = mpad; a.npad = npad; a.uplo = uplo;
    a.ldc = ldc; a.ea = ea; a.eb = eb; a.alpha = alpha; a.beta = beta; a.C = C; a.cstride = 0;
    a.digits = digits; a.src = src; a.k_real = k;
    for (int o = 0; o < 9; ++o) a.order[o] = o + 2;
    if (digits == 6) {  // level 6 (not drained) between 4 and 5: time to drain the two accumulators
        a.order[3] = 6;
        a.order[4] = 5;
    }
    int xp = 0;
    const double mant = frexp(alpha, &xp);  // alpha = mant 2^xp
    a.alpha_exp = (mant == 0.5 || mant == -0.5) ? xp - 1 : kNotPow2;
    float *tw;
    size_t te;
    int *ts = nullptr;
    tc_scratch(&tw, &te, &ts);
    // a status word for calls outside a solve (one per device, kept until exit)
    static int *dummy_status[kMaxDevices] = {};
    static PerDeviceOnce once;
    cudaError_t attr_err = once_per_device(once, [] {
        int dev = 0;
        cudaError_t r = cudaGetDevice(&dev);
        if (r == cudaSuccess && dev >= 0 && dev < kMaxDevices && !dummy_status[dev]) {
            int *p = nullptr;
            r = cudaMalloc((void **)&p, 8 * sizeof(int));
            if (r == cudaSuccess) r = cudaMemset(p, 0, 8 * sizeof(int));
            if (r == cudaSuccess) dummy_status[dev] = p;
        }
        return r;
    });
    if (attr_err != cudaSuccess) return attr_err;
    int dev_now = 0;
    cudaGetDevice(&dev_now);
    a.status = ts ? ts : (dev_now >= 0 && dev_now < kMaxDevices ? dummy_status[dev_now] : nullptr);
    if (!a.status) return cudaErrorInvalidDevice;
    const int tiles_m = mpad / BM, tiles_n = ceil_div(n, bn);
    auto go = [&](dim3 grid) { return wide ? oz_launch<true>(st, grid, maps, a) : oz_launch<false>(st, grid, maps, a); };
    // Few output tiles and a long K (A22 V of a panel): the K range is divided over CTAs, each
    // with at least two k-tiles, and the partial products are added in a second pass.
    const int nkt_all = ceil_div(kpad, BK);
    if (!uplo && k <= kOzSegK && part) {
        int parts = 152 / (tiles_m * tiles_n);
        if (parts > nkt_all / 2) parts = nkt_all / 2;
        if ((size_t)(parts > 0 ? parts : 1) * m * n > part_elems) parts = (int)(part_elems / ((size_t)m * n));
        if (parts > 1) {
            a.kt0 = 0; a.nkt = nkt_all; a.ktz = ceil_div(nkt_all, parts);
            parts = ceil_div(nkt_all, a.ktz);
            a.eshift = oz_shift(a.ktz * BK, digits);
            a.beta = 0.0; a.C = part; a.ldc = m; a.cstride = (size_t)m * n;
            cudaError_t e = go(dim3(tiles_m, tiles_n, parts));
            if (e != cudaSuccess) return e;
            int rg = ceil_div((long long)m * n, 256);
            EGB_COUNT_LAUNCH();
            ozaki_reduce_kernel<<<rg > 152 * 8 ? 152 * 8 : rg, 256, 0, st>>>(m, n, parts, part, beta, C, ldc);
            return cudaGetLastError();
        }
    }
    // K segments of kOzSegK (a multiple of BK): the first applies beta, the rest add
    for (int k0 = 0; k0 < kpad; k0 += kOzSegK) {
        const int k1 = min(kpad, k0 + kOzSegK);
        a.kt0 = k0 / BK;
        a.nkt = a.ktz = ceil_div(k1 - k0, BK);
        a.eshift = oz_shift(k1 - k0, digits);
        a.beta = k0 == 0 ? beta : 1.0;
        cudaError_t e = go(dim3(tiles_m, tiles_n));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace egb
