// Digit slicing for the sliced tensor-core updates (gemm_oz.cu): balancing
// exponents, and the K-major BF16 digit slices of both operands.
#pragma once

#include <cuda_bf16.h>

#include <type_traits>

#include "common.cuh"
#include "df64.cuh"

namespace rbt {

// ---- binary exponents

// Binary exponent e of a nonzero value (|x| < 2^e <= 2 |x|); kNoExp for zero.
// kNoExp is the int whose four bytes are 0x80, so that one memset initializes
// the atomicMax targets below.
constexpr int kNoExp = (int)0x80808080u;
// exponent of a row or column with an entry that is not finite (double
// operands), above every exponent that occurs
constexpr int kBadExp = 1 << 28;

__device__ __forceinline__ int exp_of(float x)
{
    if (x == 0.f) return kNoExp;
    int e;
    frexpf(x, &e);
    return e;
}

__device__ __forceinline__ int exp_of(df64 x) { return exp_of(x.hi); }

// The same for a double (subnormals included); kBadExp for Inf and NaN: a row
// of A or a column of B that holds one makes its row or column of C NaN, as
// the products would (an exact zero's product with it is NaN too).
__device__ __forceinline__ int exp_of(double x)
{
    const long long m = __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll;
    const int ex = (int)(m >> 52);
    if (ex == 0x7FF) return kBadExp;
    if (m == 0) return kNoExp;
    return ex ? ex - 1022 : 64 - __clzll(m) - 1074;
}

__device__ __forceinline__ int finite_exp(int e) { return e == kBadExp ? kNoExp : e; }

namespace oz {

constexpr int BETA = 7;       // bits per digit
constexpr int kDigits64 = 9;  // digits of double operands: 63 bits
// an operand's element type, by its digits
template <int S> using elem_t = std::conditional_t<S == kDigits64, double, df64>;

// WIDE (the seven-digit factorization): the leading digit uses the eighth bit
// that a bf16 integer has (up to 256) and may be as large as 128, so the scale
// is a bit finer.  An accumulator of weight t then holds at most (t + 1) K 2^12
// (two products of a leading digit and another, 2^13 each): 9 K 2^12 <= 2^24
// for K <= 448.  Half the error of plain seven digits; with rows and columns
// scaled over three decades refinement at n = 40003 is at the edge of what
// those converge for (steps to 1e-13 on four systems: 4, 3, 6, 8; with the
// eighth bit 3, 2, 2, 4).

// ---- digits

// The S balanced base-128 digits of an entry, each plus 64: unsigned 7-bit
// fields of 28-bit words, least significant first (adding 64 to every digit
// turns balanced digits into plain ones, so no carry runs from digit to
// digit).  The leading digit is whatever is left on top: in [-64, 64], its
// field up to 128, or with WIDE in [-128, 128] and without the 64.
template <int S> struct Fields {
    unsigned w[3];
};
constexpr unsigned kBias4 = 64u * (1u + 128u + 128u * 128u + 128u * 128u * 128u);
constexpr unsigned kMask28 = (1u << 28) - 1;
// the 64s of the digits above the low four (S <= 8)
template <int S, bool WIDE> constexpr unsigned high_bias()
{
    return S == 8 ? kBias4 : (kBias4 & ((1u << (7 * (S - (WIDE ? 5 : 4)))) - 1));
}

// Y = rint(hi 2^(7 S - e)) + rint(lo 2^(7 S - e)) for v = hi + lo, |v| <=
// 2^(e-1) (|Y| <= 2^(7 S - 1)), or 2^e with WIDE: each scaled part is split at 2^28 into an
// integer multiple and a remainder that the conversion rounds, so the words
// come from 32-bit integers.  The scaling is two exact multiplications by
// powers of two (a part that underflows on the way would round to 0 anyway).
template <int S, bool WIDE> __device__ __forceinline__ Fields<S> fields(df64 v, int e)
{
    static_assert(S >= 5 && S <= 8 && BETA == 7, "the split at 2^28 leaves at most four digits above it");
    const int s = S * BETA - e;
    float hs, ls;
    if (s >= -250 && s <= 250) {
        const int s1 = s >> 1;
        const float f1 = __int_as_float((s1 + 127) << 23), f2 = __int_as_float((s - s1 + 127) << 23);
        hs = v.hi * f1 * f2;
        ls = v.lo * f1 * f2;
    } else {
        hs = ldexpf(v.hi, s);
        ls = ldexpf(v.lo, s);
    }
    const float hh = rintf(hs * 0x1p-28f), lh = rintf(ls * 0x1p-28f);
    const int low = __float2int_rn(fmaf(-hh, 0x1p28f, hs)) + __float2int_rn(fmaf(-lh, 0x1p28f, ls));  // |low| <= 2^28
    const int lb = low + (int)kBias4;
    constexpr unsigned kBiasHigh = high_bias<S, WIDE>();
    const int hb = __float2int_rn(hh) + __float2int_rn(lh) + (lb >> 28) + (int)kBiasHigh;
    Fields<S> f;
    f.w[0] = (unsigned)lb & kMask28;
    f.w[1] = (unsigned)hb;
    f.w[2] = 0;
    return f;
}

// round(v 2^(63 - e)), |v| < 2^(e-1): the significand shifted to an integer of
// at most 62 bits (rounded only where bits fall below 2^(e - 63)).
template <int S, bool WIDE> __device__ __forceinline__ Fields<S> fields(double v, int e)
{
    static_assert(S == kDigits64 && BETA == 7, "two words of four digits and a leading one");
    const long long bits = __double_as_longlong(v);
    const int ex = (int)(bits >> 52) & 0x7FF;
    const long long m = (bits & 0xFFFFFFFFFFFFFll) | (ex ? 1ll << 52 : 0ll);
    const int sh = (ex ? ex : 1) - 1075 + S * BETA - e;  // at most 9
    long long y = sh >= 0 ? m << sh : (sh > -60 ? (m + (1ll << (-sh - 1))) >> -sh : 0ll);
    if (bits < 0) y = -y;
    const unsigned long long b = (unsigned long long)kBias4 * ((1ull << 28) + 1) + (64ull << 56) + (unsigned long long)y;
    Fields<S> f;
    f.w[0] = (unsigned)b & kMask28;
    f.w[1] = (unsigned)(b >> 28) & kMask28;
    f.w[2] = (unsigned)(b >> 56);
    return f;
}

// all digits zero
template <int S, bool WIDE> __device__ __forceinline__ Fields<S> no_digits()
{
    Fields<S> f;
    f.w[0] = kBias4;
    f.w[1] = S == 9 ? kBias4 : high_bias<S, WIDE>();
    f.w[2] = 64;
    return f;
}

// Digit p (0 = most significant) of two neighbouring entries as a bf16 pair:
// a field under the exponent of 128 is the bf16 of 128 + field, and one packed
// subtraction of 192 leaves the digits, exactly.
template <int S, int P, bool WIDE> __device__ __forceinline__ unsigned pack2(const Fields<S> &a, const Fields<S> &b)
{
    constexpr int L = S - 1 - P, W = L / 4, SH = 7 * (L % 4);
    unsigned w;
    if constexpr (P == 0 && WIDE) {
        // through float: 2^23 + 2^22 + d, less 2^23 + 2^22, whose upper half is the bf16
        const float x = __int_as_float(0x4B400000 + ((int)a.w[W] >> SH)) - 12582912.0f;
        const float y = __int_as_float(0x4B400000 + ((int)b.w[W] >> SH)) - 12582912.0f;
        return __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
    }
    if (P == 0)
        w = (a.w[W] >> SH) + ((b.w[W] >> SH) << 16) + 0x43004300u;
    else
        w = ((a.w[W] >> SH) & 0x7Fu) | (((b.w[W] >> SH) & 0x7Fu) << 16) | 0x43004300u;
    __nv_bfloat162 x;
    memcpy(&x, &w, 4);
    x = __hsub2(x, __floats2bfloat162_rn(192.f, 192.f));
    memcpy(&w, &x, 4);
    return w;
}

// A digit (an integer of at most 8 significant bits) as a bf16.
__device__ __forceinline__ __nv_bfloat16 bf16_of_digit(int r) { return __int2bfloat16_rn(r); }

// ---- balancing exponents of a standalone update

// k-balancing exponents, stored as atomicMax targets (initialized to kNoExp):
// ka[k] = max over rows of E(A_ik), kb[k] = max over columns of E(B_kj).  (A
// factorization gets them from its panel TRSMs instead.)  One launch for both:
// blocks [0, na) take A (block b: column k = b / ca, rows of chunk b % ca,
// 4096 rows each; with ta 64 of its rows, stored as columns), the rest take B
// (64 columns each; threads over k).
template <typename TE>
__global__ void __launch_bounds__(256) kexp_kernel(int M, int K, int N, int ca, int na, int ta,
                                                   const TE *__restrict__ A, int64_t lda, const TE *__restrict__ B,
                                                   int64_t ldb, int *ka, int *kb)
{
    const int b = blockIdx.x;
    if (b < na && !ta) {
        const int k = b / ca, chunk = b % ca;
        int e = kNoExp;
        const int r1 = min(M, (chunk + 1) * 4096);
#pragma unroll 8
        for (int r = chunk * 4096 + threadIdx.x; r < r1; r += 256) e = max(e, finite_exp(exp_of(A[r + (int64_t)k * lda])));
        for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
        if (threadIdx.x % 32 == 0 && e > kNoExp) atomicMax(ka + k, e);
        return;
    }
    // B, or an A given as its transpose (ta: K x M): 64 columns
    const bool is_a = b < na;
    const TE *src = is_a ? A : B;
    const int64_t ld = is_a ? lda : ldb;
    const int c0 = (is_a ? b : b - na) * 64, c1 = min(is_a ? M : N, c0 + 64);
    for (int k = threadIdx.x; k < K; k += 256) {
        int e = kNoExp;
#pragma unroll 8
        for (int c = c0; c < c1; c++) e = max(e, finite_exp(exp_of(src[k + (int64_t)c * ld])));
        if (e > kNoExp) atomicMax((is_a ? ka : kb) + k, e);
    }
}

// t_k of the balancing, from the largest exponents a of column k of A and b of
// row k of B (0 where one of them is all zero)
__device__ __forceinline__ int kshift(int a, int b)
{
    if (a == kNoExp || b == kNoExp) return 0;
    const int d = b - a;
    return d >= 0 ? d / 2 : -((1 - d) / 2);  // floor(d / 2)
}

// ---- slicing

// One operand: stored rows x K (by_rows; the slices' rows are its rows) or K x
// rows (its columns), column-major.  Its k are scaled by 2^(sign t_k), sign 1
// for A (or its transpose stored K x M) and -1 for B.  Slice p goes to rows p rows_p ..
// of a K-major [S rows_p][Kp] bf16 array (zeros past rows and K), the row
// exponents to exps.  The balancing exponents of A's columns are the larger
// of ka and ka2, those of B's rows kb; without kb the balancing is A's alone.
template <typename TE> struct SliceJob {
    const TE *src;
    int64_t ld;
    int rows, rows_p;
    const int *ka, *ka2, *kb;
    __nv_bfloat16 *out;
    int *exps;
    int by_rows, sign, blocks;
};
template <typename TE> struct SliceJobs {
    SliceJob<TE> job[4];
    int K, Kp;
};

constexpr int kSliceRows = 16;  // rows of A per CTA

template <int S, bool WIDE> __device__ __forceinline__ void store4(const Fields<S> (&f)[4], __nv_bfloat16 *out, int64_t slice)
{
    // four neighbouring k of every digit: 8-byte stores
    auto put = [&](auto p) {
        constexpr int P = decltype(p)::value;
        *reinterpret_cast<uint2 *>(out + P * slice) = make_uint2(pack2<S, P, WIDE>(f[0], f[1]), pack2<S, P, WIDE>(f[2], f[3]));
    };
    put(std::integral_constant<int, 0>());
    put(std::integral_constant<int, 1>());
    put(std::integral_constant<int, 2>());
    put(std::integral_constant<int, 3>());
    put(std::integral_constant<int, 4>());
    put(std::integral_constant<int, 5>());
    put(std::integral_constant<int, 6>());
    if constexpr (S >= 8) put(std::integral_constant<int, 7>());
    if constexpr (S >= 9) put(std::integral_constant<int, 8>());
}

template <int S> constexpr size_t slice_smem_bytes(int Kp)
{
    return (size_t)Kp * sizeof(int) + (size_t)kSliceRows * (Kp + 2) * sizeof(elem_t<S>);
}

// Up to four jobs in one launch, each entry read once.  A: 16 rows per CTA
// through a shared tile (read down the columns, 128-byte segments; written
// along k); B: LPC lanes per column with its K entries in registers (LPC = 16
// for K <= 64, 32 for K <= 512).
template <int S, int LPC, bool WIDE>
__global__ void __launch_bounds__(256) slice_kernel(const __grid_constant__ SliceJobs<elem_t<S>> jobs)
{
    using TE = elem_t<S>;
    extern __shared__ __align__(16) unsigned char slice_smem[];
    __shared__ int smax[8][kSliceRows];
    const int K = jobs.K, Kp = jobs.Kp, tid = threadIdx.x;
    TE *tile = reinterpret_cast<TE *>(slice_smem);
    int *ts = reinterpret_cast<int *>(tile + kSliceRows * (Kp + 2));
    int blk = blockIdx.x, which = 0;
    while (which < 3 && blk >= jobs.job[which].blocks) blk -= jobs.job[which++].blocks;
    const SliceJob<TE> &J = jobs.job[which];
    const int rows = J.rows;
    const int64_t slice = (int64_t)J.rows_p * Kp;
    auto shifts = [&]() {  // t_k of every k
        for (int k = tid; k < Kp; k += 256) {
            const int a = k < K ? max(J.ka[k], J.ka2[k]) : kNoExp;
            ts[k] = a == kNoExp ? 0 : J.kb ? kshift(a, J.kb[k]) : -a;
        }
    };
    if (J.by_rows) {
        const int ld_t = Kp + 2, r = tid % kSliceRows, kl = tid / kSliceRows;
        const int m = blk * kSliceRows + r;
#pragma unroll 8
        for (int k = kl; k < Kp; k += 16)
            tile[r * ld_t + k] = (m < rows && k < K) ? J.src[m + (int64_t)k * J.ld] : TE(0);
        shifts();
        __syncthreads();
        int emax = kNoExp;  // max over k of E(A_mk 2^t_k)
        for (int k = kl; k < Kp; k += 16) {
            const int e = exp_of(tile[r * ld_t + k]);
            if (e != kNoExp) emax = max(emax, e == kBadExp ? e : e + ts[k]);
        }
        emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, 16));
        if (tid % 32 < 16) smax[tid / 32][r] = emax;
        __syncthreads();
        const int row = tid / 16, kq = tid % 16, mm = blk * kSliceRows + row;
        int e = smax[0][row];
#pragma unroll
        for (int w = 1; w < 8; w++) e = max(e, smax[w][row]);
        e = e == kNoExp ? 0 : (e == kBadExp ? e : e + (WIDE ? 0 : 1));
        if (kq == 0 && mm < rows) J.exps[mm] = e;
        for (int k = 4 * kq; k < Kp; k += 64) {
            Fields<S> f[4];
#pragma unroll
            for (int u = 0; u < 4; u++)
                f[u] = e != kBadExp ? fields<S, WIDE>(tile[row * ld_t + k + u], e - ts[k + u]) : no_digits<S, WIDE>();
            store4<S, WIDE>(f, J.out + (int64_t)mm * Kp + k, slice);
        }
    } else {
        constexpr int CPB = 256 / LPC, NI = LPC == 16 ? 1 : 4;
        const int l = tid % LPC, c = blk * CPB + tid / LPC;
        const bool in = c < rows;
        const TE *src = J.src + (in ? (int64_t)c * J.ld : 0);
        TE v[NI][4];
#pragma unroll
        for (int i = 0; i < NI; i++)
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int k = 4 * l + 4 * LPC * i + u;
                v[i][u] = (in && k < K) ? src[k] : TE(0);
            }
        shifts();
        __syncthreads();
        const int sg = J.sign;
        int emax = kNoExp;  // max over k of E(B_kc 2^-t_k)
#pragma unroll
        for (int i = 0; i < NI; i++)
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int k = 4 * l + 4 * LPC * i + u;
                const int e = exp_of(v[i][u]);
                if (k < K && e != kNoExp) emax = max(emax, e == kBadExp ? e : e + sg * ts[k]);
            }
#pragma unroll
        for (int o = LPC / 2; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
        const int e = emax == kNoExp ? 0 : (emax == kBadExp ? emax : emax + (WIDE ? 0 : 1));
        if (l == 0 && in) J.exps[c] = e;
        if (c >= J.rows_p) return;
#pragma unroll
        for (int i = 0; i < NI; i++) {
            const int k = 4 * l + 4 * LPC * i;
            if (k >= Kp) break;
            Fields<S> f[4];
#pragma unroll
            for (int u = 0; u < 4; u++) f[u] = e != kBadExp ? fields<S, WIDE>(v[i][u], e - sg * ts[k + u]) : no_digits<S, WIDE>();
            store4<S, WIDE>(f, J.out + (int64_t)c * Kp + k, slice);
        }
    }
}

}  // namespace oz
}  // namespace rbt
