// Triangular solves with the GENP factors (sm_103a): (L U)^{-1} B and
// (L U)^{-T} B in one persistent launch.
//
// What bounds a solve.  Reading the factors once takes n^2 entries of HBM
// traffic (12.8 GB, 1.9 ms at n = 40003 in pairs), but block b of 64 rows
// cannot finish before block b - 1: 2 n / 64 dependent steps.  The step's
// length (publish, see, multiply by one 64 x 64 block, finish the diagonal
// block) is what a solve costs for few right-hand sides; with many, the
// multiply-adds on the FP32 or FP64 pipe are.
//
// Tasks.  A task is one 64-row block of one triangle for one group of R
// right-hand sides; the groups are independent chains.  CTAs take tasks from
// a device counter in solve order, all of L (or U^T) before U (or L^T), and
// only ever wait on tasks taken earlier, which belong to running CTAs: the
// chain always advances.  A task streams its row block's columns of every
// earlier block (the next block's entries are loaded while the current one
// is multiplied), then finishes its diagonal block with the precomputed
// inverse plus one correction step (x0 = D^-1 r, x = x0 + D^-1 (r - D x0)).
//
// Messages.  A solved block is published as its values alone: the solution
// arrays are filled with an all-ones pattern (a NaN no arithmetic returns)
// before the launch, and a reader waits until no such pattern is left in the
// 64 values.  That is one store and one load on the chain where values, a
// fence and a flag need two of each.  Only warp 0 of a CTA polls, and a CTA
// d blocks behind the front polls d times less often, so that the readers
// in flight do not queue up on the front's cache lines.  Every wait is
// bounded and records a timeout in err instead of hanging; it then goes on
// with what it has, publishing ordinary values, and no later wait lasts.
//
// Rounding does not depend on timing: each thread adds its columns in solve
// order and the partial sums meet in a fixed order.
//
// Measured on GB300 per solve (both triangles), this form against one launch
// per triangle with flags (one column) and a blocked sweep of two launches
// per 64 rows (four columns and more): pairs, n = 8197, 1 / 8 / 32 right-hand
// sides 1.83 / 28.3 / 33.5 ms -> 1.00 / 1.14 / 2.27 ms; double 2.20 / 44.5 /
// 52.5 -> 1.86 / 2.27 / 4.62 ms; pairs, one column, n = 40003: 11.0 -> 5.0 ms.
// A step takes 3.9 us in pairs, 7.2 in double (its block products run at two
// FP64 multiply-adds a clock), 1.4 in float.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "df64.cuh"
#include "genp_internal.cuh"

namespace rbt {

constexpr int kTrsvNB = 64;
constexpr int kTrsvThreads = 256;
constexpr int kTrsvLd = kTrsvNB + 4;  // shared rows of 68: four lanes of 4 rows fall on different 8-byte banks

// An entry of the stored factor in the solve's arithmetic type T: the same
// type, a float widened to double, or a double-float pair rounded to double.
template <typename T, typename TF> __device__ __forceinline__ T elem_as(TF v) { return T(v); }
template <> __device__ __forceinline__ double elem_as<double, df64>(df64 v) { return df_to_double(v); }

template <typename T> __device__ __forceinline__ T from_double(double v) { return T(v); }
template <> __device__ __forceinline__ df64 from_double<df64>(double v) { return df_from_double(v); }
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(float v) { return (double)v; }
__device__ __forceinline__ double to_double(df64 v) { return df_to_double(v); }

// A running sum of products.  Double-float: the leading part stays exact by
// TwoSum; its errors gather in one float and the products' own errors and
// cross terms, smaller by the ratio of a product to the sum, in another: 12
// FP32 operations a multiply-add, one dependent addition a step, and one
// rounding at the sum's scale.  Both floats are folded in after every block's
// few terms (left to grow over a whole row their own rounding grows with the
// number of terms: first backward error of an n = 40003 solve 2.8e-8 instead
// of 9.6e-10).
template <typename T> struct Acc {
    T s = T(0);
    __device__ __forceinline__ void mac(T a, T b) { s = fma(a, b, s); }
    __device__ __forceinline__ void fold() {}
    __device__ __forceinline__ T value() const { return s; }
};
template <> struct Acc<df64> {
    float h = 0.f, l = 0.f, c = 0.f;
    __device__ __forceinline__ void mac(df64 a, df64 b)
    {
        const float p = __fmul_rn(a.hi, b.hi);
        const float pe = __fmaf_rn(a.hi, b.hi, -p);
        float s, e;
        two_sum(h, p, s, e);
        h = s;
        l = __fadd_rn(l, e);
        c = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fadd_rn(c, pe)));
    }
    __device__ __forceinline__ void fold()
    {
        fast_two_sum(h, __fadd_rn(l, c), h, l);
        c = 0.f;
    }
    __device__ __forceinline__ df64 value() const { return df_norm(h, __fadd_rn(l, c)); }
};

// ---- published values
template <typename T> struct Word {
    using type = unsigned long long;
};
template <> struct Word<float> {
    using type = unsigned int;
};
template <typename T> __device__ __forceinline__ bool unset(T v)
{
    typename Word<T>::type w;
    memcpy(&w, &v, sizeof(T));
    return w == ~(typename Word<T>::type)0;
}
// two consecutive published values (p even-indexed)
template <typename T> __device__ __forceinline__ void peek2(const T *p, T &a, T &b)
{
    if constexpr (sizeof(T) == 8) {
        unsigned long long x, y;
        asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
        memcpy(&a, &x, 8);
        memcpy(&b, &y, 8);
    } else {
        unsigned int x, y;
        asm volatile("ld.relaxed.gpu.global.v2.b32 {%0, %1}, [%2];" : "=r"(x), "=r"(y) : "l"(p) : "memory");
        memcpy(&a, &x, 4);
        memcpy(&b, &y, 4);
    }
}
template <typename T> __device__ __forceinline__ T peek1(const T *p)
{
    T a;
    if constexpr (sizeof(T) == 8) {
        unsigned long long x;
        asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(x) : "l"(p) : "memory");
        memcpy(&a, &x, 8);
    } else {
        unsigned int x;
        asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
        memcpy(&a, &x, 4);
    }
    return a;
}
template <typename T> __device__ __forceinline__ void publish(T *p, T v)
{
    if constexpr (sizeof(T) == 8) {
        unsigned long long x;
        memcpy(&x, &v, 8);
        if (x == ~0ull) x = 0x7FFFFFFF7FFFFFFFull;  // another NaN (in both halves of a pair)
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(x) : "memory");
    } else {
        unsigned int x;
        memcpy(&x, &v, 4);
        if (x == ~0u) x = 0x7FFFFFFFu;
        asm volatile("st.relaxed.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
    }
}

// A bounded wait: call after each look that found a value unset; false once
// the wait is over (the time limit, or a timeout seen from another CTA; both
// are looked at on every sixteenth call, off the chain's usual path).
struct Wait {
    unsigned long long t0 = 0;
    unsigned looks = 0;
    __device__ __forceinline__ bool go_on(int *err, long long wait_ns)
    {
        if (++looks % 16 != 0) return true;
        if (*((volatile int *)err) != 0) return false;
        const unsigned long long t = global_ns();
        if (t0 == 0) {
            t0 = t;
        } else if ((long long)(t - t0) > wait_ns) {
            atomicExch(err, 1);
            return false;
        }
        return true;
    }
};

// Inverses of the 64 x 64 diagonal blocks of the two triangles a solve uses
// (blockIdx.y = 0: L or U^T, 1: U or L^T; unit diagonal where the factor has
// one), row-major, zero outside the matrix.  Four lanes per column, entry k
// of the column on lane k mod 4: the substitution is right-looking, so its
// chain is one multiply, one shuffle and one multiply-add per row, the rest
// independent; the upper triangle is solved with both indices reversed.  A
// warp (eight columns) starts at its first column's row.  In double the
// block's 44 k multiply-adds bound it (11 us at two a clock); one thread per
// column with a left-looking sum took 60 us.
template <typename T, typename TF>
__global__ void __launch_bounds__(256) diag_inv_kernel(int64_t n, const TF *__restrict__ LU, int64_t lda, int trans,
                                                       T *__restrict__ inv, int64_t nblk)
{
    extern __shared__ __align__(16) unsigned char inv_smem[];
    typedef T Row[kTrsvNB + 1];
    Row *D = reinterpret_cast<Row *>(inv_smem);
    Row *X = D + kTrsvNB;
    T *rd = reinterpret_cast<T *>(X + kTrsvNB);
    const int tid = threadIdx.x;
    const bool lower = blockIdx.y == 0;
    const int64_t pb = blockIdx.x, r0 = pb * kTrsvNB;
    const int kb = (int)(n - r0 < kTrsvNB ? n - r0 : kTrsvNB);
    const bool unit = lower != (trans != 0);
    auto at = [&](int i) { return lower ? i : kTrsvNB - 1 - i; };  // index of the reversed block
    for (int e = tid; e < kTrsvNB * kTrsvNB; e += 256) {
        const int r = trans ? e / kTrsvNB : e % kTrsvNB, p = trans ? e % kTrsvNB : e / kTrsvNB;
        const bool in = r < kb && p < kb && (lower ? p <= r : p >= r);
        T v = T(p == r ? 1 : 0);
        if (in && !(p == r && unit))
            v = elem_as<T>(trans ? LU[(r0 + p) + (r0 + r) * lda] : LU[(r0 + r) + (r0 + p) * lda]);
        D[at(r)][at(p)] = v;
        if (p == r) rd[at(r)] = T(1) / v;
    }
    __syncthreads();
    const int c = tid / 4, q = tid % 4, gbase = tid & 28;
    T x[16];
#pragma unroll
    for (int r = 0; r < 16; r++) x[r] = T(q + 4 * r == c ? 1 : 0);
    const int first = (tid / 32) * 2;  // the warp's first column, in rows of four
    for (int i4 = 0; i4 < 16; i4++) {  // x[r] holds entry q + 4 (i4 + r)
        if (i4 >= first) {
#pragma unroll
            for (int ii = 0; ii < 4; ii++) {
                const int i = 4 * i4 + ii;
                const T xi = shfl_idx(x[0], gbase | ii) * rd[i];
                if (q == ii) x[0] = xi;
                if (q > ii) x[0] = x[0] - D[q + 4 * i4][i] * xi;
#pragma unroll
                for (int r = 1; r < 16; r++)
                    if (i4 + r < 16) x[r] = x[r] - D[q + 4 * (i4 + r)][i] * xi;
            }
        }
        X[q + 4 * i4][c] = x[0];
#pragma unroll
        for (int r = 0; r < 15; r++) x[r] = x[r + 1];
    }
    __syncthreads();
    T *out = inv + ((int64_t)blockIdx.y * nblk + pb) * kTrsvNB * kTrsvNB;
    for (int e = tid; e < kTrsvNB * kTrsvNB; e += 256) {
        const int r = e / kTrsvNB, p = e % kTrsvNB;
        out[e] = (r < kb && p < kb) ? X[at(r)][at(p)] : T(0);
    }
}

template <typename T> constexpr size_t diag_inv_smem_bytes()
{
    return (2 * kTrsvNB * (kTrsvNB + 1) + kTrsvNB) * sizeof(T);
}

// B <- (L U)^{-1} B or (L U)^{-T} B, n x nrhs, in T arithmetic with B in
// double.  xpub: the two published solutions (first triangle's, second's),
// npad x nrhs each, all ones on entry; counter: -1 on entry.
//
// Streaming, TRANS = 0: warp w takes columns 8 w .. 8 w + 7 of each block and
// lane l the rows l and l + 32 (256-byte column segments); TRANS = 1 (the
// stored block is its transpose): lane group cq = tid mod 16 takes columns
// cq + 16 v and rows tid / 16 + 16 w (128-byte segments along the stored
// columns).  Finishing: four lanes per row, combined by shuffles, so that a
// block product costs one barrier.
template <typename T, typename TF, int R, bool TRANS>
__global__ void __launch_bounds__(kTrsvThreads, 2)
trsv_chain_kernel(int64_t n, int64_t nrhs, const TF *__restrict__ LU, int64_t lda, double *B, int64_t ldb, T *xpub,
                  int64_t npad, unsigned *counter, int *err, const T *__restrict__ inv, unsigned first_task,
                  long long wait_ns)
{
    // dynamic shared memory (T): D and Di (64 x 68 each), two blocks of
    // published values, two right-hand-side blocks, the partial sums
    constexpr int NROW = TRANS ? 4 : 2, NCOL = TRANS ? 4 : 8;  // a thread's part of a block
    extern __shared__ __align__(16) unsigned char chain_smem[];
    T *D = reinterpret_cast<T *>(chain_smem);
    T *Di = D + kTrsvNB * kTrsvLd;
    T *xb = Di + kTrsvNB * kTrsvLd;           // [2][R][64]
    T *xs = xb + 2 * R * kTrsvNB;             // [2][R][64]
    T *red = xs + 2 * R * kTrsvNB;            // [NP][R][64]
    __shared__ unsigned s_task;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t nblk = npad / kTrsvNB;
    const int64_t ng = (nrhs + R - 1) / R;
    const int row4 = tid / 4, q4 = tid % 4;   // finishing: row and lane of its quad
    for (;;) {
        if (tid == 0) s_task = first_task + atomicAdd(counter, 1u) + 1u;
        __syncthreads();
        int64_t t = s_task;
        __syncthreads();
        if (t >= 2 * nblk * ng) return;
        const bool lower = t < nblk * ng;
        if (!lower) t -= nblk * ng;
        const int64_t b = t / ng, c0 = (t % ng) * R;
        const int nc = R == 1 ? 1 : (int)(nrhs - c0 < R ? nrhs - c0 : R);
        const int64_t pb = lower ? b : nblk - 1 - b;
        const int64_t r0 = pb * kTrsvNB;
        const int kb = (int)(n - r0 < kTrsvNB ? n - r0 : kTrsvNB);
        T *xout = xpub + (lower ? 0 : npad * nrhs);
        const bool unit = lower != TRANS;
        // The thread's part of the block in the columns of solve step s.  Rows
        // past the matrix read its last row (their sums are not used); the
        // columns past it, in the one partial block, are zeros.
        const TF *rowp[NROW];
#pragma unroll
        for (int i = 0; i < NROW; i++) {
            const int64_t r = r0 + (TRANS ? tid / 16 + 16 * i : lane + 32 * i);
            rowp[i] = LU + (r < n ? r : n - 1) * (TRANS ? lda : 1);
        }
        auto load_block = [&](int64_t s, TF(&m)[16]) {
            const int64_t p0 = (lower ? s : nblk - 1 - s) * kTrsvNB + (TRANS ? tid % 16 : 8 * warp);
            if (p0 / kTrsvNB * kTrsvNB + kTrsvNB <= n) {
#pragma unroll
                for (int u = 0; u < NCOL; u++) {
                    const int64_t off = TRANS ? p0 + 16 * u : (p0 + u) * lda;
#pragma unroll
                    for (int i = 0; i < NROW; i++) m[i * NCOL + u] = rowp[i][off];
                }
            } else {
#pragma unroll
                for (int u = 0; u < NCOL; u++) {
                    const int64_t p = p0 + (TRANS ? 16 * u : u);
#pragma unroll
                    for (int i = 0; i < NROW; i++)
                        m[i * NCOL + u] = p < n ? rowp[i][TRANS ? p : p * lda] : TF(0);
                }
            }
        };
        TF m[16];
        if (b > 0) load_block(0, m);
        const T *di = inv + ((lower ? 0 : nblk) + pb) * kTrsvNB * kTrsvNB;
        for (int e = tid; e < kTrsvNB * kTrsvNB; e += kTrsvThreads) {
            // only the triangle being solved with, unit diagonal where the factor has one
            const int r = TRANS ? e / kTrsvNB : e % kTrsvNB, p = TRANS ? e % kTrsvNB : e / kTrsvNB;
            T v = T(0);
            if (r < kb && p < kb && (lower ? p <= r : p >= r))
                v = (p == r && unit) ? T(1)
                                     : elem_as<T>(TRANS ? LU[(r0 + p) + (r0 + r) * lda] : LU[(r0 + r) + (r0 + p) * lda]);
            D[r * kTrsvLd + p] = v;
            Di[(e / kTrsvNB) * kTrsvLd + e % kTrsvNB] = di[e];
        }
        // the block's right-hand sides (its row on each of the quad's lanes)
        T rhs[R];
#pragma unroll
        for (int c = 0; c < R; c++) {
            rhs[c] = T(0);
            if (c < nc && row4 < kb) {
                if (lower) {
                    rhs[c] = from_double<T>(B[r0 + row4 + (c0 + c) * ldb]);
                } else {
                    const T *src = xpub + (c0 + c) * npad + r0 + row4;
                    Wait wt;
                    while (unset(rhs[c] = peek1(src)) && wt.go_on(err, wait_ns)) __nanosleep(64);
                }
            }
        }
        Acc<T> acc[NROW][R];
        // warp 0: lane l holds the published values 2 l and 2 l + 1 of the next block
        T nx[R][2];
        auto peek_block = [&](int64_t s) {
            const T *src = xout + c0 * npad + (lower ? s : nblk - 1 - s) * kTrsvNB + 2 * lane;
#pragma unroll
            for (int c = 0; c < R; c++) {
                nx[c][0] = nx[c][1] = T(0);
                if (c < nc) peek2(src + c * npad, nx[c][0], nx[c][1]);
            }
        };
        if (warp == 0 && b > 0) peek_block(0);
        for (int64_t s = 0; s < b; s++) {
            TF mn[16];
            if (s + 1 < b) load_block(s + 1, mn);
            T *x = xb + (s & 1) * R * kTrsvNB;
            if (warp == 0) {
                Wait wt;
                for (;;) {
                    bool miss = false;
#pragma unroll
                    for (int c = 0; c < R; c++) miss |= unset(nx[c][0]) | unset(nx[c][1]);
                    if (!__any_sync(0xffffffffu, miss)) break;
                    bool on = wt.go_on(err, wait_ns);
                    on = __all_sync(0xffffffffu, on);
                    if (!on) break;
                    const int64_t behind = b - 1 - s;
                    if (behind > 1) __nanosleep(behind < 16 ? 100 * (unsigned)behind : 1600);
                    peek_block(s);
                }
#pragma unroll
                for (int c = 0; c < R; c++) {
                    x[c * kTrsvNB + 2 * lane] = nx[c][0];
                    x[c * kTrsvNB + 2 * lane + 1] = nx[c][1];
                }
                if (s + 1 < b) peek_block(s + 1);
            }
            // one barrier a block: the other buffer is rewritten only after
            // every thread has passed the next one
            __syncthreads();
#pragma unroll
            for (int u = 0; u < NCOL; u++) {
                const int p = TRANS ? tid % 16 + 16 * u : 8 * warp + u;
                T xv[R];
#pragma unroll
                for (int c = 0; c < R; c++) xv[c] = x[c * kTrsvNB + p];
#pragma unroll
                for (int i = 0; i < NROW; i++) {
                    const T mv = elem_as<T>(m[i * NCOL + u]);
#pragma unroll
                    for (int c = 0; c < R; c++) acc[i][c].mac(mv, xv[c]);
                }
            }
#pragma unroll
            for (int i = 0; i < NROW; i++)
#pragma unroll
                for (int c = 0; c < R; c++) acc[i][c].fold();
#pragma unroll
            for (int e = 0; e < 16; e++) m[e] = mn[e];
        }
        // partial sums of the rows
#pragma unroll
        for (int i = 0; i < NROW; i++)
#pragma unroll
            for (int c = 0; c < R; c++) {
                T v = acc[i][c].value();
                if (TRANS) {
#pragma unroll
                    for (int o = 8; o > 0; o >>= 1) v = v + shfl_xor(v, o);
                    if (tid % 16 == 0) red[c * kTrsvNB + tid / 16 + 16 * i] = v;
                } else {
                    red[(warp * R + c) * kTrsvNB + lane + 32 * i] = v;
                }
            }
        __syncthreads();
        auto quad_sum = [](T v) {
            v = v + shfl_xor(v, 1);
            return v + shfl_xor(v, 2);
        };
#pragma unroll
        for (int c = 0; c < R; c++) {
            T v;
            if (TRANS) {
                v = red[c * kTrsvNB + row4];
            } else {
                v = quad_sum(red[(q4 * R + c) * kTrsvNB + row4] + red[((q4 + 4) * R + c) * kTrsvNB + row4]);
            }
            if (row4 < kb) rhs[c] = rhs[c] - v;
            if (q4 == 0) xs[c * kTrsvNB + row4] = rhs[c];
        }
        __syncthreads();
        auto product = [&](const T *Mx, const T *v, T(&out)[R]) {
            Acc<T> a0[R], a1[R];
#pragma unroll
            for (int u = 0; u < 16; u += 2) {
                const int p = 4 * u + q4;
                const T m0 = Mx[row4 * kTrsvLd + p], m1 = Mx[row4 * kTrsvLd + p + 4];
#pragma unroll
                for (int c = 0; c < R; c++) {
                    a0[c].mac(m0, v[c * kTrsvNB + p]);
                    a1[c].mac(m1, v[c * kTrsvNB + p + 4]);
                }
            }
#pragma unroll
            for (int c = 0; c < R; c++) out[c] = quad_sum(a0[c].value() + a1[c].value());
        };
        T x0[R], y[R];
        T *xs1 = xs + R * kTrsvNB;
        product(Di, xs, x0);  // x0 = Di r
        if (q4 == 0)
#pragma unroll
            for (int c = 0; c < R; c++) xs1[c * kTrsvNB + row4] = x0[c];
        __syncthreads();
        product(D, xs1, y);  // r - D x0
        if (q4 == 0)
#pragma unroll
            for (int c = 0; c < R; c++) xs[c * kTrsvNB + row4] = rhs[c] - y[c];
        __syncthreads();
        product(Di, xs, y);
        if (q4 == 0)
#pragma unroll
            for (int c = 0; c < R; c++)
                if (c < nc) {
                    const T v = row4 < kb ? x0[c] + y[c] : T(0);
                    publish(xout + (c0 + c) * npad + r0 + row4, v);
                    if (!lower && row4 < kb) B[r0 + row4 + (c0 + c) * ldb] = to_double(v);
                }
        __syncthreads();  // xs, red and the blocks are rewritten by the next task
    }
}

template <typename T, int R, bool TRANS> constexpr size_t chain_smem_bytes()
{
    return (2 * kTrsvNB * kTrsvLd + 4 * R * kTrsvNB + (TRANS ? 1 : 8) * R * kTrsvNB) * sizeof(T);
}

// Scratch of a solve: [0] timeout flag (cleared by the public entry point or
// the solve driver, once per call: it stays set across the refinement steps
// of one call); from byte 256 the part set to all ones before each launch
// (task counter, then the published solutions); then the inverses.
struct ChainScratch {
    int *err;
    unsigned *counter;
    void *xpub, *inv;
    size_t ones_bytes, total;
    int64_t nblk, npad;
};

static ChainScratch carve_chain(int64_t n, int64_t nrhs, size_t es, void *scratch)
{
    ChainScratch s;
    char *w = (char *)scratch;
    s.nblk = cdiv(n > 0 ? n : 1, kTrsvNB);
    s.npad = s.nblk * kTrsvNB;
    s.err = (int *)w;
    // published values are read two at a time, 16 bytes: the rest starts on such
    // a boundary wherever the caller's buffer does (at most 12 bytes on, out of
    // the 256 that chain_scratch_bytes adds)
    w = (char *)(((uintptr_t)w + 15) / 16 * 16);
    s.counter = (unsigned *)(w + 256);
    s.xpub = w + 512;
    s.ones_bytes = 256 + 2 * (size_t)s.npad * (size_t)(nrhs > 0 ? nrhs : 1) * es;
    const size_t at = (256 + s.ones_bytes + 255) / 256 * 256;
    s.inv = w + at;
    s.total = at + 2 * (size_t)s.nblk * kTrsvNB * kTrsvNB * es;
    return s;
}

static size_t chain_scratch_bytes(int64_t n, int64_t nrhs, size_t es)
{
    return carve_chain(n, nrhs, es, nullptr).total + 256;
}

template <typename T, typename TF, int R, bool TRANS>
static rbt_status launch_chain(int64_t n, int64_t nrhs, const TF *LU, int64_t lda, double *B, int64_t ldb,
                               const ChainScratch &s, cudaStream_t stream)
{
    static PerDeviceOnce once;
    static std::atomic<int> per_sm_known{0};
    constexpr size_t smem = chain_smem_bytes<T, R, TRANS>();
    rbt_status st = smem_opt_in(once, trsv_chain_kernel<T, TF, R, TRANS>, (int)smem);
    if (st != RBT_OK) return st;
    int per_sm = per_sm_known.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        RBT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, trsv_chain_kernel<T, TF, R, TRANS>,
                                                                   kTrsvThreads, smem));
        per_sm = per_sm > 0 ? per_sm : 1;
        per_sm_known.store(per_sm, std::memory_order_relaxed);
    }
    const int64_t ng = cdiv(nrhs, R);
    const int64_t grid = std::min<int64_t>((int64_t)device_sm_count() * per_sm, 2 * s.nblk * ng);
    // the test stall starts the queue past block 0, which is then never solved
    const unsigned first = debug_stall() == RBT_STALL_CHAIN ? (unsigned)ng : 0u;
    trsv_chain_kernel<T, TF, R, TRANS><<<(unsigned)grid, kTrsvThreads, smem, stream>>>(
        n, nrhs, LU, lda, B, ldb, (T *)s.xpub, s.npad, s.counter, s.err, (const T *)s.inv, first, wait_limit_ns());
    RBT_LAUNCH_CHECK();
    return RBT_OK;
}

// Right-hand sides per task.  A step of the chain gets longer with R (four
// block products per right-hand side), the factors are read fewer times, and
// the chains of different groups run side by side: R = 1 is fastest until
// the n^2 nrhs multiply-adds, not the 2 n / 64 steps, decide.  Both costs
// grow alike in n, so the lines lie at n nrhs.  Microseconds per solve, GB300:
//   pairs   n = 8197:  16 rhs 1598 (R = 1) / 1780 (2);   32 rhs 2810 / 2266
//           n = 20001:  8 rhs 4512 / 4658;               16 rhs 7915 / 6429
//   float   n = 8197:   4 rhs 418 / 459 / 644 (R = 4);   16 rhs 1017 / 658 / 692
//           n = 4001:  32 rhs 417 / 290 / 352;           64 rhs 744 / 449 / 384
//           n = 4001:  256 / 1024 rhs 1021 / 3421 at R = 4 (blocked sweep 30.7 / 118.8 ms;
//                      pairs 3.7 / 14.2, sweep 99 / 386 ms)
// In double the FP64 pipe is the bound either way (32 rhs at n = 8197: 4610 /
// 5488): always one.  Pairs with R = 4 would spill.
template <typename T, typename TF, bool TRANS>
static rbt_status run_chain(int64_t n, int64_t nrhs, const TF *LU, int64_t lda, double *B, int64_t ldb,
                            const ChainScratch &s, cudaStream_t stream)
{
    if constexpr (std::is_same<T, float>::value) {
        if (n * nrhs > 200000) return launch_chain<T, TF, 4, TRANS>(n, nrhs, LU, lda, B, ldb, s, stream);
        if (n * nrhs > 60000) return launch_chain<T, TF, 2, TRANS>(n, nrhs, LU, lda, B, ldb, s, stream);
    } else if constexpr (std::is_same<T, df64>::value) {
        if (n * nrhs > 200000) return launch_chain<T, TF, 2, TRANS>(n, nrhs, LU, lda, B, ldb, s, stream);
    }
    return launch_chain<T, TF, 1, TRANS>(n, nrhs, LU, lda, B, ldb, s, stream);
}

template <typename T, typename TF>
static rbt_status lu_solve_chain(int64_t n, int64_t nrhs, const TF *LU, int64_t lda, int trans, double *B,
                                 int64_t ldb, void *scratch, bool have_inv, cudaStream_t stream)
{
    ProfScope ps(kProfSolve, stream);
    const ChainScratch s = carve_chain(n, nrhs, sizeof(T), scratch);
    if (!have_inv) {
        static PerDeviceOnce once;
        rbt_status st = smem_opt_in(once, diag_inv_kernel<T, TF>, (int)diag_inv_smem_bytes<T>());
        if (st != RBT_OK) return st;
        diag_inv_kernel<T, TF><<<dim3((unsigned)s.nblk, 2), 256, diag_inv_smem_bytes<T>(), stream>>>(
            n, LU, lda, trans, (T *)s.inv, s.nblk);
        RBT_LAUNCH_CHECK();
    }
    RBT_CUDA_TRY(cudaMemsetAsync(s.counter, 0xff, s.ones_bytes, stream));
    return trans ? run_chain<T, TF, true>(n, nrhs, LU, lda, B, ldb, s, stream)
                 : run_chain<T, TF, false>(n, nrhs, LU, lda, B, ldb, s, stream);
}

// genp_solve / genp_solve_wp after validation, without clearing the timeout
// flag at the front of work (the caller owns its lifetime).  have_inv: work
// still holds the inverses of an earlier call with the same factors,
// precision, orientation, nrhs and entry point.
rbt_status genp_solve_run(int64_t n, int64_t nrhs, int32_t prec, const void *LU, int64_t lda, int32_t trans,
                          double *B, int64_t ldb, void *work, bool have_inv, cudaStream_t stream)
{
    if (n == 0 || nrhs == 0) return RBT_OK;
    const int t = trans ? 1 : 0;
    if (prec == RBT_F64)
        return lu_solve_chain<double, double>(n, nrhs, (const double *)LU, lda, t, B, ldb, work, have_inv, stream);
    if (is_df64_storage(prec))
        return lu_solve_chain<df64, df64>(n, nrhs, (const df64 *)LU, lda, t, B, ldb, work, have_inv, stream);
    return lu_solve_chain<float, float>(n, nrhs, (const float *)LU, lda, t, B, ldb, work, have_inv, stream);
}

// In double arithmetic with factors stored in a lower precision: each entry
// is widened as it is read, so the solve reads the factors' own bytes and the
// only error beyond the factors' is that of a double substitution.
rbt_status genp_solve_wp_run(int64_t n, int64_t nrhs, int32_t prec, const void *LU, int64_t lda, int32_t trans,
                             double *B, int64_t ldb, void *work, bool have_inv, cudaStream_t stream)
{
    if (n == 0 || nrhs == 0) return RBT_OK;
    const int t = trans ? 1 : 0;
    if (prec == RBT_F64)
        return lu_solve_chain<double, double>(n, nrhs, (const double *)LU, lda, t, B, ldb, work, have_inv, stream);
    if (is_df64_storage(prec))
        return lu_solve_chain<double, df64>(n, nrhs, (const df64 *)LU, lda, t, B, ldb, work, have_inv, stream);
    return lu_solve_chain<double, float>(n, nrhs, (const float *)LU, lda, t, B, ldb, work, have_inv, stream);
}

}  // namespace rbt

using namespace rbt;

extern "C" {

size_t genp_solve_workspace(int64_t n, int64_t nrhs, int32_t prec)
{
    if (n <= 0 || nrhs <= 0) return 0;
    return chain_scratch_bytes(n, nrhs, prec == RBT_F64 || is_df64_storage(prec) ? 8 : 4);
}

// Solve flag at the front of the workspace: nonzero after a call whose chained
// triangular solve gave up waiting (the result is then undefined).  The public
// calls clear it on entry; the *_run forms (the solve driver's) never clear it,
// so that one timeout stays visible for the rest of the driver's call.
rbt_status genp_solve(int64_t n, int64_t nrhs, int32_t prec, const void *LU, int64_t lda, int32_t trans,
                      double *B, int64_t ldb, void *work, size_t work_bytes, cudaStream_t stream)
{
    if (n < 0 || nrhs < 0 || prec < RBT_F64 || prec > kLastPrec) return RBT_ERR_ARG;
    if (lda < (n > 1 ? n : 1) || ldb < (n > 1 ? n : 1)) return RBT_ERR_ARG;
    if (n == 0 || nrhs == 0) return RBT_OK;
    if (!LU || !B) return RBT_ERR_ARG;
    if (work_bytes < genp_solve_workspace(n, nrhs, prec) || !work) return RBT_ERR_WORKSPACE;
    RBT_CUDA_TRY(cudaMemsetAsync(work, 0, sizeof(int), stream));
    return genp_solve_run(n, nrhs, prec, LU, lda, trans, B, ldb, work, false, stream);
}

size_t genp_solve_wp_workspace(int64_t n, int64_t nrhs)
{
    if (n <= 0 || nrhs <= 0) return 0;
    return chain_scratch_bytes(n, nrhs, sizeof(double));
}

rbt_status genp_solve_wp(int64_t n, int64_t nrhs, int32_t prec, const void *LU, int64_t lda, int32_t trans,
                         double *B, int64_t ldb, void *work, size_t work_bytes, cudaStream_t stream)
{
    if (n < 0 || nrhs < 0 || prec < RBT_F64 || prec > kLastPrec) return RBT_ERR_ARG;
    if (lda < (n > 1 ? n : 1) || ldb < (n > 1 ? n : 1)) return RBT_ERR_ARG;
    if (n == 0 || nrhs == 0) return RBT_OK;
    if (!LU || !B) return RBT_ERR_ARG;
    if (work_bytes < genp_solve_wp_workspace(n, nrhs) || !work) return RBT_ERR_WORKSPACE;
    RBT_CUDA_TRY(cudaMemsetAsync(work, 0, sizeof(int), stream));
    return genp_solve_wp_run(n, nrhs, prec, LU, lda, trans, B, ldb, work, false, stream);
}

}  // extern "C"
