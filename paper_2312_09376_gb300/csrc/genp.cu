// Gaussian elimination with no pivoting (sm_103a); its triangular solves are in
// trsv.cu.
//
// Blocked right-looking LU without row exchanges (Sec. 1; the GENP step of
// Eq. precond).  Without pivoting the diagonal block needs nothing from the
// rows below it, so each block step is
//   1. factor the kb x kb diagonal block in shared memory (one CTA),
//   2. U12 <- L11^{-1} A12 and L21 <- A21 U11^{-1} (independent columns /
//      rows, both at once),
//   3. A22 <- A22 - L21 U12 (the dense contraction: all but O(n^2 kb) of the
//      2n^3/3 flops).
// Step 3 runs on the tensor cores for the TF32 / BF16 precisions (gemm_tc.cu)
// and as a register-tiled SIMT kernel for double and float.
//
// Pivot status: d_info starts at -1.  The diagonal kernel writes the global
// index of the first pivot that is zero or not finite and stops; every later
// kernel of the factorization reads d_info first and returns at once when it
// is set, so the enqueued remainder costs almost nothing.
#include "common.cuh"
#include "genp_internal.cuh"
#include "df64.cuh"
#include "oz_slice.cuh"

#include <type_traits>

namespace rbt {

__device__ __forceinline__ bool info_set(const int64_t *info)
{
    return *((volatile const int64_t *)info) >= 0;
}

template <typename T> __device__ __forceinline__ bool bad_pivot(T p)
{
    return p == T(0) || !isfinite(p);
}

// ---------------------------------------------------------------- diagonal

// Unblocked Doolittle on the kb x kb block at (k0, k0); kb <= kMaxNB.  256
// threads: thread (i0, q) = (tid % 64, tid / 64) updates rows i0 + 64 r in
// the columns c = q (mod 4), so each elimination step is one barrier and a
// quarter row of independent multiply-adds per row of the thread.  The
// multipliers l_ij are kept in registers and stored into column j during the
// next step, when no thread reads column j any more.
template <typename T>
__global__ void __launch_bounds__(256) diag_factor_kernel(int64_t k0, int kb, T *A, int64_t lda, int64_t *info)
{
    constexpr int RPT = kMaxNB / 64;  // rows per thread
    extern __shared__ unsigned char smem_raw[];
    T *a = reinterpret_cast<T *>(smem_raw);  // kb x kb, column-major, ld = kb
    if (info_set(info)) return;
    const int tid = threadIdx.x, nt = blockDim.x;
    for (int e = tid; e < kb * kb; e += nt) {
        int i = e % kb, j = e / kb;
        a[e] = A[(k0 + i) + (k0 + j) * lda];
    }
    __syncthreads();
    const int i0 = tid % 64, q = tid / 64;
    T pend[RPT];
    int pend_j = -1;
    for (int j = 0; j < kb; j++) {
        const T p = a[j + j * kb];
        if (bad_pivot(p)) {  // every thread reads the same pivot: a uniform exit
            if (tid == 0) *info = k0 + j;
            break;
        }
        if (pend_j >= 0) {
#pragma unroll
            for (int r = 0; r < RPT; r++) {
                const int i = i0 + 64 * r;
                if (i > pend_j && i < kb) a[i + pend_j * kb] = pend[r];
            }
            pend_j = -1;
        }
        const int c0 = j + 1 + ((q - (j + 1)) & 3);
#pragma unroll
        for (int r = 0; r < RPT; r++) {
            const int i = i0 + 64 * r;
            if (i > j && i < kb) {
                const T l = a[i + j * kb] / p;
                for (int c = c0; c < kb; c += 4) a[i + c * kb] -= l * a[j + c * kb];
                pend[r] = l;
            }
        }
        if (q == 0) pend_j = j;
        __syncthreads();
    }
    if (pend_j >= 0) {
#pragma unroll
        for (int r = 0; r < RPT; r++) {
            const int i = i0 + 64 * r;
            if (i > pend_j && i < kb) a[i + pend_j * kb] = pend[r];
        }
    }
    __syncthreads();
    // write back (the partial factor too when stopped: the caller ignores it)
    for (int e = tid; e < kb * kb; e += nt) {
        int ii = e % kb, jj = e / kb;
        A[(k0 + ii) + (k0 + jj) * lda] = a[e];
    }
}

// ------------------------------------------------------------------ TRSMs

// Both TRSMs of a panel step in one launch, four lanes per vector:
//   blocks [0, nbu):        U12 <- L11^{-1} A12, a vector is a column of A12
//                           (unit forward substitution, x_i = a_i - sum_{p<i} L_ip x_p);
//   blocks [nbu, nbu+nbl):  L21 <- A21 U11^{-1}, a vector is a row of A21
//                           (x_j = (a_j - sum_{p<j} x_p U_pj) / U_jj).
// 64 vectors per CTA, vector v on lanes 4 v' .. 4 v' + 3 of one warp; lane q
// owns the entries i = q (mod 4) of its vector.  The substitution is
// right-looking in blocks of four entries: the four lanes finish entries
// j0 .. j0 + 3 (lane q the entry j0 + q: scale by the reciprocal of the
// pivot, broadcast by shuffle, the later lanes subtract it), then every lane
// subtracts the four new values from each entry it owns past the block.
// The serial part of a block is four scalings and shuffles; the rest are
// independent multiply-adds (the panel has only (n - k) / 64 CTAs of work).
constexpr int kTrsmVec = 64, kTrsmLanes = 4, kTrsmThreads = kTrsmVec * kTrsmLanes;
// padded shared-memory strides: the four lanes of a vector read the diagonal
// block at i, i+1, i+2, i+3 and the vector's entries at the same offsets;
// ld kb + 1 for the block and 68 for the vectors keep them off one bank
constexpr int kTrsmXS = kTrsmVec + 4;
template <typename T> constexpr size_t trsm_smem_bytes(int kb)
{
    return ((size_t)kb * (kb + 1) + (size_t)kb * kTrsmXS + (size_t)kb) * sizeof(T);
}

template <typename T>
__global__ void __launch_bounds__(kTrsmThreads) trsm_panel_kernel(int64_t k0, int kb, int64_t n, T *A, int64_t lda,
                                                                  int nbu, const int64_t *info)
{
    extern __shared__ unsigned char smem_raw[];
    const int ldm = kb + 1;
    T *Mt = reinterpret_cast<T *>(smem_raw);  // kb x kb diagonal block (ld kb + 1)
    T *X = Mt + kb * ldm;                      // kb x 64, X[e * kTrsmXS + v]
    T *rd = X + kb * kTrsmXS;                  // 1 / U_jj (the L21 part)
    if (info_set(info)) return;
    const int tid = threadIdx.x;
    const int q = tid % kTrsmLanes, v = tid / kTrsmLanes;
    const bool upper = (int)blockIdx.x < nbu;  // the U12 part
    const int64_t v0 = k0 + kb + (int64_t)(upper ? blockIdx.x : blockIdx.x - nbu) * kTrsmVec;
    for (int e = tid; e < kb * kb; e += kTrsmThreads) {
        const int i = e % kb, j = e / kb;
        Mt[i + j * ldm] = A[(k0 + i) + (k0 + j) * lda];
    }
    // coalesced tile load: consecutive threads walk down a column of A
    for (int e = tid; e < kb * kTrsmVec; e += kTrsmThreads) {
        if (upper) {
            const int i = e % kb, c = e / kb;
            const int64_t col = v0 + c;
            X[i * kTrsmXS + c] = col < n ? A[(k0 + i) + col * lda] : T(0);
        } else {
            const int r = e % kTrsmVec, j = e / kTrsmVec;
            const int64_t row = v0 + r;
            X[j * kTrsmXS + r] = row < n ? A[row + (k0 + j) * lda] : T(0);
        }
    }
    __syncthreads();
    if (!upper) {
        for (int j = tid; j < kb; j += kTrsmThreads) rd[j] = T(1) / Mt[j + j * ldm];
        __syncthreads();
    }
    // m(i, j): the factor entry that couples entry j into entry i
    auto coef = [&](int i, int j) { return upper ? Mt[i + j * ldm] : Mt[j + i * ldm]; };
    const int gbase = (tid & 31) & ~(kTrsmLanes - 1);  // first lane of this vector's group
    for (int j0 = 0; j0 < kb; j0 += kTrsmLanes) {
        const int jn = kb - j0 < kTrsmLanes ? kb - j0 : kTrsmLanes;  // the same on every lane
        T own = q < jn ? X[(j0 + q) * kTrsmXS + v] : T(0);
        T xs[kTrsmLanes];
#pragma unroll
        for (int jj = 0; jj < kTrsmLanes; jj++) {
            xs[jj] = T(0);
            if (jj < jn) {
                T x = own;
                if (!upper && q == jj) x = x * rd[j0 + jj];
                if (q == jj) own = x;
                x = shfl_idx(x, gbase | jj);
                xs[jj] = x;
                if (q > jj && q < jn) own = own - coef(j0 + q, j0 + jj) * x;
            }
        }
        if (q < jn) X[(j0 + q) * kTrsmXS + v] = own;
        if (jn == kTrsmLanes) {
            for (int i = j0 + kTrsmLanes + q; i < kb; i += kTrsmLanes) {
                T a = X[i * kTrsmXS + v];
#pragma unroll
                for (int jj = 0; jj < kTrsmLanes; jj++) a = a - coef(i, j0 + jj) * xs[jj];
                X[i * kTrsmXS + v] = a;
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < kb * kTrsmVec; e += kTrsmThreads) {
        if (upper) {
            const int i = e % kb, c = e / kb;
            const int64_t col = v0 + c;
            if (col < n) A[(k0 + i) + col * lda] = X[i * kTrsmXS + c];
        } else {
            const int r = e % kTrsmVec, j = e / kTrsmVec;
            const int64_t row = v0 + r;
            if (row < n) A[row + (k0 + j) * lda] = X[j * kTrsmXS + r];
        }
    }
}

// ------------------------------------------- blocks of at most 64 columns
//
// A multiply-subtract of the elimination.  In double-float the sum is
// renormalized but not the product (15 operations instead of 19);
// renormalizing only every fourth one (12) makes unrefined backward errors two
// to three times larger.
constexpr int kP = 64;  // columns of a block
constexpr int kQ = 16;  // columns of a panel inside it

template <typename T> __device__ __forceinline__ void sub_mul(T &a, T c, T x) { a = fma(-c, x, a); }
template <> __device__ __forceinline__ void sub_mul<df64>(df64 &a, df64 c, df64 x)
{
    const float p = __fmul_rn(-c.hi, x.hi);
    const float pe = __fmaf_rn(-c.hi, x.hi, -p);
    float s, e;
    two_sum(a.hi, p, s, e);
    a = df_norm(s, __fadd_rn(e, __fadd_rn(a.lo, __fmaf_rn(-c.lo, x.hi, __fmaf_rn(-c.hi, x.lo, pe)))));
}

// N independent ones, a[i] -= c[i] x, written stage by stage: each stage's
// operations are independent, where one entry after the other leaves the
// instruction order a single dependent chain.
template <int N, typename T> __device__ __forceinline__ void sub_mul_n(T (&a)[N], const T (&c)[N], T x)
{
#pragma unroll
    for (int i = 0; i < N; i++) a[i] = fma(-c[i], x, a[i]);
}
template <int N> __device__ __forceinline__ void sub_mul_n(df64 (&a)[N], const df64 (&c)[N], df64 x)
{
    float p[N], l[N], s[N], b[N], u[N];
#pragma unroll
    for (int i = 0; i < N; i++) p[i] = __fmul_rn(-c[i].hi, x.hi);
#pragma unroll
    for (int i = 0; i < N; i++) l[i] = __fmaf_rn(-c[i].hi, x.hi, -p[i]);
#pragma unroll
    for (int i = 0; i < N; i++) s[i] = __fadd_rn(a[i].hi, p[i]);
#pragma unroll
    for (int i = 0; i < N; i++) l[i] = __fmaf_rn(-c[i].hi, x.lo, l[i]);
#pragma unroll
    for (int i = 0; i < N; i++) b[i] = __fsub_rn(s[i], a[i].hi);
#pragma unroll
    for (int i = 0; i < N; i++) l[i] = __fmaf_rn(-c[i].lo, x.hi, l[i]);
#pragma unroll
    for (int i = 0; i < N; i++) u[i] = __fsub_rn(s[i], b[i]);
#pragma unroll
    for (int i = 0; i < N; i++) p[i] = __fsub_rn(p[i], b[i]);
#pragma unroll
    for (int i = 0; i < N; i++) u[i] = __fsub_rn(a[i].hi, u[i]);
#pragma unroll
    for (int i = 0; i < N; i++) l[i] = __fadd_rn(a[i].lo, l[i]);
#pragma unroll
    for (int i = 0; i < N; i++) u[i] = __fadd_rn(u[i], p[i]);
#pragma unroll
    for (int i = 0; i < N; i++) l[i] = __fadd_rn(u[i], l[i]);
#pragma unroll
    for (int i = 0; i < N; i++) a[i].hi = __fadd_rn(s[i], l[i]);
#pragma unroll
    for (int i = 0; i < N; i++) s[i] = __fsub_rn(a[i].hi, s[i]);
#pragma unroll
    for (int i = 0; i < N; i++) a[i].lo = __fsub_rn(l[i], s[i]);
}

// a / p from r, an approximate reciprocal of p (of its leading part in
// double-float): the quotient's residual is taken once more (as in a division
// by Newton's iteration), so a step costs one reciprocal and the quotients a
// few multiply-adds each, at the accuracy of the division.  Pivots near the
// ends of the exponent range take the division itself.
__device__ __forceinline__ bool mid_range(double p) { return fabs(p) > 1e-30 && fabs(p) < 1e30; }
__device__ __forceinline__ bool mid_range(float p) { return fabsf(p) > 1e-30f && fabsf(p) < 1e30f; }
__device__ __forceinline__ bool mid_range(df64 p) { return mid_range(p.hi); }
template <typename T> __device__ __forceinline__ T recip(T p);
template <> __device__ __forceinline__ float recip<float>(float p) { return __frcp_rn(p); }
template <> __device__ __forceinline__ df64 recip<df64>(df64 p) { return df64(__frcp_rn(p.hi)); }
// a float's reciprocal and one Newton step (2^-46): the FP64 pipe's operations
// are the chain's long ones, and the quotient's residual step follows anyway
template <> __device__ __forceinline__ double recip<double>(double p)
{
    const double r = (double)__frcp_rn((float)p);
    return ::fma(r, ::fma(-p, r, 1.0), r);
}
template <typename T> __device__ __forceinline__ T quotient(T a, T p, T r, bool mid)
{
    if (!mid) return a / p;
    const T l = a * r;
    return fma(fma(-l, p, a), r, l);
}
template <> __device__ __forceinline__ df64 quotient<df64>(df64 a, df64 p, df64 r, bool mid)
{
    if (!mid) return a / p;
    const float q = __fmul_rn(a.hi, r.hi);
    const float t = __fmaf_rn(-q, p.hi, a.hi);  // exact: q p.hi agrees with a.hi to a few units
    const float d = __fmaf_rn(-q, p.lo, __fadd_rn(t, a.lo));
    return df_norm(q, __fmul_rn(d, r.hi));
}

// Diagonal block (kb <= 64): one CTA, four lanes per row, in panels of 16
// columns.  Inside a panel a step is the pivot row's at most 16 entries
// published through shared memory with the pivot's reciprocal, one barrier, a
// quotient and at most four multiply-subtracts a lane: the chain of 64 steps
// is what the kernel costs, so nothing else is on it.  Then the panel's rows
// of the columns to the right (a 16-step substitution, four lanes a column)
// and the rank-16 update of the rest (up to 12 independent entries a lane).
template <typename T>
__global__ void __launch_bounds__(256, 1) diag64_kernel(int64_t k0, int kb, T *A, int64_t lda, int64_t *info)
{
    constexpr int LD = kP + 1;
    __shared__ T S[kP * LD];  // the block, row-major
    __shared__ T urow[2][kQ];
    __shared__ T piv[2][2];
    if (info_set(info)) return;
    const int tid = threadIdx.x, i = tid / 4, q = tid % 4, gbase = tid & 28;
    for (int e = tid; e < kP * kP; e += 256) {
        const int r = e % kP, c = e / kP;
        S[r * LD + c] = (r < kb && c < kb) ? A[(k0 + r) + (k0 + c) * lda] : T(0);
    }
    __syncthreads();
    bool stop = false;
    for (int c0 = 0; c0 < kb && !stop; c0 += kQ) {
        T a[4];
#pragma unroll
        for (int r = 0; r < 4; r++) a[r] = S[i * LD + c0 + q + 4 * r];
#pragma unroll
        for (int jj = 0; jj < kQ; jj++) {
            const int j = c0 + jj;
            if (stop || j >= kb) continue;  // the same in every thread
            T *u = urow[jj & 1], *pv = piv[jj & 1];
            if (i == j) {
                if (q == jj % 4) {
                    pv[0] = a[jj / 4];
                    pv[1] = recip(a[jj / 4]);
                }
#pragma unroll
                for (int r = jj / 4; r < 4; r++) u[q + 4 * r] = a[r];
            }
            __syncthreads();
            const T p = pv[0];
            if (bad_pivot(p)) {  // every thread reads the same pivot: a uniform exit
                if (tid == 0) *info = k0 + j;
                stop = true;
                continue;
            }
            if ((i | 7) > j) {  // some row of the warp is below the pivot
                const T l = quotient(shfl_idx(a[jj / 4], gbase | (jj % 4)), p, pv[1], mid_range(p));
                if (i > j) {
                    T w[4], v[4];
#pragma unroll
                    for (int r = 0; r < 4; r++) {
                        w[r] = a[r];
                        v[r] = u[q + 4 * r];
                    }
                    sub_mul_n(w, v, l);
                    if (q > jj % 4) a[jj / 4] = w[jj / 4];
                    if (q == jj % 4) a[jj / 4] = l;
#pragma unroll
                    for (int r = jj / 4 + 1; r < 4; r++) a[r] = w[r];
                }
            }
        }
        if (i >= c0)
#pragma unroll
            for (int r = 0; r < 4; r++) S[i * LD + c0 + q + 4 * r] = a[r];
        __syncthreads();
        const int c1 = c0 + kQ;
        if (c1 >= kb || stop) continue;
        // rows c0 .. c1 - 1 of the columns right of the panel
        if (i < kP - c1) {
            const int c = c1 + i;
#pragma unroll
            for (int r = 0; r < 4; r++) a[r] = S[(c0 + q + 4 * r) * LD + c];
#pragma unroll
            for (int jj = 0; jj < kQ; jj++) {
                const T x = shfl_idx(a[jj / 4], gbase | (jj % 4));
                T w[4], l[4];
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    w[r] = a[r];
                    l[r] = S[(c0 + q + 4 * r) * LD + c0 + jj];
                }
                sub_mul_n(w, l, x);
                if (q > jj % 4) a[jj / 4] = w[jj / 4];
#pragma unroll
                for (int r = jj / 4 + 1; r < 4; r++) a[r] = w[r];
            }
#pragma unroll
            for (int r = 0; r < 4; r++) S[(c0 + q + 4 * r) * LD + c] = a[r];
        }
        __syncthreads();
        // the rest: rows and columns from c1 on
        if (i >= c1) {
            const int nc = (kP - c1) / 4;  // 12, 8 or 4 columns a lane
            for (int g = 0; g < nc; g += 4) {
                const int cg = c1 + q + 4 * g;
                T w[4], u[4];
#pragma unroll
                for (int r = 0; r < 4; r++) w[r] = S[i * LD + cg + 4 * r];
#pragma unroll 4
                for (int k = 0; k < kQ; k++) {
#pragma unroll
                    for (int r = 0; r < 4; r++) u[r] = S[(c0 + k) * LD + cg + 4 * r];
                    sub_mul_n(w, u, S[i * LD + c0 + k]);
                }
#pragma unroll
                for (int r = 0; r < 4; r++) S[i * LD + cg + 4 * r] = w[r];
            }
        }
        __syncthreads();
    }
    __syncthreads();
    // write back (the partial factor too when stopped: the caller ignores it)
    for (int e = tid; e < kP * kP; e += 256) {
        const int r = e % kP, c = e / kP;
        if (r < kb && c < kb) A[(k0 + r) + (k0 + c) * lda] = S[r * LD + c];
    }
}

// Both TRSMs of a step, U12 <- L11^{-1} A12 (blocks [0, nbu), a vector is a
// column) and L21 <- A21 U11^{-1} (the other blocks, a vector is a row): the
// substitution runs right-looking down each vector, VEC vectors per CTA on
// LANES lanes each (lane q holds the entries q + LANES r in registers), the
// block's coefficients in shared memory.  Each thread carries NV vectors, so
// that a coefficient read serves NV multiply-subtracts (with one, the
// shared-memory reads bound the double-float kernel).  The loop runs LANES
// steps at a time and then moves each lane's entries down by one register,
// which makes the finished ones a[0] (a fixed register) without unrolling all
// 64 steps; entries past the block's end are skipped four at a time (a test of
// each would leave no independent instructions to interleave).  Entries come
// and go without staging.  kmax, when given, receives the exponents that
// balance the sliced updates (gemm_oz.cu): for each k the largest over the
// panel's own rows, the rows below it, its columns, and the columns right of
// it, each in an array of kKmax ints.
template <typename T, int VEC, int LANES, int NV>
__global__ void __launch_bounds__(VEC * LANES / NV)
trsm64_kernel(int64_t k0, int kb, int64_t n, T *A, int64_t lda, int nbu, const int64_t *info, int64_t panel_end,
              int *kmax)
{
    constexpr int E = kP / LANES, NT = VEC * LANES / NV;
    // M(k, j), the entry that couples j into k, at k + 65 j (past the last
    // column: read with the last entries' groups, never used)
    __shared__ T Mt[kP * (kP + 1) + kP];
    __shared__ T rd[kP];
    __shared__ int kx[kP];
    if (info_set(info)) return;
    const int tid = threadIdx.x, q = tid % LANES, gbase = tid & 31 & ~(LANES - 1);
    const bool upper = (int)blockIdx.x < nbu;
    const int64_t first = k0 + kb + (int64_t)(upper ? blockIdx.x : blockIdx.x - nbu) * VEC;
    const int64_t es = upper ? 1 : lda;
    T a[NV][E];
    T *base[NV];  // entry e at base[e * es]
    bool in[NV];
#pragma unroll
    for (int w = 0; w < NV; w++) {
        const int64_t v = first + tid / LANES + w * (VEC / NV);
        in[w] = v < n;
        base[w] = upper ? A + k0 + v * lda : A + v + k0 * lda;
#pragma unroll
        for (int r = 0; r < E; r++)
            a[w][r] = (in[w] && q + LANES * r < kb) ? base[w][(q + LANES * r) * es] : T(0);
    }
    for (int e = tid; e < kP * kP; e += NT) {
        const int i = e % kP, j = e / kP;
        const T m = (i < kb && j < kb) ? A[(k0 + i) + (k0 + j) * lda] : T(0);
        Mt[upper ? i + j * (kP + 1) : j + i * (kP + 1)] = m;
    }
    for (int j = tid; j < kP; j += NT) {
        rd[j] = (j < kb && !upper) ? T(1) / A[(k0 + j) + (k0 + j) * lda] : T(1);
        kx[j] = kNoExp;
    }
    __syncthreads();
    for (int jb = 0; LANES * jb < kb; jb++) {
#pragma unroll
        for (int jj = 0; jj < LANES; jj++) {
            const int j = LANES * jb + jj;
            const T *m = Mt + j * (kP + 1) + q + LANES * jb;
            T x[NV];
#pragma unroll
            for (int w = 0; w < NV; w++) {
                if (q == jj && !upper) a[w][0] = a[w][0] * rd[j];
                x[w] = shfl_idx(a[w][0], gbase | jj);
                if (q > jj) sub_mul(a[w][0], m[0], x[w]);
            }
#pragma unroll
            for (int g = 1; g < E; g += 4)
                if (jb + g < E) {
                    constexpr int G = 4;
                    T c[G];
#pragma unroll
                    for (int r = 0; r < G; r++) c[r] = g + r < E ? m[LANES * (g + r)] : T(0);
#pragma unroll
                    for (int w = 0; w < NV; w++) {
                        T v[G];
#pragma unroll
                        for (int r = 0; r < G; r++) v[r] = g + r < E ? a[w][g + r] : T(0);
                        sub_mul_n(v, c, x[w]);
#pragma unroll
                        for (int r = 0; r < G; r++)
                            if (g + r < E) a[w][g + r] = v[r];
                    }
                }
        }
        const int c = q + LANES * jb;
        int e = kNoExp;
#pragma unroll
        for (int w = 0; w < NV; w++)
            if (in[w] && c < kb) {
                base[w][c * es] = a[w][0];
                e = max(e, finite_exp(exp_of(a[w][0])));
            }
        if (kmax) {
#pragma unroll
            for (int o = LANES; o < 32; o <<= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
            if ((tid & 31) < LANES && e > kNoExp) atomicMax(kx + c, e);
        }
#pragma unroll
        for (int w = 0; w < NV; w++)
#pragma unroll
            for (int r = 0; r + 1 < E; r++) a[w][r] = a[w][r + 1];
    }
    if (kmax) {
        __syncthreads();
        // first is at a distance from k0 + kb that VEC divides, and the panel's
        // end at one that 64 divides: a CTA's vectors lie on one side of it
        int *to = kmax + (upper ? 2 : 0) * kKmax + (first < panel_end ? 0 : kKmax);
        for (int j = tid; j < kb; j += NT)
            if (kx[j] > kNoExp) atomicMax(to + j, kx[j]);
    }
}

template <typename T, int VEC, int LANES, int NV>
static void launch_trsm64(int64_t k, int kb, int64_t n, T *A, int64_t lda, const int64_t *info, int64_t panel_end,
                          int *kmax, cudaStream_t stream)
{
    const int nbv = (int)cdiv(n - k - kb, VEC);
    trsm64_kernel<T, VEC, LANES, NV><<<(unsigned)(2 * nbv), VEC * LANES / NV, 0, stream>>>(k, kb, n, A, lda, nbv, info,
                                                                                          panel_end, kmax);
}

// ------------------------------------------------------------- SIMT GEMM

// C (M x N) -= Am (M x K) * Bm (K x N); column-major; register tiles TM x TN.
template <typename T, int BM, int BN, int BK, int TM, int TN>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
gemm_sub_kernel(int64_t M, int64_t N, int K, const T *__restrict__ Am, int64_t lda_a,
                const T *__restrict__ Bm, int64_t ldb_b, T *C, int64_t ldc, const int64_t *info)
{
    constexpr int NT = (BM / TM) * (BN / TN);
    __shared__ T sa[BK][BM + 1];
    __shared__ T sb[BK][BN + 1];
    if (info && info_set(info)) return;
    const int tid = threadIdx.x;
    const int tx = tid % (BM / TM), ty = tid / (BM / TM);
    const int64_t m0 = (int64_t)blockIdx.x * BM, n0 = (int64_t)blockIdx.y * BN;
    T acc[TM][TN];
#pragma unroll
    for (int i = 0; i < TM; i++)
#pragma unroll
        for (int j = 0; j < TN; j++) acc[i][j] = T(0);

    for (int k0 = 0; k0 < K; k0 += BK) {
        for (int e = tid; e < BM * BK; e += NT) {
            int i = e % BM, k = e / BM;
            int64_t gi = m0 + i;
            sa[k][i] = (gi < M && k0 + k < K) ? Am[gi + (int64_t)(k0 + k) * lda_a] : T(0);
        }
        for (int e = tid; e < BN * BK; e += NT) {
            int k = e % BK, j = e / BK;
            int64_t gj = n0 + j;
            sb[k][j] = (gj < N && k0 + k < K) ? Bm[(k0 + k) + gj * ldb_b] : T(0);
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < BK; k++) {
            T ra[TM], rb[TN];
#pragma unroll
            for (int i = 0; i < TM; i++) ra[i] = sa[k][tx + i * (BM / TM)];
#pragma unroll
            for (int j = 0; j < TN; j++) rb[j] = sb[k][ty + j * (BN / TN)];
#pragma unroll
            for (int i = 0; i < TM; i++)
#pragma unroll
                for (int j = 0; j < TN; j++) acc[i][j] = fma(ra[i], rb[j], acc[i][j]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < TN; j++) {
        int64_t gj = n0 + ty + j * (BN / TN);
        if (gj >= N) continue;
#pragma unroll
        for (int i = 0; i < TM; i++) {
            int64_t gi = m0 + tx + i * (BM / TM);
            if (gi < M) C[gi + gj * ldc] -= acc[i][j];
        }
    }
}

// Double-float C -= A B.  The product of two pairs keeps the exact error of
// the leading product (one FMA) and the two cross terms; the running sum keeps
// its leading part exact with TwoSum and gathers every error term in a float
// accumulator that is folded in once at the end (about 12 FP32 operations per
// multiply-add instead of about 18 with a renormalized sum each step).
constexpr int kDfBM = 64, kDfBN = 64, kDfBK = 16, kDfTM = 4, kDfTN = 4;

__global__ void __launch_bounds__(256)
gemm_sub_df64_kernel(int64_t M, int64_t N, int K, const df64 *__restrict__ Am, int64_t lda_a,
                     const df64 *__restrict__ Bm, int64_t ldb_b, df64 *C, int64_t ldc, const int64_t *info)
{
    __shared__ float sah[kDfBK][kDfBM + 4], sal[kDfBK][kDfBM + 4];
    __shared__ float sbh[kDfBK][kDfBN + 4], sbl[kDfBK][kDfBN + 4];
    if (info && info_set(info)) return;
    const int tid = threadIdx.x;
    const int tx = tid % (kDfBM / kDfTM), ty = tid / (kDfBM / kDfTM);
    const int64_t m0 = (int64_t)blockIdx.x * kDfBM, n0 = (int64_t)blockIdx.y * kDfBN;
    float ah[kDfTM][kDfTN], al[kDfTM][kDfTN];
#pragma unroll
    for (int i = 0; i < kDfTM; i++)
#pragma unroll
        for (int j = 0; j < kDfTN; j++) ah[i][j] = al[i][j] = 0.f;

    for (int k0 = 0; k0 < K; k0 += kDfBK) {
        for (int e = tid; e < kDfBM * kDfBK; e += 256) {
            int i = e % kDfBM, k = e / kDfBM;
            int64_t gi = m0 + i;
            df64 v = (gi < M && k0 + k < K) ? Am[gi + (int64_t)(k0 + k) * lda_a] : df64(0);
            sah[k][i] = v.hi;
            sal[k][i] = v.lo;
        }
        for (int e = tid; e < kDfBN * kDfBK; e += 256) {
            int k = e % kDfBK, j = e / kDfBK;
            int64_t gj = n0 + j;
            df64 v = (gj < N && k0 + k < K) ? Bm[(k0 + k) + gj * ldb_b] : df64(0);
            sbh[k][j] = v.hi;
            sbl[k][j] = v.lo;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kDfBK; k++) {
            float xh[kDfTM], xl[kDfTM], yh[kDfTN], yl[kDfTN];
#pragma unroll
            for (int i = 0; i < kDfTM; i++) {
                xh[i] = sah[k][tx + i * (kDfBM / kDfTM)];
                xl[i] = sal[k][tx + i * (kDfBM / kDfTM)];
            }
#pragma unroll
            for (int j = 0; j < kDfTN; j++) {
                yh[j] = sbh[k][ty + j * (kDfBN / kDfTN)];
                yl[j] = sbl[k][ty + j * (kDfBN / kDfTN)];
            }
#pragma unroll
            for (int i = 0; i < kDfTM; i++)
#pragma unroll
                for (int j = 0; j < kDfTN; j++) {
                    float p = __fmul_rn(xh[i], yh[j]);
                    float pe = __fmaf_rn(xh[i], yh[j], -p);
                    float s, se;
                    two_sum(ah[i][j], p, s, se);
                    ah[i][j] = s;
                    float l = __fadd_rn(al[i][j], __fadd_rn(se, pe));
                    l = __fmaf_rn(xh[i], yl[j], l);
                    al[i][j] = __fmaf_rn(xl[i], yh[j], l);
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < kDfTN; j++) {
        int64_t gj = n0 + ty + j * (kDfBN / kDfTN);
        if (gj >= N) continue;
#pragma unroll
        for (int i = 0; i < kDfTM; i++) {
            int64_t gi = m0 + tx + i * (kDfBM / kDfTM);
            if (gi < M) {
                df64 acc = df_norm(ah[i][j], al[i][j]);
                C[gi + gj * ldc] = C[gi + gj * ldc] - acc;
            }
        }
    }
}

// Large double-float updates: a persistent kernel, one 256-thread CTA per SM,
// 128 x 128 output tiles dealt round-robin, each thread an 8 x 8 register
// tile (two 4-row and two 4-column strips).  Operand k-slices of 16 travel
// by cp.async (8-byte copies: a leading dimension may be odd) into a
// 3-stage shared-memory ring that runs on across tile boundaries, so the
// next tile's first slices and, through an L2 prefetch, its block of C
// arrive while the current tile still computes.
constexpr int kDf2BM = 128, kDf2BN = 128, kDf2BK = 16, kDf2Stages = 3;
constexpr int kDf2StageElems = kDf2BK * kDf2BM + kDf2BN * kDf2BK;   // df64 elements per stage
constexpr size_t kDf2Smem = (size_t)kDf2Stages * kDf2StageElems * sizeof(df64);

__device__ __forceinline__ void cp_async8(void *smem, const void *gmem, bool valid)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    // src-size 0 fills the 8 bytes with zeros and reads nothing
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 8 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__global__ void __launch_bounds__(256, 1)
gemm_sub_df64_pipe_kernel(int64_t M, int64_t N, int K, const df64 *__restrict__ Am, int64_t lda_a,
                          const df64 *__restrict__ Bm, int64_t ldb_b, df64 *__restrict__ C, int64_t ldc,
                          const int64_t *info)
{
    extern __shared__ __align__(16) unsigned char df2_smem[];
    df64 *ring = reinterpret_cast<df64 *>(df2_smem);
    if (info && info_set(info)) return;
    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t tiles_m = (M + kDf2BM - 1) / kDf2BM;
    const int64_t ntiles = tiles_m * ((N + kDf2BN - 1) / kDf2BN);
    if ((int64_t)blockIdx.x >= ntiles) return;
    const int ksteps = (K + kDf2BK - 1) / kDf2BK;
    const int64_t my_tiles = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
    const int64_t total = my_tiles * ksteps;

    // stage s of this CTA's sequence: tile blockIdx.x + (s / ksteps) * gridDim.x, k-slice s % ksteps
    auto issue = [&](int64_t s) {
        const int64_t t = blockIdx.x + (s / ksteps) * gridDim.x;
        const int k0 = (int)(s % ksteps) * kDf2BK;
        const int64_t m0 = (t % tiles_m) * kDf2BM, n0 = (t / tiles_m) * kDf2BN;
        df64 *sa = ring + (s % kDf2Stages) * kDf2StageElems;
        df64 *sb = sa + kDf2BK * kDf2BM;
#pragma unroll
        for (int q = 0; q < (kDf2BM * kDf2BK) / 256; q++) {
            const int e = tid + q * 256;
            const int i = e % kDf2BM, k = e / kDf2BM;
            const bool ok = m0 + i < M && k0 + k < K;
            cp_async8(sa + k * kDf2BM + i, ok ? Am + (m0 + i) + (int64_t)(k0 + k) * lda_a : Am, ok);
        }
#pragma unroll
        for (int q = 0; q < (kDf2BN * kDf2BK) / 256; q++) {
            const int e = tid + q * 256;
            const int k = e % kDf2BK, j = e / kDf2BK;
            const bool ok = n0 + j < N && k0 + k < K;
            cp_async8(sb + j * kDf2BK + k, ok ? Bm + (k0 + k) + (n0 + j) * ldb_b : Bm, ok);
        }
    };

#pragma unroll
    for (int s = 0; s < kDf2Stages - 1; s++) {
        if (s < total) issue(s);
        cp_async_commit();
    }
    float ah[8][8], al[8][8];
    for (int64_t s = 0; s < total; s++) {
        cp_async_wait<kDf2Stages - 2>();
        // every thread's copies of stage s have landed, and every thread is
        // done with stage s - 1, whose buffer the next issue refills
        __syncthreads();
        if (s + kDf2Stages - 1 < total) issue(s + kDf2Stages - 1);
        cp_async_commit();
        const int kstep = (int)(s % ksteps);
        const int64_t t = blockIdx.x + (s / ksteps) * gridDim.x;
        const int64_t m0 = (t % tiles_m) * kDf2BM, n0 = (t / tiles_m) * kDf2BN;
        if (kstep == 0) {
#pragma unroll
            for (int i = 0; i < 8; i++)
#pragma unroll
                for (int j = 0; j < 8; j++) ah[i][j] = al[i][j] = 0.f;
            // pull this CTA's next block of C towards L2: 128 columns, nine
            // addresses each (one per 16 rows, plus the last row)
            const int64_t tn = t + gridDim.x;
            if (tn < ntiles) {
                const int64_t pm = (tn % tiles_m) * kDf2BM, pn = (tn / tiles_m) * kDf2BN;
                for (int q = tid; q < kDf2BN * 9; q += 256) {
                    const int c = q / 9, r = q % 9;
                    const int64_t gi = pm + (r < 8 ? r * 16 : kDf2BM - 1), gj = pn + c;
                    if (gi < M && gj < N)
                        asm volatile("prefetch.global.L2 [%0];" ::"l"(C + gi + gj * ldc));
                }
            }
        }
        const df64 *sa = ring + (s % kDf2Stages) * kDf2StageElems;
        const df64 *sb = sa + kDf2BK * kDf2BM;
#pragma unroll 2
        for (int k = 0; k < kDf2BK; k++) {
            float xh[8], xl[8], yh[8], yl[8];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const float4 u0 = *reinterpret_cast<const float4 *>(sa + k * kDf2BM + h * 64 + tx * 4);
                const float4 u1 = *reinterpret_cast<const float4 *>(sa + k * kDf2BM + h * 64 + tx * 4 + 2);
                xh[h * 4 + 0] = u0.x; xl[h * 4 + 0] = u0.y;
                xh[h * 4 + 1] = u0.z; xl[h * 4 + 1] = u0.w;
                xh[h * 4 + 2] = u1.x; xl[h * 4 + 2] = u1.y;
                xh[h * 4 + 3] = u1.z; xl[h * 4 + 3] = u1.w;
#pragma unroll
                for (int jj = 0; jj < 4; jj++) {
                    const float2 v = *reinterpret_cast<const float2 *>(sb + (h * 64 + ty * 4 + jj) * kDf2BK + k);
                    yh[h * 4 + jj] = v.x;
                    yl[h * 4 + jj] = v.y;
                }
            }
#pragma unroll
            for (int i = 0; i < 8; i++)
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    float p = __fmul_rn(xh[i], yh[j]);
                    float pe = __fmaf_rn(xh[i], yh[j], -p);
                    float s2, se;
                    two_sum(ah[i][j], p, s2, se);
                    ah[i][j] = s2;
                    float l = __fadd_rn(al[i][j], __fadd_rn(se, pe));
                    l = __fmaf_rn(xh[i], yl[j], l);
                    al[i][j] = __fmaf_rn(xl[i], yh[j], l);
                }
        }
        if (kstep == ksteps - 1) {
            // C -= acc, two columns (16 entries) per batch so that their loads overlap
#pragma unroll
            for (int jb = 0; jb < 8; jb += 2) {
                df64 cv[2][8];
#pragma unroll
                for (int jj = 0; jj < 2; jj++) {
                    const int j = jb + jj;
                    const int64_t gj = n0 + (j < 4 ? ty * 4 + j : 64 + ty * 4 + (j - 4));
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        const int64_t gi = m0 + (i < 4 ? tx * 4 + i : 64 + tx * 4 + (i - 4));
                        cv[jj][i] = (gi < M && gj < N) ? C[gi + gj * ldc] : df64(0);
                    }
                }
#pragma unroll
                for (int jj = 0; jj < 2; jj++) {
                    const int j = jb + jj;
                    const int64_t gj = n0 + (j < 4 ? ty * 4 + j : 64 + ty * 4 + (j - 4));
#pragma unroll
                    for (int i = 0; i < 8; i++) {
                        const int64_t gi = m0 + (i < 4 ? tx * 4 + i : 64 + tx * 4 + (i - 4));
                        if (gi < M && gj < N) C[gi + gj * ldc] = cv[jj][i] - df_norm(ah[i][j], al[i][j]);
                    }
                }
            }
        }
    }
    cp_async_wait<0>();
}

template <typename T>
rbt_status gemm_sub_simt(int64_t M, int64_t N, int K, const T *Am, int64_t lda_a, const T *Bm, int64_t ldb_b,
                         T *C, int64_t ldc, const int64_t *info, cudaStream_t stream)
{
    if (M <= 0 || N <= 0 || K <= 0) return RBT_OK;
    if (std::is_same<T, df64>::value) {
        if (M >= 2048 && N >= 2048) {
            // large updates: the persistent pipelined 128 x 128 kernel, one CTA per SM
            static PerDeviceOnce once;
            rbt_status cst = smem_opt_in(once, gemm_sub_df64_pipe_kernel, (int)kDf2Smem);
            if (cst != RBT_OK) return cst;
            const int64_t ntiles = cdiv(M, kDf2BM) * cdiv(N, kDf2BN);
            const int64_t grid = std::min<int64_t>(ntiles, device_sm_count());
            gemm_sub_df64_pipe_kernel<<<(unsigned)grid, 256, kDf2Smem, stream>>>(
                M, N, K, (const df64 *)Am, lda_a, (const df64 *)Bm, ldb_b, (df64 *)C, ldc, info);
        } else {
            dim3 grid((unsigned)cdiv(M, kDfBM), (unsigned)cdiv(N, kDfBN));
            gemm_sub_df64_kernel<<<grid, 256, 0, stream>>>(M, N, K, (const df64 *)Am, lda_a, (const df64 *)Bm, ldb_b,
                                                           (df64 *)C, ldc, info);
        }
    } else if (sizeof(T) == 8) {
        dim3 grid((unsigned)cdiv(M, 64), (unsigned)cdiv(N, 64));
        gemm_sub_kernel<T, 64, 64, 16, 4, 4><<<grid, 256, 0, stream>>>(M, N, K, Am, lda_a, Bm, ldb_b, C, ldc, info);
    } else {
        dim3 grid((unsigned)cdiv(M, 128), (unsigned)cdiv(N, 128));
        gemm_sub_kernel<T, 128, 128, 16, 8, 8><<<grid, 256, 0, stream>>>(M, N, K, Am, lda_a, Bm, ldb_b, C, ldc, info);
    }
    RBT_LAUNCH_CHECK();
    return RBT_OK;
}

template rbt_status gemm_sub_simt<double>(int64_t, int64_t, int, const double *, int64_t, const double *, int64_t,
                                          double *, int64_t, const int64_t *, cudaStream_t);
template rbt_status gemm_sub_simt<float>(int64_t, int64_t, int, const float *, int64_t, const float *, int64_t,
                                         float *, int64_t, const int64_t *, cudaStream_t);
template rbt_status gemm_sub_simt<df64>(int64_t, int64_t, int, const df64 *, int64_t, const df64 *, int64_t,
                                        df64 *, int64_t, const int64_t *, cudaStream_t);

// ------------------------------------------------------------ factor driver

// Which kernels take a step of kb columns, nb but in the last one.  The 64-column
// ones up to 64 (the only ones that deliver kmax), but a
// narrow step in double or float fills a quarter or half of diag64_kernel's panels
// and a few of trsm64_kernel's lanes.  Milliseconds of a factorization, both older
// kernels / older diagonal factor only / both 64-column ones:
//   double n = 1003  nb 16: 3.29 / 3.22 / 3.60    nb 32: 3.07 / 2.87 / 3.38
//          n = 2500  nb 16: 15.49 / 15.78 / 16.75  nb 32: 14.81 / 14.76 / 16.04
//   float  n = 1003  nb 16: 2.29 / 2.16 / 2.29    nb 32: 1.60 / 1.41 / 1.54
// (double-float: the 64-column ones throughout.)
template <typename T> static bool use_diag64(int kb, int nb, const int *kmax)
{
    return kb <= kP && (kmax || nb > 32 || std::is_same<T, df64>::value);
}
template <typename T> static bool use_trsm64(int kb, int nb, const int *kmax)
{
    return kb <= kP && (kmax || nb > 16 || !std::is_same<T, double>::value);
}

template <typename T>
rbt_status genp_panel_steps(int64_t n, T *A, int64_t lda, int64_t *info, int nb, int64_t k0, int64_t k_end,
                            bool trailing_simt, cudaStream_t stream, int64_t panel_end, int *kmax)
{
    for (int64_t k = k0; k < k_end; k += nb) {
        int kb = (int)(n - k < nb ? n - k : nb);
        int64_t rest = n - k - kb;
        {
            ProfScope ps(kProfPanel, stream);
            if (use_diag64<T>(kb, nb, kmax)) {
                diag64_kernel<T><<<1, 256, 0, stream>>>(k, kb, A, lda, info);
            } else {
                size_t sm = (size_t)kb * kb * sizeof(T);
                diag_factor_kernel<T><<<1, 256, sm, stream>>>(k, kb, A, lda, info);
            }
            RBT_LAUNCH_CHECK();
            if (rest <= 0) continue;
            if (use_trsm64<T>(kb, nb, kmax)) {
                if constexpr (std::is_same<T, double>::value)
                    launch_trsm64<T, 8, 16, 1>(k, kb, n, A, lda, info, panel_end, kmax, stream);
                else if (2 * cdiv(rest, 64) >= kNumSMs)
                    launch_trsm64<T, 64, 4, 2>(k, kb, n, A, lda, info, panel_end, kmax, stream);
                else
                    launch_trsm64<T, 16, 8, 1>(k, kb, n, A, lda, info, panel_end, kmax, stream);
            } else {
                size_t sm_t = trsm_smem_bytes<T>(kb);
                const int nbv = (int)cdiv(rest, kTrsmVec);
                trsm_panel_kernel<T><<<(unsigned)(2 * nbv), kTrsmThreads, sm_t, stream>>>(k, kb, n, A, lda, nbv, info);
            }
            RBT_LAUNCH_CHECK();
        }
        if (trailing_simt) {
            ProfScope ps(kProfUpdate, stream);
            T *a21 = A + (k + kb) + k * lda;
            T *a12 = A + k + (k + kb) * lda;
            T *a22 = A + (k + kb) + (k + kb) * lda;
            rbt_status st = gemm_sub_simt<T>(rest, rest, kb, a21, lda, a12, lda, a22, lda, info, stream);
            if (st != RBT_OK) return st;
        }
    }
    return RBT_OK;
}

template rbt_status genp_panel_steps<double>(int64_t, double *, int64_t, int64_t *, int, int64_t, int64_t, bool,
                                             cudaStream_t, int64_t, int *);
template rbt_status genp_panel_steps<float>(int64_t, float *, int64_t, int64_t *, int, int64_t, int64_t, bool,
                                            cudaStream_t, int64_t, int *);
template rbt_status genp_panel_steps<df64>(int64_t, df64 *, int64_t, int64_t *, int, int64_t, int64_t, bool,
                                           cudaStream_t, int64_t, int *);

template <typename T> static rbt_status configure_smem(int nb)
{
    static PerDeviceOnce once;
    return once_per_device(once, [nb]() -> rbt_status {
        size_t sm = (size_t)nb * nb * sizeof(T);
        int tri = (int)trsm_smem_bytes<T>(nb);
        RBT_CUDA_TRY(cudaFuncSetAttribute(diag_factor_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        RBT_CUDA_TRY(cudaFuncSetAttribute(trsm_panel_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, tri));
        return RBT_OK;
    });
}

rbt_status genp_configure(int prec, int nb)
{
    (void)nb;
    if (is_df64_storage(prec)) return configure_smem<df64>(kMaxNB);
    if (prec == RBT_F64) return configure_smem<double>(kMaxNB);
    return configure_smem<float>(kMaxNB);
}

}  // namespace rbt

using namespace rbt;

extern "C" {

size_t genp_factor_workspace(int64_t n, int32_t prec, int32_t nb)
{
    return genp_factor_workspace_impl(n, prec, nb);
}

rbt_status genp_factor(int64_t n, int32_t prec, void *A, int64_t lda, int64_t *d_info, void *work,
                       size_t work_bytes, int32_t nb, cudaStream_t stream)
{
    if (n < 0 || lda < (n > 1 ? n : 1) || !d_info || prec < RBT_F64 || prec > kLastPrec) return RBT_ERR_ARG;
    if (nb < 0 || nb > kMaxNB) return RBT_ERR_ARG;
    RBT_CUDA_TRY(cudaMemsetAsync(d_info, 0xff, sizeof(int64_t), stream));  // -1
    if (n == 0) return RBT_OK;
    if (!A) return RBT_ERR_ARG;
    if (work_bytes < genp_factor_workspace_impl(n, prec, nb)) return RBT_ERR_WORKSPACE;
    return genp_factor_impl(n, prec, A, lda, d_info, work, work_bytes, nb, stream);
}

}  // extern "C"
