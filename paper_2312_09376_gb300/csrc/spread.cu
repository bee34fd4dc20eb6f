// Are a double matrix's rows and columns filled with entries of like size?
//
// The sliced double update (gemm_oz.cu) keeps 63 bits relative to the largest
// entry of each row of L21 and column of U12, ten more than an entry has.
// Against |L| |U| that is no less than double arithmetic gives as long as the
// entries of a row and of a column are of like size, up to row and column
// scalings (which the slicing takes out).  Where many entries are zero or
// tiny, elimination fills in values far below their row's maximum, and those
// would lose relative accuracy; a single entry far above the others costs them
// the bits itself (one of 2^60 in a Gaussian matrix: 1e-11 of |L| |U|).
//
// The test fits e_ij = r_i + c_j to the binary exponents by the rows' and
// columns' means (of the entries that are not zero).  An entry is small if it
// is zero or lies more than six bits below the fit, and large if it lies more
// than nine above it.  A matrix passes with no large entry off the diagonal (a
// diagonal one is a pivot and in no product) and no more than a quarter of any
// row or column small, so that a row and a column have at least half of their
// factors in common.  A matrix D_r G D_c with entries of G of like size passes
// as G does.  Why there: error of a 448-column panel's product in units of |L|
// |U|, root mean square (an emulation at n = 800), double 2e-17 to 1e-16;
// sliced 3e-21 for Gaussian entries, 9e-18 and 5e-17 with 3000 of them raised
// by 2^8 and 2^10, 2e-18, 1e-17, 4e-17 and 1.5e-16 with every second one (i + j
// odd) lowered by 2^8, 2^10, 2^12 and 2^14.  Two passes over the matrix: 0.35 ms
// at n = 8197.
#include "common.cuh"
#include "genp_internal.cuh"

namespace rbt {

constexpr int kSpreadRows = 256, kSpreadCols = 64;
constexpr float kSmallBits = 6.f, kLargeBits = 9.f;
constexpr int kFitThreads = 1024;

// Exponent field of |x| (0 for zero and subnormals, which count as zeros).
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// Sum of exponents (low 32 bits: n 2047 < 2^32) and number of entries.
typedef unsigned long long ExpSum;
__device__ __forceinline__ float exp_mean(ExpSum s)
{
    const unsigned n = (unsigned)(s >> 32);
    return n ? (float)((double)(unsigned)s / n) : 0.f;
}

// FIT: r[i], c[j] <- exponent sums of row i and column j (zeroed beforehand).
// Otherwise: nr[i], nc[j] <- small entries of row i and column j against the
// fit rf[i] + cf[j]; *most <- INT_MAX where an entry is large.
// One row per thread, 64 columns per CTA; a warp's 32 rows of a column meet by
// a warp reduction, so a CTA issues one atomic per row and one per warp and
// column.
template <bool FIT>
__global__ void __launch_bounds__(kSpreadRows)
spread_kernel(int64_t n, const double *__restrict__ A, int64_t lda, ExpSum *r, ExpSum *c, const float *__restrict__ rf,
              const float *__restrict__ cf, int *nr, int *nc, int *most)
{
    const int64_t i = (int64_t)blockIdx.x * kSpreadRows + threadIdx.x;
    const int64_t j0 = (int64_t)blockIdx.y * kSpreadCols;
    const int jn = (int)(n - j0 < kSpreadCols ? n - j0 : kSpreadCols);
    const int lane = threadIdx.x & 31;
    const bool in = i < n;
    const float ri = !FIT && in ? rf[i] : 0.f;
    unsigned sum = 0, count = 0;
    bool large = false;
#pragma unroll 8
    for (int j = 0; j < jn; j++) {
        const double a = in ? A[i + (j0 + j) * lda] : 0.0;
        const unsigned e = (unsigned)exp_field(a);
        if (FIT) {
            sum += e;
            count += e != 0;
            // 32 exponents below 2^16, 32 entries above 2^20
            const unsigned w = __reduce_add_sync(0xffffffffu, e + (e ? 1u << 20 : 0u));
            if (lane == 0) atomicAdd(c + j0 + j, (ExpSum)(w >> 20) << 32 | (w & 0xFFFFFu));
        } else {
            const float d = (float)(int)e - (ri + cf[j0 + j]);
            const bool small = in && (e == 0 || d < -kSmallBits);
            large = large || (in && e != 0 && d > kLargeBits && i != j0 + j);
            count += small;
            const unsigned b = __ballot_sync(0xffffffffu, small);
            if (lane == 0 && b) atomicAdd(nc + j0 + j, __popc(b));
        }
    }
    if (in && FIT) atomicAdd(r + i, (ExpSum)count << 32 | sum);
    if (in && !FIT && count) atomicAdd(nr + i, (int)count);
    if (large) atomicMax(most, INT32_MAX);
}

// rf[i] = mean of row i, cf[j] = mean of column j less the mean of all.
__global__ void __launch_bounds__(kFitThreads) fit_kernel(int64_t n, const ExpSum *__restrict__ r,
                                                          const ExpSum *__restrict__ c, float *rf, float *cf)
{
    __shared__ ExpSum s_sum[kFitThreads / 32], s_count[kFitThreads / 32];
    ExpSum sum = 0, count = 0;
    for (int64_t i = threadIdx.x; i < n; i += kFitThreads) {
        const ExpSum v = r[i];
        sum += (unsigned)v;
        count += v >> 32;
        rf[i] = exp_mean(v);
    }
    auto warp_sum = [](ExpSum v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    };
    sum = warp_sum(sum);
    count = warp_sum(count);
    if (threadIdx.x % 32 == 0) {
        s_sum[threadIdx.x / 32] = sum;
        s_count[threadIdx.x / 32] = count;
    }
    __syncthreads();
    sum = warp_sum(s_sum[threadIdx.x % 32]);
    count = warp_sum(s_count[threadIdx.x % 32]);
    const float all = count ? (float)((double)sum / (double)count) : 0.f;
    for (int64_t j = threadIdx.x; j < n; j += kFitThreads) cf[j] = exp_mean(c[j]) - all;
}

// out[0] <- max of v[0 .. n) (zeroed beforehand)
__global__ void __launch_bounds__(256) max_kernel(int64_t n, const int *__restrict__ v, int *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int m = __reduce_max_sync(0xffffffffu, i < n ? v[i] : 0);
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// exponent sums, small entries and *most (zeroed together), then the fit
static size_t spread_zeroed(int64_t n) { return (size_t)n * (2 * sizeof(ExpSum) + 2 * sizeof(int)) + 8; }

size_t spread_workspace(int64_t n) { return spread_zeroed(n) + (size_t)n * 2 * sizeof(float); }

rbt_status evenly_spread(int64_t n, const double *A, int64_t lda, void *scratch, bool *even, cudaStream_t stream)
{
    ExpSum *r = (ExpSum *)scratch, *c = r + n;
    int *nr = (int *)(c + n), *nc = nr + n, *most = nc + n;
    float *rf = (float *)((char *)scratch + spread_zeroed(n)), *cf = rf + n;
    RBT_CUDA_TRY(cudaMemsetAsync(scratch, 0, spread_zeroed(n), stream));
    const dim3 grid((unsigned)cdiv(n, kSpreadRows), (unsigned)cdiv(n, kSpreadCols));
    spread_kernel<true><<<grid, kSpreadRows, 0, stream>>>(n, A, lda, r, c, rf, cf, nr, nc, most);
    RBT_LAUNCH_CHECK();
    fit_kernel<<<1, kFitThreads, 0, stream>>>(n, r, c, rf, cf);
    RBT_LAUNCH_CHECK();
    spread_kernel<false><<<grid, kSpreadRows, 0, stream>>>(n, A, lda, r, c, rf, cf, nr, nc, most);
    RBT_LAUNCH_CHECK();
    max_kernel<<<(unsigned)cdiv(2 * n, 256), 256, 0, stream>>>(2 * n, nr, most);
    RBT_LAUNCH_CHECK();
    int h = 0;
    RBT_CUDA_TRY(cudaMemcpyAsync(&h, most, sizeof(int), cudaMemcpyDeviceToHost, stream));
    RBT_CUDA_TRY(cudaStreamSynchronize(stream));
    *even = 4 * (int64_t)h <= n;
    return RBT_OK;
}

}  // namespace rbt
