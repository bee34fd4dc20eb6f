// Are a double matrix's rows and columns filled with entries of like size?
//
// The sliced double update (gemm_oz.cu) keeps 63 bits relative to the largest
// entry of each row of L21 and column of U12, ten more than an entry has.
// Against |L| |U| that is no less than double arithmetic gives as long as most
// entries of a row and of a column are of the size of its largest, up to row
// and column scalings (which the slicing takes out); where many entries are
// zero or tiny, elimination fills in values far below their row's maximum,
// and those would lose relative accuracy.  The test: with r_i and c_j the
// binary exponents of the row and column maxima and g of the largest entry, a
// matrix D_r G D_c with entries of G of like size has a_ij near 2^(r_i + c_j -
// g); an entry more than 2^12 below that (or zero) is small, and no row and no
// column may have more than half of its entries small.  Two passes over the
// matrix: 0.2 ms at n = 8197.
#include "common.cuh"
#include "genp_internal.cuh"

namespace rbt {

constexpr int kSpreadRows = 256, kSpreadCols = 64;
constexpr int kSmallBits = 12;

// Exponent field of |x| (0 for zero and subnormals).
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7FF; }

// PASS 0: r[i], c[j] <- largest exponent fields (zeroed beforehand).
// PASS 1: nr[i], nc[j] <- small entries of row i and column j.
// One row per thread, 64 columns per CTA; a warp's 32 rows of a column meet by
// a warp reduction, so a CTA issues one atomic per row and one per warp and
// column.
template <int PASS>
__global__ void __launch_bounds__(kSpreadRows) spread_kernel(int64_t n, const double *__restrict__ A, int64_t lda,
                                                             int *r, int *c, const int *g, int *nr, int *nc)
{
    const int64_t i = (int64_t)blockIdx.x * kSpreadRows + threadIdx.x;
    const int64_t j0 = (int64_t)blockIdx.y * kSpreadCols;
    const int jn = (int)(n - j0 < kSpreadCols ? n - j0 : kSpreadCols);
    const int lane = threadIdx.x & 31;
    const bool in = i < n;
    const int ri = PASS == 1 && in ? r[i] - *g - kSmallBits : 0;
    int mine = 0;
#pragma unroll 8
    for (int j = 0; j < jn; j++) {
        const double a = in ? A[i + (j0 + j) * lda] : 0.0;
        const int e = exp_field(a);
        if (PASS == 0) {
            mine = max(mine, e);
            const int m = __reduce_max_sync(0xffffffffu, e);
            if (lane == 0) atomicMax(c + j0 + j, m);
        } else {
            const bool small = in && (a == 0.0 || e < ri + c[j0 + j]);
            mine += small;
            const unsigned b = __ballot_sync(0xffffffffu, small);
            if (lane == 0 && b) atomicAdd(nc + j0 + j, __popc(b));
        }
    }
    if (in && PASS == 0) atomicMax(r + i, mine);
    if (in && PASS == 1 && mine) atomicAdd(nr + i, mine);
}

// out[0] <- max of v[0 .. n) (zeroed beforehand)
__global__ void __launch_bounds__(256) max_kernel(int64_t n, const int *__restrict__ v, int *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int m = __reduce_max_sync(0xffffffffu, i < n ? v[i] : 0);
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

size_t spread_workspace(int64_t n) { return (size_t)(4 * n + 2) * sizeof(int); }

rbt_status evenly_spread(int64_t n, const double *A, int64_t lda, void *scratch, bool *even, cudaStream_t stream)
{
    int *r = (int *)scratch, *c = r + n, *nr = c + n, *nc = nr + n, *g = nc + n, *most = g + 1;
    RBT_CUDA_TRY(cudaMemsetAsync(scratch, 0, spread_workspace(n), stream));
    const dim3 grid((unsigned)cdiv(n, kSpreadRows), (unsigned)cdiv(n, kSpreadCols));
    spread_kernel<0><<<grid, kSpreadRows, 0, stream>>>(n, A, lda, r, c, g, nr, nc);
    RBT_LAUNCH_CHECK();
    max_kernel<<<(unsigned)cdiv(n, 256), 256, 0, stream>>>(n, r, g);
    RBT_LAUNCH_CHECK();
    spread_kernel<1><<<grid, kSpreadRows, 0, stream>>>(n, A, lda, r, c, g, nr, nc);
    RBT_LAUNCH_CHECK();
    max_kernel<<<(unsigned)cdiv(2 * n, 256), 256, 0, stream>>>(2 * n, nr, most);
    RBT_LAUNCH_CHECK();
    int h = 0;
    RBT_CUDA_TRY(cudaMemcpyAsync(&h, most, sizeof(int), cudaMemcpyDeviceToHost, stream));
    RBT_CUDA_TRY(cudaStreamSynchronize(stream));
    *even = 2 * (int64_t)h <= n;
    return RBT_OK;
}

}  // namespace rbt
