// Double-float GENP update on BF16 tensor cores by exact integer slicing
// (sm_103a): C -= A B with A, B, C stored as double-float pairs.
//
// The product is split so that every tensor-core operation is exact, in the
// manner of the Ozaki scheme (Ozaki, Ogita, Oishi, Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication", Numer. Algorithms 59, 2012):
//   * each row i of A is scaled by 2^-e_i (|A_i.| < 2^(e_i - 1)) and each
//     column j of B by 2^-f_j, then written as S = 8 (or 7) balanced
//     base-128 digits,
//         A_ik = 2^e_i sum_p a_ik^(p) 2^(-7p),  a^(p) integers, |a^(p)| <= 64,
//     which BF16 (8 significant bits) holds exactly;
//   * the digit matrices are multiplied on the tensor cores with FP32
//     accumulation; a digit product is at most 2^12, and the at most S K
//     products of one weight sum exactly below 2^24 for K <= 512;
//   * products of equal weight t = p + q (t <= S + 1: 36 products for S = 8,
//     28 for S = 7) share a TMEM accumulator, and the epilogue folds the S
//     accumulators back into double-float: C_ij -= 2^(e_i + f_j) sum_t acc_t 2^(-7 t).
// The representation keeps 7S bits relative to each row's and column's
// largest entry; the dropped digit products (t >= S + 2) weigh about
// 2^-(7S - 3) of those per k.  The error is relative to those maxima, not to
// each entry, so it is larger than a double-float product's where rows or
// columns mix large and small entries.  GENP's panels do: column k of L21 carries 1/u_kk and row
// k of U12 carries u_kk, so a row of L21 spans many binades across k.  Before
// slicing, each k is therefore balanced by an exact power of two,
//     A_ik B_kj = (A_ik 2^t_k) (B_kj 2^-t_k),
//     t_k = floor((E(B_k.) - E(A_.k)) / 2),  E = binary exponent of the max,
// which brings the largest entries of column k of A and row k of B to the
// same binade (on RBT-transformed GENP panels the bound relative to the
// entrywise one drops from about 2^12 to 2^4 in the median).
//
// Double operands (RBT_F64, from n = 768) take the same route with nine
// digits: 63 bits relative to the row and column maxima, ten more than an
// entry has, 45 products, K <= 448 (9 K 2^12 <= 2^24), 48-column tiles (nine
// accumulators in TMEM), the fold in 64-bit integers.  Measured against the
// FP64-pipe update (first backward errors of unrefined solves, n = 600 ..
// 8197, depths 1 .. 3, both butterflies, rows and columns scaled by up to
// 10^3: geometric mean of the ratio 0.3 .. 1.7 per family, 0.96 over all).
// Entry by entry that holds where rows and columns are filled with entries of
// like size; a sparse matrix's fill-in can be smaller than its row's maximum
// by more than the ten spare bits, so rbt_solve asks first (spread.cu).  The
// FP64 pipe's 1.2 TFLOP/s bounded such factorizations: update class at n =
// 8197 307 ms, now 14.3 ms and 1.6 ms of slicing.
//
// Kernel: persistent, one CTA per SM, 128 x 64 output tiles (S accumulators
// x 64 columns in the 512 TMEM columns) dealt round-robin in an L2-friendly
// grouped order; a TMA producer warp streams 32-element K slabs of all S
// digit slices of A and of B (64-byte rows, 64-byte swizzle) through a
// 2-stage ring across tile boundaries; one thread issues the MMAs of a slab
// (24 for S = 8, 20 for S = 7: each digit of A against up to four adjacent
// digit slices of B, N <= 256); eight epilogue warps fold the accumulators
// and update C while the next tile's first slabs load.  Bounded waits as in the TF32 / BF16
// kernel.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "df64.cuh"
#include "gemm_tc.cuh"
#include "genp_internal.cuh"
#include "oz_slice.cuh"

namespace rbt {
namespace oz {

constexpr int BM = 128;
// TMEM holds one 128 x BN FP32 accumulator per digit weight t = 2 .. S + 1 in
// 512 columns: 64 columns each for S = 7 and 8, 48 for S = 9.
template <int S> constexpr int BN = S <= 8 ? 64 : 48;
// digit slices of B that one MMA covers (N = 256, or 240 of 48-column slices)
template <int S> constexpr int QN = 256 / BN<S>;
constexpr int KSLAB = 32;   // bf16 elements per 64-byte row
constexpr int A_SLICE_BYTES = BM * 64;
template <int S> constexpr int B_SLICE_BYTES = BN<S> * 64;
// S digits per operand: the stage ring is sized per digit count
template <int S> constexpr int kStageBytes = S * (A_SLICE_BYTES + B_SLICE_BYTES<S>);  // S = 8: 96 KB, 9: 99 KB
template <int S> constexpr int kStages = (227 * 1024 - 2048) / kStageBytes<S>;        // 2
template <int S> constexpr int kSmemBytes = kStages<S> * kStageBytes<S> + 1024 + 256;
constexpr int kOzEpiWarps = 8;                    // epilogue warps (two per TMEM lane quarter)
constexpr int kProdWarp = kOzEpiWarps;            // TMA producer
constexpr int kMmaWarp = kOzEpiWarps + 1;         // MMA issuer, TMEM owner
constexpr int kOzThreads = (kOzEpiWarps + 2) * 32;
constexpr int TMEM_COLS = 512;
// a digit product is at most 64 * 64 = 2^12 and a weight holds at most S of
// them per k: S * K * 2^12 <= 2^24 keeps every accumulation exact
template <int S> constexpr int KMAX = S <= 8 ? 512 : 448;
// the factorizations' panels: with seven digits the leading one is wide
// (oz_slice.cuh), (S + 2) K 2^12 <= 2^24
template <int S> constexpr bool kWide = S == 7;
template <int S> constexpr int kOuterNB = kWide<S> ? 448 : KMAX<S>;
constexpr int kMaxDigits = 8;    // of double-float operands
static_assert(kMaxDigits * KMAX<8> * 4096 <= (1 << 24) && kDigits64 * KMAX<9> * 4096 <= (1 << 24) &&
                  (7 + 2) * kOuterNB<7> * 4096 <= (1 << 24),
              "digit accumulation must stay exact");
static_assert(kMaxDigits * BN<8> <= TMEM_COLS && kDigits64 * BN<9> <= TMEM_COLS,
              "one accumulator per digit weight in TMEM");
static_assert(kStages<9> >= 2 && kStages<8> >= 2 && kStages<7> >= 2, "at least double buffering");
constexpr int kGroupM = 16;  // row tiles per group of the tile order (L2 reuse of the digit slices)

struct Status {
    int err;
};


__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of bar, for at most wait_ns of %globaltimer.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, Status *st, long long wait_ns)
{
    if (mbar_test(bar, parity)) return true;  // the common case: no timer read
    const unsigned long long t0 = global_ns();
    while (!mbar_test(bar, parity)) {
        if ((long long)(global_ns() - t0) > wait_ns) {
            atomicExch(&st->err, (int)RBT_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(smem_u32(dst)), "l"((uint64_t)map), "r"(x), "r"(y), "r"(smem_u32(bar))
        : "memory");
}

// K-major, 64-byte swizzle: 8-row groups 512 bytes apart.
__device__ __forceinline__ uint64_t smem_desc64(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFF) >> 4);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(512 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)4 << 61;  // SWIZZLE_64B
    return d;
}

// instruction descriptor for an M = 128, N = n BF16 x BF16 -> FP32 MMA (n a multiple of 16, <= 256)
__host__ __device__ constexpr uint32_t idesc_n(int n)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16_n(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t *r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// Wait for this thread's TMEM loads; the loaded registers are operands, so
// that no use of them is scheduled before the wait.
__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]),
                   "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
                 :
                 : "memory");
}

__device__ __forceinline__ void tmem_ld24(uint32_t taddr, uint32_t (&r)[24])
{
    tmem_ld8(taddr, r);
    tmem_ld8(taddr + 8, r + 8);
    tmem_ld8(taddr + 16, r + 16);
}

__device__ __forceinline__ void tmem_wait24(uint32_t (&r)[24])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23])
                 :
                 : "memory");
}

// An integer of |v| < 2^51 as a double, in one FP64 addition (the conversion
// instruction is no faster than that here, and an exact one in int32 is not
// wide enough).
__device__ __forceinline__ double double_of(long long v)
{
    return __longlong_as_double(0x4338000000000000ll + v) - 6755399441055744.0;  // 1.5 * 2^52
}

// C - v 2^e, v exact or rounded once; e outside the double exponents takes
// the library's scaling.
__device__ __forceinline__ double sub_scaled(double c, double v, int e)
{
    if (e > -1000 && e < 900) return ::fma(-v, __longlong_as_double((long long)(e + 1023) << 52), c);
    return c - ldexp(v, e);
}

__device__ __forceinline__ float pow2f(int e)
{
    // 2^e for the normal range of float
    e = e < -126 ? -126 : (e > 127 ? 127 : e);
    return __int_as_float((e + 127) << 23);
}

// Bounded wait that also gives up when another role of the CTA has given up
// (*abort set); a timeout records RBT_ERR_TIMEOUT and raises *abort.
__device__ __forceinline__ bool mbar_wait_ab(uint64_t *bar, uint32_t parity, Status *st, volatile int *abort,
                                             long long wait_ns)
{
    if (mbar_test(bar, parity)) return true;  // the common case: no timer read
    const unsigned long long t0 = global_ns();
    while (!mbar_test(bar, parity)) {
        if (*abort) return false;
        if ((long long)(global_ns() - t0) > wait_ns) {
            atomicExch(&st->err, (int)RBT_ERR_TIMEOUT);
            *abort = 1;
            return false;
        }
    }
    return true;
}

// One product of a launch: C (M x N, ldc) -= A B from the digit slices (padded
// row counts Mp, Np of one slice) and the row / column exponents.
template <int S> struct Problem {
    int M, N, Mp, Np;
    const int *ea, *fb;
    elem_t<S> *C;
    int64_t ldc;
    int tiles_m, tiles_n;
    int64_t ntiles;
};

// Output tile i of this CTA: tiles dealt round-robin over the grid, the first
// problem's before the second's, in a grouped order.  Groups of kGroupM row
// tiles, columns outer and rows inner within a group: the tiles in flight at
// one time share a band of kGroupM x 128 rows of A's digit slices and a few
// column tiles of B's, both L2-resident, instead of every wave streaming A's
// slices from DRAM.  Returns the problem.
template <int S>
__device__ __forceinline__ int tile_origin(int64_t i, const Problem<S> &p0, const Problem<S> &p1, int &m0, int &n0)
{
    int64_t t = blockIdx.x + i * gridDim.x;
    const int which = t >= p0.ntiles;
    if (which) t -= p0.ntiles;
    const int tiles_m = which ? p1.tiles_m : p0.tiles_m, tiles_n = which ? p1.tiles_n : p0.tiles_n;
    const int64_t per_group = (int64_t)kGroupM * tiles_n;
    const int grp = (int)(t / per_group), in_grp = (int)(t % per_group);
    const int first_m = grp * kGroupM;
    const int gm = tiles_m - first_m < kGroupM ? tiles_m - first_m : kGroupM;
    m0 = (first_m + in_grp % gm) * BM;
    n0 = (in_grp / gm) * BN<S>;
    return which;
}

// One or two products of the same K (the second may have no tiles), tensor
// maps of their slices (slice p of A at rows p Mp + m).  Every wait gives up
// after wait_ns (then st->err records the timeout, the other roles stop, and
// TMEM is freed as usual); with no_copy set (a test stall) the producer issues
// no copy at all, so the MMA warp's first wait runs out.
//
// Persistent, one CTA per SM, warp-specialized:
//   warp kProdWarp   (one lane) TMA producer, running ahead over the slabs of
//                    this CTA's whole tile sequence through the STAGES ring;
//   warp kMmaWarp    (one lane) MMA issuer; owns the TMEM allocation;
//   warps 0 .. 7     epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 and
//                    columns 32 (w / 4) .. + 31 of each accumulator.
// The accumulators fill all 512 TMEM columns, so the next tile's MMAs wait
// for the epilogue to release them (tmem_empty, signalled as soon as the
// last accumulator has been read, before its arithmetic and the update of
// C); the next tile's first slabs are loaded meanwhile, and each tile's
// block of C is prefetched into L2 while that tile's MMAs run.
// RAW (testing only): the epilogue writes the S accumulators themselves to
// raw[(t M + m) N + n] of the one problem instead of folding them into C.
template <bool RAW, int S>
__global__ void __launch_bounds__(kOzThreads, 1)
oz_update_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                 const __grid_constant__ CUtensorMap tmap_a1, const __grid_constant__ CUtensorMap tmap_b1,
                 const __grid_constant__ Problem<S> p0, const __grid_constant__ Problem<S> p1, int K,
                 const int64_t *info, Status *st, long long wait_ns, int no_copy, float *__restrict__ raw)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t *full = (uint64_t *)(smem + kStages<S> * kStageBytes<S>);
    uint64_t *empty = full + kStages<S>;
    uint64_t *tmem_full = empty + kStages<S>;
    uint64_t *tmem_empty = tmem_full + 1;
    uint64_t *drain = tmem_empty + 1;
    uint32_t *tmem_slot = (uint32_t *)(drain + 1);
    volatile int *abort = (volatile int *)(tmem_slot + 1);

    static_assert(S >= 5 && S <= kDigits64, "digit count");
    if (*((volatile const int64_t *)info) >= 0) return;
    const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
    const int64_t ntiles = p0.ntiles + p1.ntiles;
    if ((int64_t)blockIdx.x >= ntiles) return;
    const int64_t my_tiles = (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x;
    const int nk = (K + KSLAB - 1) / KSLAB;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages<S>; s++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[s])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(tmem_full)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(tmem_empty)), "r"(kOzEpiWarps)
                     : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(drain)) : "memory");
        *abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    if (warp == kProdWarp) {
        if (lane == 0) {
            int64_t g = 0;
            for (int64_t i = 0; i < my_tiles && !*abort && !no_copy; i++) {
                int m0, n0;
                const int which = tile_origin<S>(i, p0, p1, m0, n0);
                const CUtensorMap *ta = which ? &tmap_a1 : &tmap_a, *tb = which ? &tmap_b1 : &tmap_b;
                const int Mp = which ? p1.Mp : p0.Mp, Np = which ? p1.Np : p0.Np;
                for (int kt = 0; kt < nk; kt++, g++) {
                    const int s = (int)(g % kStages<S>);
                    const int64_t r = g / kStages<S>;
                    if (r > 0 && !mbar_wait_ab(&empty[s], (uint32_t)((r - 1) & 1), st, abort, wait_ns)) break;
                    unsigned char *sa = smem + s * kStageBytes<S>;
                    unsigned char *sb = sa + S * A_SLICE_BYTES;
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(&full[s])),
                                 "r"(kStageBytes<S>)
                                 : "memory");
                    for (int p = 0; p < S; p++) {
                        tma_load_2d(sa + p * A_SLICE_BYTES, ta, kt * KSLAB, p * Mp + m0, &full[s]);
                        tma_load_2d(sb + p * B_SLICE_BYTES<S>, tb, kt * KSLAB, p * Np + n0, &full[s]);
                    }
                }
            }
            // before the CTA may end: every load issued into a stage has landed
            for (int s = 0; s < kStages<S> && s < g; s++) {
                const int64_t last = g - 1 - ((g - 1 - s) % kStages<S>);  // last load issued into stage s
                mbar_wait(&full[s], (uint32_t)((last / kStages<S>) & 1), st, wait_ns);
            }
        }
        __syncwarp();
    } else if (warp == kMmaWarp) {
        if (lane == 0) {
            int64_t g = 0;
            for (int64_t i = 0; i < my_tiles && !*abort; i++) {
                if (i > 0 && !mbar_wait_ab(tmem_empty, (uint32_t)((i - 1) & 1), st, abort, wait_ns)) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                bool ok = true;
                for (int kt = 0; kt < nk; kt++, g++) {
                    const int s = (int)(g % kStages<S>);
                    if (!mbar_wait_ab(&full[s], (uint32_t)((g / kStages<S>) & 1), st, abort, wait_ns)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = smem_u32(smem + s * kStageBytes<S>);
                    const uint32_t sb = sa + S * A_SLICE_BYTES;
                    // Digit p of A meets digits q = 1 .. S + 1 - p of B, whose
                    // accumulators (weights p + q) are adjacent in TMEM and whose
                    // slices are adjacent in shared memory: one MMA covers up to
                    // QN of them (N <= 256).  p = 1 writes every accumulator first.
#pragma unroll
                    for (int p = 1; p <= S; p++) {
#pragma unroll
                        for (int q0 = 1; q0 <= S + 1 - p; q0 += QN<S>) {
                            const int nq = (S + 1 - p - q0 + 1) < QN<S> ? (S + 1 - p - q0 + 1) : QN<S>;
                            const uint32_t dcol = tmem + (uint32_t)((p + q0 - 2) * BN<S>);
#pragma unroll
                            for (int kk = 0; kk < 2; kk++) {
                                const uint32_t acc = (kt > 0 || p > 1 || kk > 0) ? 1u : 0u;
                                mma_bf16_n(dcol, smem_desc64(sa + (p - 1) * A_SLICE_BYTES + kk * 32),
                                           smem_desc64(sb + (q0 - 1) * B_SLICE_BYTES<S> + kk * 32), idesc_n(nq * BN<S>),
                                           acc);
                            }
                        }
                    }
                    mma_commit(&empty[s]);
                }
                if (!ok) break;
                mma_commit(tmem_full);
            }
            // every MMA issued has completed before TMEM is released
            mma_commit(drain);
            mbar_wait(drain, 0, st, wait_ns);
        }
        __syncwarp();
    } else {
        // epilogue warps
        constexpr int EC = BN<S> / 2;  // columns per warp
        const int q = warp % 4, ch = warp / 4;  // TMEM lane quarter, half of the tile's columns
        const uint32_t lane_base = (uint32_t)(q * 32) << 16;
        for (int64_t i = 0; i < my_tiles; i++) {
            int m0, n0;
            const int which = tile_origin<S>(i, p0, p1, m0, n0);
            const int M = which ? p1.M : p0.M, N = which ? p1.N : p0.N;
            const int64_t ldc = which ? p1.ldc : p0.ldc;
            elem_t<S> *__restrict__ C = which ? p1.C : p0.C;
            const int *__restrict__ ea = which ? p1.ea : p0.ea, *__restrict__ fb = which ? p1.fb : p0.fb;
            const int row = m0 + q * 32 + lane;
            const bool rok = row < M;
            const int cbase = ch * EC;
            // this tile's block of C towards L2 while its MMAs run: BN
            // columns, nine addresses each (one per 16 rows and the last row)
            if (!RAW)
                for (int e = threadIdx.x; e < BN<S> * 9; e += kOzEpiWarps * 32) {
                    const int c = e / 9, r = e % 9;
                    const int gi = m0 + (r < 8 ? r * 16 : BM - 1), gj = n0 + c;
                    if (gi < M && gj < N) asm volatile("prefetch.global.L2 [%0];" ::"l"(C + gi + (int64_t)gj * ldc));
                }
            const int er = (!RAW && rok) ? ea[row] : 0;
            bool ok = mbar_wait_ab(tmem_full, (uint32_t)(i & 1), st, abort, wait_ns);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t base = tmem + lane_base + (uint32_t)cbase;
            if constexpr (RAW) {
#pragma unroll 1
                for (int t = 0; t < S; t++) {
                    uint32_t a[EC];
                    tmem_ld32(base + (uint32_t)(t * BN<S>), a);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (rok)
                        for (int j = 0; j < EC; j++) {
                            const int col = n0 + cbase + j;
                            if (col < N) raw[((int64_t)t * M + row) * N + col] = __uint_as_float(a[j]);
                        }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tmem_empty)) : "memory");
                continue;
            }
            if constexpr (S == kDigits64) {
                // Double.  The accumulators are integers, and the product is
                // (H 2^28 + L) 2^(e_i + f_j - 70) with H = sum_{t <= 6} acc_t
                // 2^(7 (6 - t)) and L = sum_{t >= 7} acc_t 2^(7 (10 - t)):
                // gathered in 64-bit integers (neighbours first in 32 bits,
                // within 2^31: at most (t - 1) K 2^12 each), |H| < 2^50 and
                // |L| < 2^45 become doubles exactly.  Four FP64 operations an
                // entry, after the accumulators are released: nine
                // multiply-adds would take the FP64 pipe as long as the
                // tile's MMAs take the tensor pipe.
                long long H[EC], L[EC];
                uint32_t r0[EC], r1[EC];
                tmem_ld24(base, r0);
                tmem_ld24(base + (uint32_t)BN<S>, r1);
                tmem_wait24(r0);
                tmem_wait24(r1);
                auto both = [](uint32_t hi, uint32_t lo) {
                    return __float2int_rn(__uint_as_float(hi)) * 128 + __float2int_rn(__uint_as_float(lo));
                };
#pragma unroll
                for (int j = 0; j < EC; j++) H[j] = both(r0[j], r1[j]);                       // t = 2, 3
                auto next = [&](int t, bool pair) {  // accumulators t and t + 1
                    tmem_ld24(base + (uint32_t)((t - 2) * BN<S>), r0);
                    if (pair) tmem_ld24(base + (uint32_t)((t - 1) * BN<S>), r1);
                    tmem_wait24(r0);
                    if (pair) tmem_wait24(r1);
                };
                next(4, true);
#pragma unroll
                for (int j = 0; j < EC; j++) H[j] = (H[j] << 14) + both(r0[j], r1[j]);        // 4, 5
                next(6, false);
#pragma unroll
                for (int j = 0; j < EC; j++) H[j] = (H[j] << 7) + __float2int_rn(__uint_as_float(r0[j]));
                next(7, true);
#pragma unroll
                for (int j = 0; j < EC; j++) L[j] = both(r0[j], r1[j]);                       // 7, 8
                next(9, true);
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tmem_empty)) : "memory");
#pragma unroll
                for (int j = 0; j < EC; j++) L[j] = (L[j] << 14) + both(r0[j], r1[j]);        // 9, 10
                if (rok) {
#pragma unroll
                    for (int j0 = 0; j0 < EC; j0 += 8) {
                        double cv[8];
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            const int col = n0 + cbase + j0 + j;
                            cv[j] = col < N ? C[row + (int64_t)col * ldc] : 0.0;
                        }
#pragma unroll
                        for (int j = 0; j < 8; j++) {
                            const int col = n0 + cbase + j0 + j;
                            if (col < N) {
                                const int ef = fb[col];
                                const double v = ::fma(double_of(H[j0 + j]), 0x1p28, double_of(L[j0 + j]));
                                C[row + (int64_t)col * ldc] =
                                    (er >= kBadExp || ef >= kBadExp) ? NAN : sub_scaled(cv[j], v, er + ef - 7 * (S + 1));
                            }
                        }
                    }
                }
                continue;
            } else {
            // fold sum_t acc_t 2^(-7 t) into pairs (h, l), exactly term by
            // term, one accumulator (EC columns) at a time.  Two register
            // buffers: the next accumulator's TMEM load is issued before the
            // current one is folded; the accumulators go back to the MMA warp
            // as soon as the last of them has landed, before its fold.
            float h[EC], l[EC];
            uint32_t r0[EC], r1[EC];
            tmem_ld32(base, r0);
            tmem_wait32(r0);
            tmem_ld32(base + (uint32_t)BN<S>, r1);
#pragma unroll
            for (int j = 0; j < EC; j++) {
                h[j] = __uint_as_float(r0[j]) * pow2f(-2 * BETA);
                l[j] = 0.f;
            }
#pragma unroll
            for (int t = 1; t < S; t++) {
                uint32_t(&cur)[EC] = (t & 1) ? r1 : r0;
                uint32_t(&nxt)[EC] = (t & 1) ? r0 : r1;
                tmem_wait32(cur);
                if (t + 1 < S) tmem_ld32(base + (uint32_t)((t + 1) * BN<S>), nxt);
                if (t == S - 1) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tmem_empty)) : "memory");
                }
                const float w = pow2f(-(t + 2) * BETA);
#pragma unroll
                for (int j = 0; j < EC; j++) {
                    float s, e;
                    two_sum(h[j], __uint_as_float(cur[j]) * w, s, e);
                    h[j] = s;
                    l[j] = __fadd_rn(l[j], e);
                }
            }
            // C -= the folded product, eight columns per round of loads (outside
            // the accumulators' hold: the next tile's MMAs are running)
            if (rok) {
#pragma unroll
                for (int j0 = 0; j0 < EC; j0 += 8) {
                    df64 cv[8];
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int col = n0 + cbase + j0 + j;
                        cv[j] = col < N ? C[row + (int64_t)col * ldc] : df64(0);
                    }
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        const int col = n0 + cbase + j0 + j;
                        if (col < N) {
                            const float sc = pow2f(er + fb[col]);
                            C[row + (int64_t)col * ldc] = cv[j] - df_norm(h[j0 + j] * sc, l[j0 + j] * sc);
                        }
                    }
                }
            }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == kMmaWarp) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
    }
}

__global__ void status_to_info_kernel(const Status *st, int64_t *info)
{
    if (st->err != 0 && *info < 0) *info = -2;
}

// ---------------------------------------------------------------- host side

static PFN_cuTensorMapEncodeTiled_v12000 get_encode()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    });
    return fn;
}

static bool make_map(CUtensorMap *map, const void *base, int rows, int Kp, int box_rows)
{
    auto enc = get_encode();
    if (!enc) return false;
    cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)Kp * 2};
    cuuint32_t box[2] = {(cuuint32_t)KSLAB, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static inline int64_t rup(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

}  // namespace oz

size_t oz_update_workspace(int64_t M, int64_t N, int64_t K, int digits)
{
    using namespace oz;
    const int64_t S = digits;
    const int64_t Mp = rup(M, BM), Np = rup(N, digits == kDigits64 ? BN<9> : BN<8>), Kp = rup(K, KSLAB);
    return (size_t)rup(S * Mp * Kp * 2, 1024) + (size_t)rup(S * Np * Kp * 2, 1024) + (size_t)rup(Mp * 4, 256) +
           (size_t)rup(Np * 4, 256) + 2 * (size_t)rup(Kp * 4, 256) + 256;
}

namespace oz {

template <int S> static rbt_status configure()
{
    static PerDeviceOnce once, once_raw, once_out, once_wide;
    rbt_status st = smem_opt_in(once, oz_update_kernel<false, S>, kSmemBytes<S>);
    if (st == RBT_OK) st = smem_opt_in(once_out, slice_kernel<S, 32, false>, (int)slice_smem_bytes<S>(KMAX<S>));
    if (st == RBT_OK && kWide<S>)
        st = smem_opt_in(once_wide, slice_kernel<S, 32, kWide<S>>, (int)slice_smem_bytes<S>(kOuterNB<S>));
    if (st != RBT_OK || S != 8) return st;
    return smem_opt_in(once_raw, oz_update_kernel<true, 8>, kSmemBytes<8>);
}

// One update's digit slices and exponents, carved from a workspace of
// oz_update_workspace(M, N, K, S) bytes (the layout that function sizes).
struct Slices {
    __nv_bfloat16 *sa, *sb;
    int *ea, *fb, *ka, *kb;
    int64_t M, N, K, Mp, Np, Kp;
    char *end;
};

template <int S> static Slices carve(int64_t M, int64_t N, int64_t K, void *work)
{
    Slices sl;
    sl.M = M;
    sl.N = N;
    sl.K = K;
    sl.Mp = rup(M, BM);
    sl.Np = rup(N, BN<S>);
    sl.Kp = rup(K, KSLAB);
    char *w = (char *)work;
    sl.sa = (__nv_bfloat16 *)w;
    w += rup(S * sl.Mp * sl.Kp * 2, 1024);
    sl.sb = (__nv_bfloat16 *)w;
    w += rup(S * sl.Np * sl.Kp * 2, 1024);
    sl.ea = (int *)w;
    w += rup(sl.Mp * 4, 256);
    sl.fb = (int *)w;
    w += rup(sl.Np * 4, 256);
    sl.ka = (int *)w;
    w += rup(sl.Kp * 4, 256);
    sl.kb = (int *)w;
    w += rup(sl.Kp * 4, 256);
    sl.end = (char *)work + rup(w - (char *)work, 1024);
    return sl;
}

// The operands of one product C (M x N) -= A B and the balancing exponents of
// its K (ka and ka2: of A's columns, the larger counts; kb: of B's rows, or
// null to balance by A alone).
template <int S> struct Operands {
    int64_t M, N;
    const elem_t<S> *A, *B;
    elem_t<S> *C;
    const int *ka, *ka2, *kb;
    bool ta = false;  // A is stored as its transpose (K x M)
};

// One or two products of the same K and leading dimensions: the digit slices
// of all operands in one launch, the products in another.
template <int S, bool WIDE>
static rbt_status products(int count, const Operands<S> *op, const Slices *sl, int64_t K, int64_t lda, int64_t ldb,
                           int64_t ldc, const int64_t *info, void *status, unsigned max_ctas, cudaStream_t stream)
{
    using TE = elem_t<S>;
    const int Kp = (int)rup(K, KSLAB);
    {
        ProfScope pslice(kProfSlice, stream);
        SliceJobs<TE> jobs = {};
        const int per = K <= 64 ? 16 : 8;  // columns of B per CTA
        int64_t blocks = 0;
        for (int i = 0; i < count; i++) {
            const int nra = (int)(op[i].ta ? cdiv(sl[i].Mp, per) : sl[i].Mp / kSliceRows), nrb = (int)cdiv(sl[i].Np, per);
            jobs.job[2 * i] = {op[i].A, lda, (int)op[i].M, (int)sl[i].Mp, op[i].ka, op[i].ka2, op[i].kb,
                               sl[i].sa, sl[i].ea, op[i].ta ? 0 : 1, 1, nra};
            jobs.job[2 * i + 1] = {op[i].B, ldb, (int)op[i].N, (int)sl[i].Np, op[i].ka, op[i].ka2, op[i].kb,
                                   sl[i].sb, sl[i].fb, 0, -1, nrb};
            blocks += nra + nrb;
        }
        jobs.K = (int)K;
        jobs.Kp = Kp;
        if (K <= 64)
            slice_kernel<S, 16, WIDE><<<(unsigned)blocks, 256, slice_smem_bytes<S>(Kp), stream>>>(jobs);
        else
            slice_kernel<S, 32, WIDE><<<(unsigned)blocks, 256, slice_smem_bytes<S>(Kp), stream>>>(jobs);
        RBT_LAUNCH_CHECK();
    }
    ProfScope ps(kProfUpdate, stream);
    CUtensorMap ma[2], mb[2];
    Problem<S> p[2] = {};
    for (int i = 0; i < count; i++) {
        if (!make_map(&ma[i], sl[i].sa, (int)(S * sl[i].Mp), Kp, BM) ||
            !make_map(&mb[i], sl[i].sb, (int)(S * sl[i].Np), Kp, BN<S>))
            return RBT_ERR_CUDA;
        const int tm = (int)cdiv(op[i].M, BM), tn = (int)cdiv(op[i].N, BN<S>);
        p[i] = {(int)op[i].M, (int)op[i].N, (int)sl[i].Mp, (int)sl[i].Np, sl[i].ea, sl[i].fb, op[i].C, ldc, tm, tn,
                (int64_t)tm * tn};
    }
    if (count < 2) {
        ma[1] = ma[0];
        mb[1] = mb[0];
    }
    const unsigned grid = (unsigned)std::min<int64_t>(p[0].ntiles + p[1].ntiles, max_ctas);
    oz_update_kernel<false, S><<<grid, kOzThreads, kSmemBytes<S>, stream>>>(
        ma[0], mb[0], ma[1], mb[1], p[0], p[1], Kp, info, (Status *)status, wait_limit_ns(),
        debug_stall() == RBT_STALL_OZ_COPY ? 1 : 0, nullptr);
    RBT_LAUNCH_CHECK();
    return RBT_OK;
}

// A standalone update: its balancing exponents come from a pass of their own.
// by_a: t_k = -E(A_.k), so that A's digits do not depend on B and a column of C
// not on the other columns of B.
template <int S>
static rbt_status update(int64_t M, int64_t N, int64_t K, const elem_t<S> *A, int64_t lda, const elem_t<S> *B,
                         int64_t ldb, elem_t<S> *C, int64_t ldc, const int64_t *info, void *work, void *status,
                         unsigned max_ctas, cudaStream_t stream, bool ta = false, bool by_a = false)
{
    rbt_status s = configure<S>();
    if (s != RBT_OK) return s;
    const Slices sl = carve<S>(M, N, K, work);
    {
        ProfScope pslice(kProfSlice, stream);
        // both exponent arrays start at kNoExp (every byte 0x80)
        RBT_CUDA_TRY(cudaMemsetAsync(sl.ka, 0x80, (size_t)rup(sl.Kp * 4, 256) * 2, stream));
        const int ca = (int)cdiv(M, 4096), na = ta ? (int)cdiv(M, 64) : ca * (int)K;
        kexp_kernel<elem_t<S>><<<(unsigned)(na + (by_a ? 0 : cdiv(N, 64))), 256, 0, stream>>>((int)M, (int)K, (int)N, ca, na, ta, A,
                                                                              lda, B, ldb, sl.ka, sl.kb);
        RBT_LAUNCH_CHECK();
    }
    const Operands<S> op = {M, N, A, B, C, sl.ka, sl.ka, by_a ? nullptr : sl.kb, ta};
    return products<S, false>(1, &op, &sl, K, lda, ldb, ldc, info, status, max_ctas, stream);
}

}  // namespace oz

// C -= A B, all double-float column-major; K <= 512; digits = 7 or 8 per
// entry; at most max_ctas CTAs (0 = one per SM).
rbt_status oz_update(int64_t M, int64_t N, int64_t K, const df64 *A, int64_t lda, const df64 *B, int64_t ldb, df64 *C,
                     int64_t ldc, const int64_t *info, void *work, size_t work_bytes, void *status, int digits,
                     cudaStream_t stream, unsigned max_ctas)
{
    using namespace oz;
    if (M <= 0 || N <= 0 || K <= 0) return RBT_OK;
    if (digits != 7 && digits != 8) return RBT_ERR_ARG;
    if (K > KMAX<8> || M > INT32_MAX / digits || N > INT32_MAX / digits) return RBT_ERR_UNSUPPORTED;
    if (work_bytes < oz_update_workspace(M, N, K, digits)) return RBT_ERR_WORKSPACE;
    const unsigned ctas = max_ctas ? max_ctas : (unsigned)device_sm_count();
    return digits == 7 ? update<7>(M, N, K, A, lda, B, ldb, C, ldc, info, work, status, ctas, stream)
                       : update<8>(M, N, K, A, lda, B, ldb, C, ldc, info, work, status, ctas, stream);
}

size_t oz_residual_workspace(int64_t n, int64_t nrhs)
{
    return oz_update_workspace(n, nrhs, oz::KMAX<9>, oz::kDigits64) + 256;
}

// R (n x nrhs) -= A X, or A^T X, in double by nine-digit sliced products over
// pieces of 448 of the inner dimension: each reads A once, whatever the number
// of right-hand sides, where the FP64 pipe takes n^2 nrhs multiply-adds at two
// a clock and SM.  Balanced by A alone: an entry of the result is off by at most
// 2^-57 K max_k |A_ik| 2^-E_k max_k 2^E_k |X_kj| a piece, whatever the other
// columns of X hold (balanced against all of X, an isolated entry 2^40 in one
// column left the others' residuals 20 bits short).  *status (device, cleared
// by the caller) becomes nonzero when a device wait gave up.
rbt_status oz_residual(int64_t n, int64_t nrhs, const double *A, int64_t lda, bool trans, const double *X, int64_t ldx,
                       double *R, int64_t ldr, const int64_t *info, void *work, int *status, cudaStream_t stream)
{
    using namespace oz;
    for (int64_t k = 0; k < n; k += KMAX<9>) {
        const int64_t K = std::min<int64_t>(n - k, KMAX<9>);
        const rbt_status s = update<9>(n, nrhs, K, trans ? A + k : A + k * lda, lda, X + k, ldx, R, ldr, info, work, status,
                                       (unsigned)device_sm_count(), stream, trans, true);
        if (s != RBT_OK) return s;
    }
    return RBT_OK;
}

rbt_status oz_status_to_info(void *status, int64_t *info, cudaStream_t stream)
{
    oz::status_to_info_kernel<<<1, 1, 0, stream>>>((const oz::Status *)status, info);
    RBT_LAUNCH_CHECK();
    return RBT_OK;
}

namespace oz {

// The test entry point takes eight digits per entry.
constexpr int kRawDigits = 8;

// Caller digits (int8, [kRawDigits][rows][K] row-major) -> the K-major bf16 slices the
// update kernel reads ([kRawDigits][rows_p][Kp], zero padding).
__global__ void digits_to_slices_kernel(int rows, int rows_p, int K, int Kp, const int8_t *__restrict__ d,
                                        __nv_bfloat16 *__restrict__ out)
{
    const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t total = (int64_t)kRawDigits * rows_p * Kp;
    if (idx >= total) return;
    const int k = (int)(idx % Kp);
    const int64_t pr = idx / Kp;
    const int r = (int)(pr % rows_p), p = (int)(pr / rows_p);
    const int v = (r < rows && k < K) ? (int)d[((int64_t)p * rows + r) * K + k] : 0;
    out[idx] = bf16_of_digit(v);
}

}  // namespace oz

size_t oz_products_workspace(int64_t M, int64_t N, int64_t K)
{
    using namespace oz;
    if (M <= 0 || N <= 0 || K <= 0) return 0;
    const int64_t Mp = rup(M, BM), Np = rup(N, BN<kRawDigits>), Kp = rup(K, KSLAB);
    return (size_t)rup(kRawDigits * Mp * Kp * 2, 1024) + (size_t)rup(kRawDigits * Np * Kp * 2, 1024) + 256;
}

// The update kernel's copy and tensor-core pipeline on caller digits, with the
// raw-accumulator epilogue.
rbt_status oz_products(int64_t M, int64_t N, int64_t K, const int8_t *da, const int8_t *db, float *acc, void *work,
                       size_t work_bytes, cudaStream_t stream)
{
    using namespace oz;
    if (M < 0 || N < 0 || K < 0) return RBT_ERR_ARG;
    if (M == 0 || N == 0 || K == 0) return RBT_OK;
    if (!da || !db || !acc) return RBT_ERR_ARG;
    if (K > KMAX<kRawDigits> || M > INT32_MAX / kRawDigits || N > INT32_MAX / kRawDigits) return RBT_ERR_UNSUPPORTED;
    if (!work || work_bytes < oz_products_workspace(M, N, K)) return RBT_ERR_WORKSPACE;
    rbt_status s = configure<kRawDigits>();
    if (s != RBT_OK) return s;
    const int64_t Mp = rup(M, BM), Np = rup(N, BN<kRawDigits>), Kp = rup(K, KSLAB);
    char *w = (char *)work;
    __nv_bfloat16 *sa = (__nv_bfloat16 *)w;
    w += rup(kRawDigits * Mp * Kp * 2, 1024);
    __nv_bfloat16 *sb = (__nv_bfloat16 *)w;
    w += rup(kRawDigits * Np * Kp * 2, 1024);
    Status *status = (Status *)w;             // [0, 8): status word, [8, 16): "no failed pivot" (-1)
    int64_t *info = (int64_t *)(w + 8);
    RBT_CUDA_TRY(cudaMemsetAsync(w, 0, 8, stream));
    RBT_CUDA_TRY(cudaMemsetAsync(info, 0xff, 8, stream));
    const int64_t ta = (int64_t)kRawDigits * Mp * Kp, tb = (int64_t)kRawDigits * Np * Kp;
    digits_to_slices_kernel<<<(unsigned)cdiv(ta, 256), 256, 0, stream>>>((int)M, (int)Mp, (int)K, (int)Kp, da, sa);
    RBT_LAUNCH_CHECK();
    digits_to_slices_kernel<<<(unsigned)cdiv(tb, 256), 256, 0, stream>>>((int)N, (int)Np, (int)K, (int)Kp, db, sb);
    RBT_LAUNCH_CHECK();
    CUtensorMap ma, mb;
    if (!make_map(&ma, sa, (int)(kRawDigits * Mp), (int)Kp, BM) || !make_map(&mb, sb, (int)(kRawDigits * Np), (int)Kp, BN<kRawDigits>))
        return RBT_ERR_CUDA;
    const int64_t ntiles = (Mp / BM) * (Np / BN<kRawDigits>);
    const unsigned grid = (unsigned)std::min<int64_t>(ntiles, device_sm_count());
    const int tm = (int)(Mp / BM), tn = (int)(Np / BN<kRawDigits>);
    const Problem<kRawDigits> p = {(int)M, (int)N, (int)Mp, (int)Np, nullptr, nullptr, nullptr, 0, tm, tn, ntiles}, none = {};
    oz_update_kernel<true, kRawDigits><<<grid, kOzThreads, kSmemBytes<kRawDigits>, stream>>>(
        ma, mb, ma, mb, p, none, (int)Kp, info, status, wait_limit_ns(), 0, acc);
    RBT_LAUNCH_CHECK();
    return RBT_OK;
}

}  // namespace rbt

extern "C" {

size_t rbt_debug_oz_products_workspace(int64_t M, int64_t N, int64_t K)
{
    return rbt::oz_products_workspace(M, N, K);
}

rbt_status rbt_debug_oz_products(int64_t M, int64_t N, int64_t K, const int8_t *da, const int8_t *db, float *acc,
                                 void *work, size_t work_bytes, cudaStream_t stream)
{
    return rbt::oz_products(M, N, K, da, db, acc, work, work_bytes, stream);
}

}  // extern "C"

namespace rbt {

constexpr int kOzInnerNB = 64;   // panel step (double-float diagonal factor and TRSMs)

size_t oz_factor_workspace(int64_t n)
{
    if (n <= 0) return 0;
    // any digit count: an outer update's slices (far more than the two inner
    // ones'), the balancing exponents of a panel, the status word
    return std::max(oz_update_workspace(n, n, oz::KMAX<8>, 8), oz_update_workspace(n, n, oz::KMAX<9>, 9)) + 16384 +
           4 * kKmax * sizeof(int) + 256;
}

namespace {

// Two-level blocked GENP: panels of 512 columns (448 with seven digits and in
// double) factored with
// 64-column steps (diagonal factor and both TRSMs on the SIMT pipes, one
// launch of sliced tensor-core updates of the panel's remaining columns and of
// the rest of its rows), then one sliced update of the trailing matrix per
// panel.  The TRSMs leave the exponents that balance every update (per column
// of L21 and row of U12, split at the panel's end), so an update is two
// launches: slicing and products.
template <int S>
rbt_status factor_oz(int64_t n, oz::elem_t<S> *A, int64_t lda, int64_t *info, void *work, cudaStream_t stream)
{
    constexpr int kOuter = oz::kOuterNB<S>;
    rbt_status s = oz::configure<S>();
    if (s != RBT_OK) return s;
    void *status = (char *)work + oz_factor_workspace(n) - 256;
    int *kmax = (int *)status - 4 * kKmax;
    int *rows_in = kmax, *rows_below = kmax + kKmax, *cols_in = kmax + 2 * kKmax, *cols_right = kmax + 3 * kKmax;
    RBT_CUDA_TRY(cudaMemsetAsync(status, 0, 256, stream));
    const unsigned sms = (unsigned)device_sm_count();
    for (int64_t k = 0; k < n; k += kOuter) {
        const int64_t kb = n - k < kOuter ? n - k : kOuter;
        const int64_t t0 = k + kb, right = n - t0;
        if (n - k > kOzInnerNB)
            RBT_CUDA_TRY(cudaMemsetAsync(kmax, 0x80, 4 * kKmax * sizeof(int), stream));  // kNoExp
        for (int64_t j = k; j < t0; j += kOzInnerNB) {
            const int jb = (int)(t0 - j < kOzInnerNB ? t0 - j : kOzInnerNB);
            const int64_t r0 = j + jb, at = j - k;
            s = genp_panel_steps<oz::elem_t<S>>(n, A, lda, info, jb, j, r0, false, stream, t0, kmax + at);
            if (s != RBT_OK) return s;
            if (r0 >= t0) continue;
            const oz::Operands<S> op[2] = {
                {n - r0, t0 - r0, A + r0 + j * lda, A + j + r0 * lda, A + r0 + r0 * lda, rows_in + at, rows_below + at,
                 cols_in + at},
                {t0 - r0, right, A + r0 + j * lda, A + j + t0 * lda, A + r0 + t0 * lda, rows_in + at, rows_in + at,
                 cols_right + at}};
            oz::Slices sl[2];
            sl[0] = oz::carve<S>(op[0].M, op[0].N, jb, work);
            sl[1] = oz::carve<S>(op[1].M, op[1].N, jb, sl[0].end);
            s = oz::products<S, oz::kWide<S>>(right > 0 ? 2 : 1, op, sl, jb, lda, lda, lda, info, status, sms, stream);
            if (s != RBT_OK) return s;
        }
        if (right <= 0) continue;
        const oz::Operands<S> op = {right, right, A + t0 + k * lda, A + k + t0 * lda, A + t0 + t0 * lda, rows_below,
                                    rows_below, cols_right};
        const oz::Slices sl = oz::carve<S>(right, right, kb, work);
        s = oz::products<S, oz::kWide<S>>(1, &op, &sl, kb, lda, lda, lda, info, status, sms, stream);
        if (s != RBT_OK) return s;
    }
    return oz_status_to_info(status, info, stream);
}

}  // namespace

rbt_status genp_factor_oz64(int64_t n, double *A, int64_t lda, int64_t *info, void *work, size_t work_bytes,
                            cudaStream_t stream)
{
    if (work_bytes < oz_factor_workspace(n) || !work) return RBT_ERR_WORKSPACE;
    if (n > INT32_MAX / oz::kDigits64) return RBT_ERR_UNSUPPORTED;
    return factor_oz<oz::kDigits64>(n, A, lda, info, work, stream);
}

// digits = 7 or 8 per entry of the sliced operands
rbt_status genp_factor_oz(int64_t n, df64 *A, int64_t lda, int64_t *info, void *work, size_t work_bytes, int digits,
                          cudaStream_t stream)
{
    if (work_bytes < oz_factor_workspace(n) || !work) return RBT_ERR_WORKSPACE;
    if (digits != 7 && digits != 8) return RBT_ERR_ARG;
    if (n > INT32_MAX / oz::kMaxDigits) return RBT_ERR_UNSUPPORTED;
    return digits == 7 ? factor_oz<7>(n, A, lda, info, work, stream) : factor_oz<8>(n, A, lda, info, work, stream);
}

}  // namespace rbt
