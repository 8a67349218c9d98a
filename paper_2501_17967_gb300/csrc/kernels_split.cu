// Operator products on the 5th-generation tensor cores (tcgen05) as exact
// products of BF16 digits.
//
// The fixed-operator products of an apply -- the near-field tables, P2M, L2P,
// the W list (M2P) and the X list (P2L), their adjoints, and the multipole-to-
// local translations -- are dense real matrices (the operators) times many
// vectors (leaf values or expansion coefficients).  Each product is evaluated
// in integer arithmetic on BF16 tensor cores, with five digits per operand in
// the split modes (described first) or seven in the FP64 mode (see Fmt):
//   * each FP64 operand row (operator row, input vector) is scaled by a power
//     of two 2^E so that its entries lie in (-1/2, 1/2), rounded to a 40-bit
//     fixed-point integer X and cut into five balanced base-256 digits,
//     X = sum_a theta_a 256^(5-a), |theta_a| <= 128; every digit is an integer
//     that BF16 holds exactly (Ozaki-style error-free splitting);
//   * A v = 2^(E_A + E_v - 48) * sum_g 256^(6-g) D_g,  D_g = sum_{a+b=g} theta_a . phi_b,
//     keeping the digit pairs a + b <= 6 (15 products; what is dropped is below
//     2^-38 relative to sum_k |A_ik v_k|);
//   * each D_g (g = 2..6) accumulates in its own FP32 TMEM accumulator: every
//     product is an integer of magnitude <= 2^14 and a level sums at most
//     4 x 256 of them for g <= 5, so the accumulation is exact (< 2^24);
//   * the five levels are combined in int64 and converted to FP64 once (a
//     hardware conversion; the power-of-two scale is then added to the
//     exponent field of the bit pattern).
//
// Work decomposition: a tile is one operator times up to 48 (32) columns, done
// as one job per 128-row half of the operator.
//   B operand: the columns' digits, gathered into shared memory with 16-byte
//              asynchronous copies (cp.async), one buffer per K chunk of 128; the
//              chunks take turns (kchunk_at), so that the next tile's are gathered
//              while this tile's MMAs run;
//   A operand: the operator's digits, 128 rows x 128 columns per chunk (32 KB),
//              brought in by bulk asynchronous copies through three buffers
//              (two in the launches beside the FP64 M2L), digits in the order
//              0, 4, 1, 3, 2 (long and short chunks alternate, so copies keep up);
//   D:         5 levels x 48 (8 x 32) columns of FP32 per job, two TMEM
//              buffers, so one job's epilogue overlaps the next job's MMAs.
// One tcgen05.mma of 128 x 48 x 16 takes about as long as one of 128 x 16 x 16
// (a fixed cost per instruction), which the MMA warp now reaches.  All waits
// are bounded: a wait that runs out sets the error flag, every role stops at
// its next wait, copies and MMAs in flight are waited for (bounded), TMEM is
// freed and the kernel returns.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "bc_internal.h"
#include "pdl.h"

namespace bc {

namespace {

constexpr int kMeta = 4;           // column metadata buffers (tiles)

// The two digit formats.  S digits per operand, L levels kept (digit pairs
// a + b <= L + 1, counted from 1), tiles of N columns: L N <= 256, half of
// the TMEM columns, so that a job's epilogue overlaps the next job's MMAs.
//   5 digits (split modes): 40 bits, levels 2..6, 15 products.
//   7 digits (FP64 mode): 56 bits, levels 2..9, 34 products.  What is dropped
//   (levels >= 10) is below 2^-62 sqrt(K) of max|A'| max|x'|, what is rounded
//   (the operands to 56 bits) 2^-57 sqrt(K) of it: about a tenth of the
//   rounding of a chain of K FP64 additions (2^-53 of the running sums), so
//   the products are no less accurate than the FP64 kernels they stand for.
//   A level sums up to seven pairs; that each |D_g| <= 128 sum_a sum_k
//   |theta_a(k)| stays <= 2^24 is checked row by row when the operator's
//   digits are made (the row's digits used once per level each).
template <int S> struct Fmt;
template <> struct Fmt<kSplitSlices> { static constexpr int L = 5, N = kSplitTileN; };
template <> struct Fmt<kWideSlices> { static constexpr int L = kWideLevels, N = kWideTileN; };
static_assert(Fmt<kSplitSlices>::L * Fmt<kSplitSlices>::N <= 256 && Fmt<kWideSlices>::L * Fmt<kWideSlices>::N <= 256,
              "two TMEM job buffers");

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// UMMA shared-memory descriptor, K-major, no swizzle: core matrices of 8 rows
// x 16 bytes; lbo = byte step between core matrices along K, sbo = byte step
// between 8-row groups.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= uint64_t((saddr & 0x3FFFFu) >> 4);
    d |= uint64_t((lbo >> 4) & 0x3FFFu) << 16;
    d |= uint64_t((sbo >> 4) & 0x3FFFu) << 32;
    d |= uint64_t(1) << 46;   // descriptor version for tcgen05
    return d;                 // base offset 0, absolute LBO, SWIZZLE_NONE
}

// Instruction descriptor: kind::f16, A = B = BF16, D = F32, both K-major.
__host__ __device__ constexpr uint32_t umma_idesc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | (uint32_t(N >> 3) << 17) | (uint32_t(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// waits until at most n (0 or 1) of this thread's cp.async groups are pending
__device__ __forceinline__ void cp_async_wait_pending(int n)
{
    if (n == 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
    else asm volatile("cp.async.wait_group 1;" ::: "memory");
}

// NK MMAs along K (16 columns each) issued from one elected lane of a
// converged warp: the descriptors advance by 16 (256 bytes) per step; the
// first MMA takes `first` as its accumulate flag, the others accumulate.
template <int NK>
__device__ __forceinline__ void umma_kchain_warp(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                 uint32_t first);
template <>
__device__ __forceinline__ void umma_kchain_warp<8>(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                    uint32_t first)
{
    asm volatile(
        "{\n\t.reg .pred p, q, e;\n\t.reg .b64 a, b;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.eq.u32 q, 0, 0;\n\t"
        "mov.b64 a, %1;\n\t"
        "mov.b64 b, %2;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;}"
        ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(first)
        : "memory");
}
template <>
__device__ __forceinline__ void umma_kchain_warp<4>(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                    uint32_t first)
{
    asm volatile(
        "{\n\t.reg .pred p, q, e;\n\t.reg .b64 a, b;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "setp.eq.u32 q, 0, 0;\n\t"
        "mov.b64 a, %1;\n\t"
        "mov.b64 b, %2;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;\n\t"
        "add.s64 a, a, 16;\n\t"
        "add.s64 b, b, 16;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, q;}"
        ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(first)
        : "memory");
}

template <>
__device__ __forceinline__ void umma_kchain_warp<1>(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                    uint32_t first)
{
    asm volatile(
        "{\n\t.reg .pred p, e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;}"
        ::"r"(dtmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(first)
        : "memory");
}
template <>
__device__ __forceinline__ void umma_kchain_warp<9>(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                                    uint32_t first)
{
    umma_kchain_warp<8>(dtmem, adesc, bdesc, idesc, first);
    umma_kchain_warp<1>(dtmem, adesc + 8 * 16, bdesc + 8 * 16, idesc, 1u);
}

__device__ __forceinline__ void umma_commit_warp(uint64_t *bar)
{
    asm volatile(
        "{\n\t.reg .pred e;\n\t"
        "elect.sync _|e, 0xffffffff;\n\t"
        "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(
            smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait on an mbarrier phase by a whole warp that also gives up as soon
// as another role of the CTA has failed (*fail != 0); on running out it sets
// *fail.  The result is uniform over the warp.
__device__ __forceinline__ bool wait_bar(uint64_t *bar, uint32_t parity, long long limit, volatile int *fail)
{
    const uint32_t a = smem_u32(bar);
    for (long long it = 0; it < limit; it++) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(a), "r"(parity)
            : "memory");
        if (__any_sync(0xffffffffu, ok)) return true;
        if ((it & 31) == 31 && __any_sync(0xffffffffu, *fail != 0)) return false;
    }
    *fail = 1;
    return false;
}

// Whether an mbarrier phase has completed, without waiting (uniform over the warp).
__device__ __forceinline__ bool test_bar(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return __any_sync(0xffffffffu, ok);
}

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// S * 2^ex as an FP64 value with integer operations only (bit for bit what the
// hardware conversion and an exponent add give: S rounded to 53 bits, nearest with
// ties to even; results below the normal range, negligible in the split modes,
// become zero).  The tensor launches that run beside the
// FP64 kernels use it, since the hardware conversion occupies the FP64 pipe,
// a small fraction of the FP32 rate on this GPU.  The magnitude is
// normalised so that its leading one is bit 63; its top 53 bits, rounded by
// the 11 below them, are the significand, whose leading one (and a carry from
// rounding up to 2^53) adds into the exponent field.
__device__ __forceinline__ double i64_scaled_int(long long S, int ex)
{
    if (S == 0) return 0.0;
    const unsigned long long sgn = static_cast<unsigned long long>(S) & 0x8000000000000000ull;
    unsigned long long m = S < 0 ? 0ull - static_cast<unsigned long long>(S) : static_cast<unsigned long long>(S);
    const int lz = __clzll(static_cast<long long>(m));
    m <<= lz;
    const unsigned long long rem = m & 0x7FFull, mant = m >> 11;
    const unsigned long long up = (rem > 0x400ull || (rem == 0x400ull && (mant & 1ull))) ? 1ull : 0ull;
    const int e = 63 - lz + ex + 1023;   // biased exponent of the leading one
    if (e <= 0) return 0.0;
    return __longlong_as_double(
        static_cast<long long>((sgn | (static_cast<unsigned long long>(e - 1) << 52)) + mant + up));
}

// v * 2^ex in general (results outside the normal range too).
__device__ __noinline__ double scale_wide(double v, int ex) { return scalbn(v, ex); }

// The levels of one element as one integer, times 2^kShift of the units that the
// column's exponent counts in.
//   5 digits: sum_g D_g 256^(4-g).
//   7 digits: sum_g D_g 256^(7-g), g = 0..7: a product of vectors below 2^-1 in
//   magnitude, K <= 256 of them, so below 2^78; its last 16 bits are below the
//   rounding of the operands (2^17 and more), so it is rounded to a multiple of
//   2^16, which int64 holds, and converted once.
template <int S>
__device__ __forceinline__ long long level_sum(const int (&D)[Fmt<S>::L])
{
    if constexpr (S > 5) {
        const long long top = (long long)D[0] * 65536 + ((long long)D[1] * 256 + D[2]);
        const long long mid = (long long)D[3] * 65536 + ((long long)D[4] * 256 + D[5]);
        const long long low = ((long long)D[6] * 256 + (D[7] + 32768)) >> 16;
        return (top << 24) + mid + low;
    } else {
        const long long top = (long long)D[0] * 65536 + ((long long)D[1] * 256 + D[2]);
        return (top << 16) + ((long long)D[3] * 256 + D[4]);
    }
}
template <int S> constexpr int kShift = S > 5 ? 16 : 0;

// S balanced base-256 digits (BF16 bit patterns) of round(x * 2^(8 S - E)),
// |x| < 2^(E-1), from the FP64 bit pattern by integer operations; written to
// out[0], out[stride], ... (most significant first).  The 5-digit format
// takes subnormal entries as zero (it rounds at 2^-40 of the largest); the
// 7-digit format keeps them.
template <int S>
__device__ __forceinline__ void digits_of(long long bits, int E, uint16_t *out, int stride)
{
    int e = int((bits >> 52) & 0x7FF);
    long long X = 0;
    if (e != 0 || S > 5) {
        long long mant = bits & ((1ll << 52) - 1);
        if (e != 0) mant |= 1ll << 52; else e = 1;
        const int rs = -(e - 1075 + 8 * S - E);   // >= 54 - 8 S
        if (S > 5 && rs <= 0) X = mant << -rs;
        else X = rs >= 62 ? 0 : (mant + (1ll << (rs - 1))) >> rs;
        if (bits < 0) X = -X;
    }
#pragma unroll
    for (int a = S; a >= 2; a--) {
        int d = int(X & 255);
        if (d >= 128) d -= 256;
        X = (X - d) >> 8;
        out[(a - 1) * stride] = uint16_t(__float_as_uint(float(d)) >> 16);
    }
    out[0] = uint16_t(__float_as_uint(float(int(X))) >> 16);   // leading digit, |X| <= 128
}

// Magnitude key of a vector's exponent E: the biased exponent of its largest
// entry.  7-digit format: subnormal entries count as exponent 1, and a vector
// with an infinity or a NaN has no digits (exponent kWideExp: its products
// are formed in FP64 by the epilogue).
template <int S>
__device__ __forceinline__ int exp_key(long long bits)
{
    const int e = int((bits >> 52) & 0x7FF);
    return (S > 5 && e == 0 && (bits & ((1ll << 52) - 1)) != 0) ? 1 : e;
}

// ---------------------------------------------------------------------------
// Digits of scale * cs_k * (leaf vectors): dig[leaf][a][k], dexp[leaf] = E with
// max |scale cs v| < 2^(E-1).  One block per leaf, each thread two neighbouring
// nodes (their digits go out as one word, 41 -> 33 us at 17,491 leaves of 256 nodes
// and 7 digits; bound by integer operations); the np <= kv nodes of a leaf, then zero
// digits up to kv (even).
template <int S>
__global__ void __launch_bounds__(128) k_split_vec(int64_t nleaf, const double *__restrict__ v, double scale,
                                                   const double *__restrict__ cs, uint16_t *__restrict__ dig,
                                                   int32_t *__restrict__ dexp, const uint8_t *__restrict__ active,
                                                   int np, int kv)
{
    griddep_wait();
    griddep_launch_dependents();
    __shared__ int wmax[2][4];
    const int k = 2 * threadIdx.x, nwp = blockDim.x >> 5, w = threadIdx.x >> 5;
    double sk[2];
#pragma unroll
    for (int q = 0; q < 2; q++) sk[q] = (S > 5 && cs && k + q < np) ? scale * cs[k + q] : scale;
    int par = 0;   // the maxima of consecutive leaves in turn: one barrier per leaf
    for (int64_t leaf = blockIdx.x; leaf < nleaf; leaf += gridDim.x, par ^= 1) {
        // a discarded leaf of a truncated tree is no source: zero digits
        const bool on = !active || active[leaf];
        long long bits[2];
#pragma unroll
        for (int q = 0; q < 2; q++)
            bits[q] = __double_as_longlong(sk[q] * (on && k + q < np ? v[leaf * np + k + q] : 0.0));
        const int m = __reduce_max_sync(0xffffffffu, max(exp_key<S>(bits[0]), exp_key<S>(bits[1])));
        if ((threadIdx.x & 31) == 0) wmax[par][w] = m;
        __syncthreads();
        int emax = wmax[par][0];
        for (int q = 1; q < nwp; q++) emax = max(emax, wmax[par][q]);
        const bool wide = S > 5 && emax == 0x7FF;
        const int E = emax ? emax - 1023 + 2 : 0;
        if (k < kv) {
            uint16_t d[2][S];
#pragma unroll
            for (int q = 0; q < 2; q++) digits_of<S>(emax && !wide ? bits[q] : 0ll, E, d[q], 1);
            uint32_t *out = reinterpret_cast<uint32_t *>(dig + leaf * (S * kv) + k);
#pragma unroll
            for (int a = 0; a < S; a++) out[a * (kv / 2)] = uint32_t(d[0][a]) | uint32_t(d[1][a]) << 16;
        }
        if (k == 0) dexp[leaf] = wide ? kWideExp : E;
    }
}

// Digits of scale * s_k * (expansion coefficient k) for the vectors i in
// [i0, i1): vector i < nbox is ea[i] with column scales escale[0..63], else
// eb[i - nbox] with escale[64..127]; its 2*P1 reals (re, im interleaved)
// padded with zeros to 64.  One warp per vector: dig[i][a][64], dexp[i].
template <int S>
__global__ void __launch_bounds__(256) k_split_exp(int64_t i0, int64_t i1, int64_t nbox,
                                                   const double *__restrict__ ea, const double *__restrict__ eb,
                                                   int nreal, double scale, const double *__restrict__ escale,
                                                   uint16_t *__restrict__ dig, int32_t *__restrict__ dexp)
{
    griddep_wait();
    griddep_launch_dependents();
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
    for (int64_t i = i0 + ((blockIdx.x * int64_t(blockDim.x) + threadIdx.x) >> 5); i < i1; i += nw) {
        const int64_t box = i < nbox ? i : i - nbox;
        const double *src = (i < nbox ? ea : eb) + box * nreal;
        const double *sc = escale + (i < nbox ? 0 : kSplitKE);
        const double v0 = lane < nreal ? src[lane] : 0.0, v1 = lane + 32 < nreal ? src[lane + 32] : 0.0;
        const long long b0 = __double_as_longlong(scale * sc[lane] * v0);
        const long long b1 = __double_as_longlong(scale * sc[lane + 32] * v1);
        int m = max(exp_key<S>(b0), exp_key<S>(b1));
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        const bool wide = S > 5 && m == 0x7FF;
        const int E = m ? m - 1023 + 2 : 0;
        uint16_t *out = dig + i * (S * kSplitKE);
        digits_of<S>(m && !wide ? b0 : 0ll, E, out + lane, kSplitKE);
        digits_of<S>(m && !wide ? b1 : 0ll, E, out + lane + 32, kSplitKE);
        if (lane == 0) dexp[i] = wide ? kWideExp : E;
    }
}

// ---------------------------------------------------------------------------
// Operator x columns on tcgen05, KD = 256 or 144 (leaf vectors).
// ---------------------------------------------------------------------------
struct ColMeta {
    double *out;
    int32_t exp;    // E_v + shift - 8 (L + 1)
    int32_t flag;   // 1: multiply by 1/alpha0; 2: no digits (infinity or NaN), exp = shift
    int32_t vec;
    int32_t pad;
};

// Operator digit of the p-th chunk of a K chunk's run: the order 0, S-1, 1, S-2, ...
// alternates long and short MMA runs, so that the copies keep up.
template <int S>
__device__ __forceinline__ int chunk_digit(int p)
{
    return (p & 1) ? S - 1 - (p >> 1) : (p >> 1);
}

// The order of the K chunks (KD = 256 has two): a tile's first row-half job takes
// them as x, 1 - x, its second as 1 - x, x, and the next tile starts with the one
// that this tile did not end on, so that every chunk of B is used twice in a row
// and its buffer is free, for the next tile's gather, while the other chunk's
// MMAs run.  x: the first chunk of a tile; next_first: of the tile after it.
__device__ __forceinline__ int kchunk_at(int x, int h, int i) { return h == 0 ? x ^ i : x ^ i ^ 1; }
__device__ __forceinline__ int next_first(int x, bool two_jobs) { return two_jobs ? x ^ 1 : x; }

template <int KD, int S, bool ICVT>
struct GemmShape {
    static constexpr int N = Fmt<S>::N, L = Fmt<S>::L;
    static constexpr int KC = KD > 144 ? kSplitKC : KD;   // K columns per operator chunk and B buffer
    static constexpr int NKC = KD / KC;
    // operator chunk buffers of 128 columns: each chunk costs some 500 cycles beside its
    // MMAs (six of 64 columns in the same memory: near field of 17,491 leaves, 7 digits,
    // 550 -> 821 us); three, two where the shared memory is short (KD = 144:
    // two whole tiles of B) or left to the FP64 M2L's blocks beside (ICVT)
    static constexpr int NB = KD == 144 || ICVT ? 2 : 3;
    static constexpr int kBSlice = N * KC * 2;         // bytes of one B digit slice of a chunk
    static constexpr int kBChunk = S * kBSlice;        // bytes of one chunk of B (two buffers)
    static constexpr int kChunk = 128 * KC * 2;        // bytes of one operator chunk
    static constexpr int kSBO = (KC / 8) * 128;        // bytes between 8-row groups (A and B)
    static constexpr size_t kSmem =
        2 * size_t(kBChunk) + size_t(NB) * kChunk + kMeta * N * sizeof(ColMeta) + 64 * sizeof(uint64_t);
};

// Roles (16 warps): warp 0 issues the MMAs; warp 1 copies the operator chunks;
// warps 2-7 stage each tile's column metadata and gather its B digits, chunk by
// chunk; warps 8-15 run the epilogues (two warps per TMEM lane quarter, half of
// the columns each).
constexpr int kGemmThreads = 512;
constexpr int kGatherWarp0 = 2;
constexpr int kGatherThreads = 192;
constexpr int kEpiWarp0 = 8;
constexpr int kEpiWarps = 8;
constexpr int kTmemBuf = 256;        // TMEM columns per job buffer (5 x 48 or 8 x 32 used)
constexpr int kNoExp = 0x7FFFFFFF;   // 1/alpha0 is not a power of two

// Barriers (mbarriers in shared memory); counts in brackets:
//   lbar[b] (1)        operator chunk in buffer b has landed (bulk-copy bytes)
//   mbar[b] (1)        the MMAs reading buffer b have completed (commit)
//   job_full[r] (1)    the MMAs of the job in TMEM buffer r have completed (commit)
//   job_empty[r] (8)   the epilogue warps have read TMEM buffer r
//   b_full[u] (6)      B buffer u is filled (one arrival per gather warp)
//   b_empty[u] (1)     no MMA reads B buffer u any more (commit)
//   meta_full[t] (6), meta_empty[t] (8)   metadata buffer t (tile % 4) is filled, done with
// B buffer u holds K chunk u of the current tile (two chunks), or the tiles of
// parity u (one chunk).
struct GemmBars {
    uint64_t lbar[3], mbar[3], job_full[2], job_empty[2], b_full[2], b_empty[2], meta_full[kMeta], meta_empty[kMeta];
    uint32_t tslot;
    int fail;
};
static_assert(sizeof(GemmBars) <= 64 * sizeof(uint64_t), "barrier space");

// Row `row` of an operator times a vector without digits (an infinity or a NaN
// among its entries), in FP64: sum_k opf[k][row] (scale cs_k x_k).
__device__ __noinline__ double plain_product(const SplitGemm &gm, const SplitTile &tl, int row, int vec)
{
    const bool lo = vec < gm.nsplit;
    const double *x = lo ? gm.src0 + int64_t(vec) * gm.kvalid : gm.src1 + int64_t(vec - gm.nsplit) * gm.kvalid;
    const double *cs = lo ? gm.cs0 : gm.cs1;
    const double *op = gm.opf + tl.f_off + row;
    double s = 0.0;
    for (int k = 0; k < gm.kvalid; k++) s = fma(op[int64_t(k) * tl.frows], gm.scale * (cs ? cs[k] : 1.0) * x[k], s);
    return s;
}

// One warp's share of a job: columns [cb, ce) of its 32 TMEM lanes (row `row`
// of the tile's operator, valid where live; ea: its row exponent), from the
// levels' column blocks at ta0.  A batch of columns is worked on side by side,
// without branches, where nothing in it is special (a factor 1/alpha0 that is no
// power of two, a vector without digits, a short batch, a result outside the
// normal range): element after element, each with its own branches, the latencies
// of eight conversions stood one after another (660 cycles per element; a 60 x 32
// tile of the M2L took 5,300 cycles, its MMAs 2,400).
template <int S, bool ICVT>
__device__ __forceinline__ void epilogue_columns(const SplitGemm &gm, const SplitTile &tl, const ColMeta *M, uint32_t ta0,
                                                 int cb, int ce, int row, bool live, int ea, double inv_alpha0)
{
    constexpr int kL = Fmt<S>::L, kN = Fmt<S>::N, kQ = 4;   // columns per batch
    for (int c0 = cb; c0 < ce; c0 += kQ) {   // uniform over the warp
        __syncwarp();   // the lanes part ways below, by their results: tcgen05.ld wants the whole warp
        uint32_t d[kL][kQ];
#pragma unroll
        for (int g = 0; g < kL; g++) tmem_ld4(ta0 + uint32_t(g * kN + c0), d[g]);
        int ex[kQ], flags = c0 + kQ > ce;
        double *out[kQ];
#pragma unroll
        for (int q = 0; q < kQ; q++) {   // (past ce: another column's or stale, not used)
            ex[q] = M[c0 + q].exp + ea + kShift<S>;
            out[q] = M[c0 + q].out + tl.row0 + row;
            if (c0 + q < ce) flags |= M[c0 + q].flag;
        }
        tmem_ld_wait();
        if (!live) continue;
        long long sum[kQ];
#pragma unroll
        for (int q = 0; q < kQ; q++) {
            int D[kL];
#pragma unroll
            for (int g = 0; g < kL; g++) D[g] = __float2int_rn(__uint_as_float(d[g][q]));
            sum[q] = level_sum<S>(D);
        }
        double val[kQ];
        bool odd = flags != 0;
#pragma unroll
        for (int q = 0; q < kQ; q++) {
            if constexpr (ICVT) {
                val[q] = i64_scaled_int(sum[q], ex[q]);
            } else {
                const long long bits = __double_as_longlong(__ll2double_rn(sum[q]));
                const int es = int((bits >> 52) & 0x7FF) + ex[q];
                val[q] = sum[q] == 0 ? 0.0 : __longlong_as_double(bits + ((long long)ex[q] << 52));
                if constexpr (S > 5) odd |= sum[q] != 0 && unsigned(es - 1) >= 0x7FEu;   // es <= 0 or >= 0x7FF
                else if (sum[q] != 0 && es <= 0) val[q] = 0.0;
            }
        }
        if (!odd) {
#pragma unroll
            for (int q = 0; q < kQ; q++) *out[q] = val[q];
            continue;
        }
#pragma unroll
        for (int q = 0; q < kQ; q++) {
            if (c0 + q >= ce) continue;
            double v = val[q];
            const int f = M[c0 + q].flag;
            if constexpr (S > 5) {
                if (f & 2) v = scale_wide(plain_product(gm, tl, row, M[c0 + q].vec), M[c0 + q].exp);
                else if (sum[q] != 0) v = scale_wide(__ll2double_rn(sum[q]), ex[q]);
            }
            if (f & 1) v *= inv_alpha0;
            *out[q] = v;
        }
    }
}

// The metadata of a column: digit exponent ev, power-of-two factors folded in.
template <int S>
__device__ __forceinline__ ColMeta col_meta(const SplitCol &c, int ev, int inv_alpha_exp)
{
    ColMeta m;
    const bool plain = S > 5 && ev == kWideExp;
    m.out = c.out;
    m.exp = (c.ctl >> 1) + (plain ? 0 : ev - 8 * (Fmt<S>::L + 1));
    m.flag = c.ctl & 1;
    if (m.flag && inv_alpha_exp != kNoExp) {   // 1/alpha0 a power of two: an exponent shift
        m.exp += inv_alpha_exp;
        m.flag = 0;
    }
    if (plain) m.flag |= 2;
    m.vec = c.vec;
    m.pad = 0;
    return m;
}

// 5 digits: the second launch bound caps the registers at 64 per thread: 16
// warps x 64 leave room, in each SM sub-partition's register file, for the
// FP64 M2L blocks that run beside a near-field CTA.  Two CTAs never share an SM
// (shared memory allows one).
template <int KD, int S, bool ICVT>
__global__ void __launch_bounds__(kGemmThreads, S == kSplitSlices ? 2 : 1)
k_split_gemm(const __grid_constant__ SplitGemm gm, double inv_alpha0, int inv_alpha_exp, int32_t *__restrict__ err, long long wait_limit,
             int withhold)
{
    using Sh = GemmShape<KD, S, ICVT>;
    constexpr int kN = Sh::N, kL = Sh::L, NB = Sh::NB, NKC = Sh::NKC;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *Bs = smem, *As = smem + 2 * Sh::kBChunk;                    // 2 x kBChunk, NB x kChunk
    ColMeta *meta = reinterpret_cast<ColMeta *>(As + NB * Sh::kChunk);   // [kMeta][kN]
    GemmBars *bars = reinterpret_cast<GemmBars *>(meta + kMeta * kN);
    volatile int *fail = &bars->fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tslot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < NB; i++) {
            mbar_init(&bars->lbar[i], 1);
            mbar_init(&bars->mbar[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&bars->job_full[i], 1);
            mbar_init(&bars->job_empty[i], kEpiWarps);
            mbar_init(&bars->b_full[i], kGatherThreads / 32);
            mbar_init(&bars->b_empty[i], 1);
        }
        for (int i = 0; i < kMeta; i++) {
            mbar_init(&bars->meta_full[i], kGatherThreads / 32);
            mbar_init(&bars->meta_empty[i], kEpiWarps);
        }
        bars->fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tslot;
    // tensor memory and barriers are set up: now wait for the inputs
    griddep_wait();
    griddep_launch_dependents();
    const int step = gridDim.x;
    // B buffer and phase parity of chunk kc of the CTA's tile k
    auto bbuf = [](int k, int kc) { return NKC == 2 ? kc : k & 1; };
    auto bpar = [](int k) { return uint32_t(NKC == 2 ? k & 1 : (k >> 1) & 1); };

    if (warp == 0) {
        // ---------------- MMAs ----------------
        const uint64_t adesc0 = umma_desc(smem_u32(As), 128, Sh::kSBO);
        const uint64_t bdesc0 = umma_desc(smem_u32(Bs), 128, Sh::kSBO);
        long long G = 0, last_commit = -1;   // operator chunks consumed
        int job = 0, k = 0, x = 0;
        bool failed = false;
        for (int tile = blockIdx.x; tile < gm.ntiles && !failed; tile += step, k++) {
            const bool two = gm.tiles[tile].rows > 128;
            for (int h = 0; h <= int(two) && !failed; h++, job++) {
                const int r = job & 1;
                if (job >= 2 && !wait_bar(&bars->job_empty[r], uint32_t(((job - 2) >> 1) & 1), wait_limit, fail)) {
                    failed = true;
                    break;
                }
                for (int i = 0; i < NKC && !failed; i++) {
                    const int kc = NKC == 2 ? kchunk_at(x, h, i) : 0, u = bbuf(k, kc);
                    if (h == 0 && !wait_bar(&bars->b_full[u], bpar(k), wait_limit, fail)) {
                        failed = true;
                        break;
                    }
                    tc_fence_after();
                    for (int pos = 0; pos < S; pos++, G++) {
                        const int buf = int(G % NB);
                        if (!wait_bar(&bars->lbar[buf], uint32_t((G / NB) & 1), wait_limit, fail)) {
                            failed = true;
                            break;
                        }
                        tc_fence_after();
                        const int a = chunk_digit<S>(pos);   // 0-based digit of A
                        const int nb = min(S, kL - a);       // B digit slices 0 .. nb-1 pair with it
                        const uint64_t ad = adesc0 + uint64_t(buf) * (Sh::kChunk >> 4);
                        const uint64_t bd = bdesc0 + uint64_t(u) * (Sh::kBChunk >> 4);
                        const uint32_t dcol = tmem + uint32_t(r * kTmemBuf + a * kN);
                        // slices 0 .. nb-1 lie one after another (an nb kN-row B
                        // operand) and feed levels a .. a+nb-1, adjacent TMEM
                        // column blocks: one MMA chain of N = nb kN per chunk.  The
                        // first chunk (a = 0) starts levels 0 .. S-1; where L > S the
                        // second one starts level L-1 (its last slice, apart).
                        if (kL > S && pos == 1 && i == 0) {
                            umma_kchain_warp<Sh::KC / 16>(dcol, ad, bd, umma_idesc(128, (nb - 1) * kN), 1u);
                            umma_kchain_warp<Sh::KC / 16>(dcol + uint32_t((nb - 1) * kN), ad,
                                                          bd + uint64_t(nb - 1) * (Sh::kBSlice >> 4),
                                                          umma_idesc(128, kN), 0u);
                        } else {
                            umma_kchain_warp<Sh::KC / 16>(dcol, ad, bd, umma_idesc(128, nb * kN), pos == 0 && i == 0 ? 0u : 1u);
                        }
                        umma_commit_warp(&bars->mbar[buf]);
                        last_commit = G;
                    }
                    if (!failed && h == int(two)) umma_commit_warp(&bars->b_empty[u]);   // the tile's last use
                }
                if (failed) break;
                umma_commit_warp(&bars->job_full[r]);
            }
            x = next_first(x, two);
        }
        if (failed) {
            *fail = 1;
            int dummy = 0;   // bounded wait, without the failure shortcut
            if (last_commit >= 0)
                wait_bar(&bars->mbar[int(last_commit % NB)], uint32_t((last_commit / NB) & 1), wait_limit,
                         &dummy);
        }
    } else if (warp == 1) {
        // ---------------- operator chunk copies ----------------
        long long n = 0;   // chunks issued
        int x = 0;
        bool failed = false;
        for (int tile = blockIdx.x; tile < gm.ntiles && !failed; tile += step) {
            const SplitTile tl = gm.tiles[tile];
            const int mh = tl.rows > 128 ? 2 : 1;
            // an operator of at most 64 rows is copied twice, to rows 0-63
            // and 64-127, so that every TMEM lane quarter holds a result
            const int copies = tl.rows <= 64 ? 2 : 1;
            for (int h = 0; h < mh && !failed; h++) {
                const uint32_t bytes = uint32_t((min(128, tl.rows - 128 * h) + 7) / 8) * 8 * Sh::KC * 2;
                for (int g = 0; g < S * NKC; g++, n++) {
                    const int buf = int(n % NB);
                    // buffer free once the MMAs of chunk n - NB have completed
                    if (n >= NB &&
                        !wait_bar(&bars->mbar[buf], uint32_t(((n - NB) / NB) & 1), wait_limit, fail)) {
                        failed = true;
                        break;
                    }
                    if (withhold) continue;   // diagnostics: the MMA warp's first wait runs out
                    const int a = chunk_digit<S>(g % S), kc = NKC == 2 ? kchunk_at(x, h, g / S) : 0;
                    const uint8_t *src = gm.ops + tl.a_off + size_t((a * mh + h) * NKC + kc) * Sh::kChunk;
                    if (lane == 0) {
                        mbar_expect_tx(&bars->lbar[buf], bytes * copies);
                        for (int cp = 0; cp < copies; cp++) {
                            uint8_t *dst = As + buf * Sh::kChunk + cp * (Sh::kChunk / 2);
                            for (uint32_t q = 0; q < bytes; q += 16384)
                                bulk_g2s(dst + q, src + q, min(16384u, bytes - q), &bars->lbar[buf]);
                        }
                    }
                    __syncwarp();
                }
            }
            x = next_first(x, mh == 2);
        }
        if (failed && !withhold) {
            // copies still in flight: at most the last NB issued
            int dummy = 0;
            for (long long q = n > NB ? n - NB : 0; q < n; q++)
                wait_bar(&bars->lbar[int(q % NB)], uint32_t((q / NB) & 1), wait_limit, &dummy);
        }
    } else if (warp < kEpiWarp0) {
        // ---------------- column metadata and B gather ----------------
        // kTPC threads per column, each with its own column record (the records,
        // columns and exponents of the next tiles are in flight) and the 16-byte
        // pieces j, j + kTPC, ... of the column's chunk; no barrier among them
        constexpr int kTPC = kGatherThreads / kN, kRow = Sh::KC / 8, kPieces = S * kRow;
        static_assert(kTPC * kN == kGatherThreads, "whole columns");
        const int gt = tid - 32 * kGatherWarp0, c = gt / kTPC, j = gt % kTPC;
        const int nt = blockIdx.x < gm.ntiles ? (gm.ntiles - 1 - int(blockIdx.x)) / step + 1 : 0;
        auto tile_at = [&](int k) -> SplitTile {
            SplitTile t{};
            if (k < nt) t = gm.tiles[blockIdx.x + k * step];
            return t;
        };
        SplitTile tl = tile_at(0), tl1 = tile_at(1), tl2 = tile_at(2);
        SplitCol col{}, col1{};
        int ev = 0, x = 0;
        if (c < tl.cnt) col = gm.cols[tl.p0 + c];
        if (c < tl1.cnt) col1 = gm.cols[tl1.p0 + c];
        if (j == 0 && c < tl.cnt) ev = gm.dexp[col.vec];
        int pend = -1, pend_meta = -1;   // B buffer (and metadata) whose copies are under way
        bool ok = true;
        auto complete = [&](int allowed) {
            if (pend < 0) return;   // uniform
            if (allowed) cp_async_wait_pending(1);
            else cp_async_wait_pending(0);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bars->b_full[pend]);
                if (pend_meta >= 0) mbar_arrive(&bars->meta_full[pend_meta]);
            }
            pend = -1;
        };
        // before a wait that does not end at once, what is under way is completed:
        // the MMAs that free a buffer may need it first
        auto wait_for = [&](uint64_t *bar, uint32_t parity) -> bool {
            if (test_bar(bar, parity)) return true;
            complete(0);
            return wait_bar(bar, parity, wait_limit, fail);
        };
        for (int k = 0; k < nt && ok; k++) {
            for (int i = 0; i < NKC; i++) {
                const int kc = NKC == 2 ? x ^ i : 0, u = bbuf(k, kc), first_use = NKC == 2 ? 1 : 2;
                if (i == 0 && k >= kMeta)
                    ok = wait_for(&bars->meta_empty[k % kMeta], uint32_t(((k - kMeta) / kMeta) & 1));
                if (ok && k >= first_use) ok = wait_for(&bars->b_empty[u], bpar(k - first_use));
                if (!ok) break;   // uniform over the warp
                if (c < tl.cnt) {
                    if (i == 0 && j == 0) meta[(k % kMeta) * kN + c] = col_meta<S>(col, ev, inv_alpha_exp);
                    const uint16_t *src = gm.dig + size_t(col.vec) * (S * KD) + kc * Sh::KC;
                    uint8_t *dst = Bs + u * Sh::kBChunk + (c >> 3) * Sh::kSBO + (c & 7) * 16;
                    for (int q = j; q < kPieces; q += kTPC) {
                        const int sl = q / kRow, kg = q % kRow;
                        cp_async16(dst + sl * Sh::kBSlice + kg * 128, src + sl * KD + kg * 8);
                    }
                }
                cp_async_commit();
                complete(1);   // the previous unit
                pend = u;
                pend_meta = i == 0 ? k % kMeta : -1;
                if (i == NKC - 1) {
                    // one step of the following tiles' chains
                    x = next_first(x, tl.rows > 128);
                    tl = tl1;
                    col = col1;
                    if (j == 0 && c < tl.cnt) ev = gm.dexp[col.vec];
                    tl1 = tl2;
                    if (c < tl1.cnt) col1 = gm.cols[tl1.p0 + c];
                    tl2 = tile_at(k + 3);
                }
            }
        }
        if (ok) complete(0);
        cp_async_wait_all();
    } else {
        // ---------------- epilogues ----------------
        // warp w reads TMEM lanes 32(w%4)..32(w%4)+31.  Operators of more
        // than 64 rows: rows 32(w%4)+lane of the job's row half, warps 8-11
        // the first half of the columns, warps 12-15 the second.  Up to 64
        // rows (held twice): rows 32(w%2)+lane, lane quarters 0-1 the first
        // half of the columns and 2-3 the second, split between the two warps
        // of a quarter.
        const int wq = warp & 3, half = (warp - kEpiWarp0) >> 2;
        int job = 0, k = 0;
        bool failed = false;
        SplitTile tl{}, ntl{};
        if (blockIdx.x < gm.ntiles) ntl = gm.tiles[blockIdx.x];
        for (int tile = blockIdx.x; tile < gm.ntiles && !failed; tile += step, k++) {
            tl = ntl;
            if (tile + step < gm.ntiles) ntl = gm.tiles[tile + step];   // while this tile is worked on
            const int mh = tl.rows > 128 ? 2 : 1;
            const ColMeta *M = meta + (k % kMeta) * kN;
            if (!wait_bar(&bars->meta_full[k % kMeta], uint32_t((k / kMeta) & 1), wait_limit, fail)) break;
            for (int h = 0; h < mh; h++, job++) {
                const int r = job & 1;
                const bool small = tl.rows <= 64;
                const int row = small ? (wq & 1) * 32 + lane : h * 128 + wq * 32 + lane;
                const bool live = row < tl.rows;
                const int ea = live ? gm.op_exp[tl.exp_off + row] : 0;
                const int cb = small ? (wq >> 1) * (kN / 2) + half * (kN / 4) : half * (kN / 2);
                const int ce = min(tl.cnt, cb + (small ? kN / 4 : kN / 2));
                if (!wait_bar(&bars->job_full[r], uint32_t((job >> 1) & 1), wait_limit, fail)) {
                    failed = true;
                    break;
                }
                tc_fence_after();
                epilogue_columns<S, ICVT>(gm, tl, M, tmem + (uint32_t(wq * 32) << 16) + uint32_t(r * kTmemBuf), cb, ce,
                                          row, live, ea, inv_alpha0);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->job_empty[r]);
            }
            if (failed) break;
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->meta_empty[k % kMeta]);
        }
    }
    if (*fail && tid == 0) atomicExch(err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

// ---------------------------------------------------------------------------
// K = 64 (expansions, and leaf vectors of small orders): one operator of up to
// 128 rows is 16 KB per digit, so all its digits stay in shared memory (80 or
// 112 KB) while a CTA works through its tiles, a contiguous range of the list,
// in which consecutive tiles share an operator; the operator is fetched again
// only where it changes.  Streamed through three chunk buffers like the larger
// ones, a tile took 5.2 us, four times its MMAs: each chunk's copy latency
// stood between short MMA runs.  17,491 leaves, 30 terms, 7 digits, alone: the
// M2L's tiles 427 -> 262 us, expansion-to-leaf and W list 168 -> 134 us (176 and 87
// with the epilogue of four columns side by side: per M2L tile 4,100 cycles, its MMAs
// 2,400, its epilogue 2,600-3,500; per expansion-to-leaf tile 6,600, the epilogue
// 5,700.  Loading a batch's levels before the last one was stored spilled registers:
// 241 and 107 us).
//   warp 0      MMAs: per tile one chain per operator digit, issued back to back
//   warp 1      operator copies
//   warps 2-7   column metadata and digits: 192 / N threads per column, each with
//               its own column record (the records, columns and exponents of the
//               next three tiles are in flight), so no barrier among them;
//               three B buffers
//   warps 8-15  epilogues, two TMEM buffers
// Barriers (counts): a_full (1: bulk-copy bytes), a_free (1: commit of the last
// tile on the operator), b_full[3], meta_full[4] (6: one per gather warp),
// b_empty[3] (1: commit), job_full[2] (1: commit), job_empty[2], meta_empty[4]
// (8: one per epilogue warp).
// ---------------------------------------------------------------------------
constexpr int kB64 = 3, kM64 = kMeta;
template <int S>
struct Shape64 {
    static constexpr int N = Fmt<S>::N, L = Fmt<S>::L;
    static constexpr int kA = 128 * 64 * 2;            // bytes of one operator digit
    static constexpr int kBSlice = N * 64 * 2, kBTile = S * kBSlice;
    static constexpr size_t kSmem =
        size_t(S) * kA + kB64 * size_t(kBTile) + kM64 * N * sizeof(ColMeta) + 32 * sizeof(uint64_t);
};
struct Bars64 {
    uint64_t a_full, a_free, b_full[kB64], b_empty[kB64], meta_full[kM64], meta_empty[kM64], job_full[2], job_empty[2];
    uint32_t tslot;
    int fail;
};
static_assert(sizeof(Bars64) <= 32 * sizeof(uint64_t), "barrier space");

template <int S, bool ICVT>
__global__ void __launch_bounds__(kGemmThreads, S == kSplitSlices ? 2 : 1)
k_gemm64(const __grid_constant__ SplitGemm gm, double inv_alpha0, int inv_alpha_exp, int32_t *__restrict__ err,
         long long wait_limit, int withhold)
{
    using Sh = Shape64<S>;
    constexpr int kN = Sh::N, kL = Sh::L;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *As = smem, *Bs = smem + S * Sh::kA;
    ColMeta *meta = reinterpret_cast<ColMeta *>(Bs + kB64 * Sh::kBTile);   // [kM64][kN]
    Bars64 *bars = reinterpret_cast<Bars64 *>(meta + kM64 * kN);
    volatile int *fail = &bars->fail;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&bars->tslot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&bars->a_full, 1);
        mbar_init(&bars->a_free, 1);
        for (int i = 0; i < kB64; i++) {
            mbar_init(&bars->b_full[i], kGatherThreads / 32);
            mbar_init(&bars->b_empty[i], 1);
        }
        for (int i = 0; i < kM64; i++) {
            mbar_init(&bars->meta_full[i], kGatherThreads / 32);
            mbar_init(&bars->meta_empty[i], kEpiWarps);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&bars->job_full[i], 1);
            mbar_init(&bars->job_empty[i], kEpiWarps);
        }
        bars->fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tslot;
    griddep_wait();
    griddep_launch_dependents();
    // this CTA's tiles
    const int t0 = int(int64_t(gm.ntiles) * blockIdx.x / gridDim.x), t1 = int(int64_t(gm.ntiles) * (blockIdx.x + 1) / gridDim.x);
    const int nt = t1 - t0;

    if (warp == 0) {
        const uint64_t adesc0 = umma_desc(smem_u32(As), 128, 1024), bdesc0 = umma_desc(smem_u32(Bs), 128, 1024);
        int ops = 0;          // operators begun
        int64_t cur = -1;
        bool ok = true;
        int k = 0;
        int64_t a_off = nt > 0 ? gm.tiles[t0].a_off : -1, next = nt > 1 ? gm.tiles[t0 + 1].a_off : -1;
        for (; k < nt; k++) {
            const int64_t after = k + 2 < nt ? gm.tiles[t0 + k + 2].a_off : -1;   // used in two tiles' time
            if (a_off != cur) {
                ok = wait_bar(&bars->a_full, uint32_t(ops & 1), wait_limit, fail);
                ops++;
                cur = a_off;
            }
            const int r = k & 1, buf = k % kB64;
            if (ok && k >= 2) ok = wait_bar(&bars->job_empty[r], uint32_t(((k - 2) >> 1) & 1), wait_limit, fail);
            if (ok) ok = wait_bar(&bars->b_full[buf], uint32_t((k / kB64) & 1), wait_limit, fail);
            if (!ok) break;
            tc_fence_after();
            const uint64_t bd = bdesc0 + uint64_t(buf) * (Sh::kBTile >> 4);
#pragma unroll
            for (int a = 0; a < S; a++) {   // the chains of k_split_gemm, in the order 0..S-1
                const int nb = S < kL - a ? S : kL - a;
                const uint64_t ad = adesc0 + uint64_t(a) * (Sh::kA >> 4);
                const uint32_t dcol = tmem + uint32_t(r * kTmemBuf + a * kN);
                if (kL > S && a == 1) {
                    umma_kchain_warp<4>(dcol, ad, bd, umma_idesc(128, (nb - 1) * kN), 1u);
                    umma_kchain_warp<4>(dcol + uint32_t((nb - 1) * kN), ad, bd + uint64_t(nb - 1) * (Sh::kBSlice >> 4),
                                        umma_idesc(128, kN), 0u);
                } else {
                    umma_kchain_warp<4>(dcol, ad, bd, umma_idesc(128, nb * kN), a == 0 ? 0u : 1u);
                }
            }
            umma_commit_warp(&bars->b_empty[buf]);
            umma_commit_warp(&bars->job_full[r]);
            if (next >= 0 && next != a_off) umma_commit_warp(&bars->a_free);
            a_off = next;
            next = after;
        }
        if (!ok) {
            *fail = 1;
            int dummy = 0;   // MMAs in flight: those of the last tile issued
            if (k > 0) wait_bar(&bars->job_full[(k - 1) & 1], uint32_t(((k - 1) >> 1) & 1), wait_limit, &dummy);
        }
    } else if (warp == 1) {
        int ops = 0;
        int64_t cur = -1;
        for (int k = 0; k < nt && !withhold; k++) {
            const SplitTile tl = gm.tiles[t0 + k];
            if (tl.a_off == cur) continue;
            cur = tl.a_off;
            if (ops > 0 && !wait_bar(&bars->a_free, uint32_t((ops - 1) & 1), wait_limit, fail)) break;
            const uint32_t bytes = uint32_t((tl.rows + 7) / 8) * 1024;
            // an operator of at most 64 rows is held twice, in rows 0-63 and
            // 64-127, so that every TMEM lane quarter holds a result
            const int copies = tl.rows <= 64 ? 2 : 1;
            if (lane == 0) {
                mbar_expect_tx(&bars->a_full, uint32_t(S) * bytes * copies);
                for (int a = 0; a < S; a++)
                    for (int cp = 0; cp < copies; cp++)
                        bulk_g2s(As + a * Sh::kA + cp * (Sh::kA / 2), gm.ops + tl.a_off + int64_t(a) * tl.astride, bytes,
                                 &bars->a_full);
            }
            __syncwarp();
            ops++;
        }
        if (ops > 0) {   // a copy in flight lands before the CTA ends
            int dummy = 0;
            wait_bar(&bars->a_full, uint32_t((ops - 1) & 1), wait_limit, &dummy);
        }
    } else if (warp < kEpiWarp0) {
        // kTPC threads per column, each thread the 16-byte pieces j, j + kTPC, ...
        constexpr int kTPC = kGatherThreads / kN, kPieces = S * 8;
        static_assert(kTPC * kN == kGatherThreads, "whole columns");
        const int gt = tid - 32 * kGatherWarp0, c = gt / kTPC, j = gt % kTPC;
        SplitTile tl{}, tl1{}, tl2{};
        SplitCol col{}, col1{};
        int ev = 0;
        if (nt > 0) tl = gm.tiles[t0];
        if (nt > 1) tl1 = gm.tiles[t0 + 1];
        if (nt > 2) tl2 = gm.tiles[t0 + 2];
        if (c < tl.cnt) col = gm.cols[tl.p0 + c];
        if (c < tl1.cnt) col1 = gm.cols[tl1.p0 + c];
        if (j == 0 && c < tl.cnt) ev = gm.dexp[col.vec];
        for (int k = 0; k <= nt; k++) {
            if (k < nt) {
                bool ok = k < kM64 || wait_bar(&bars->meta_empty[k % kM64], uint32_t(((k - kM64) / kM64) & 1), wait_limit, fail);
                if (ok && k >= kB64) ok = wait_bar(&bars->b_empty[k % kB64], uint32_t(((k - kB64) / kB64) & 1), wait_limit, fail);
                if (!ok) break;   // uniform over the warp
                if (c < tl.cnt) {
                    if (j == 0) meta[(k % kM64) * kN + c] = col_meta<S>(col, ev, inv_alpha_exp);
                    const uint16_t *src = gm.dig + size_t(col.vec) * (S * 64);
                    uint8_t *dst = Bs + (k % kB64) * Sh::kBTile + (c >> 3) * 1024 + (c & 7) * 16;
                    for (int q = j; q < kPieces; q += kTPC)
                        cp_async16(dst + (q >> 3) * Sh::kBSlice + (q & 7) * 128, src + q * 8);
                }
                cp_async_commit();
            }
            if (k > 0) {   // tile k - 1 has landed
                cp_async_wait_pending(k < nt ? 1 : 0);
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&bars->b_full[(k - 1) % kB64]);
                    mbar_arrive(&bars->meta_full[(k - 1) % kM64]);
                }
            }
            // one step of the following tiles' chains
            tl = tl1;
            col = col1;
            if (j == 0 && c < tl.cnt) ev = gm.dexp[col.vec];
            tl1 = tl2;
            if (c < tl1.cnt) col1 = gm.cols[tl1.p0 + c];
            tl2.cnt = 0;
            if (k + 3 < nt) tl2 = gm.tiles[t0 + k + 3];
        }
        cp_async_wait_all();
    } else {
        // rows and columns of a warp as in k_split_gemm
        const int wq = warp & 3, half = (warp - kEpiWarp0) >> 2;
        SplitTile tl{}, ntl{};
        if (nt > 0) ntl = gm.tiles[t0];
        int exp_off = -1, ea = 0;
        for (int k = 0; k < nt; k++) {
            tl = ntl;
            if (k + 1 < nt) ntl = gm.tiles[t0 + k + 1];   // while this tile is worked on
            const int r = k & 1;
            const bool small = tl.rows <= 64;
            const int row = small ? (wq & 1) * 32 + lane : wq * 32 + lane;
            const bool live = row < tl.rows;
            if (tl.exp_off != exp_off) {
                exp_off = tl.exp_off;
                ea = live ? gm.op_exp[exp_off + row] : 0;
            }
            if (!wait_bar(&bars->meta_full[k % kM64], uint32_t((k / kM64) & 1), wait_limit, fail)) break;
            const int cb = small ? (wq >> 1) * (kN / 2) + half * (kN / 4) : half * (kN / 2);
            const int ce = min(tl.cnt, cb + (small ? kN / 4 : kN / 2));
            if (!wait_bar(&bars->job_full[r], uint32_t((k >> 1) & 1), wait_limit, fail)) break;
            tc_fence_after();
            epilogue_columns<S, ICVT>(gm, tl, meta + (k % kM64) * kN, tmem + (uint32_t(wq * 32) << 16) + uint32_t(r * kTmemBuf),
                                      cb, ce, row, live, ea, inv_alpha0);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(&bars->job_empty[r]);
                mbar_arrive(&bars->meta_empty[k % kM64]);
            }
        }
    }
    if (*fail && tid == 0) atomicExch(err, 1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

int g_sms = 0;
// Every tensor-core launch takes more than half of an SM's shared memory, so
// that no two of their CTAs share an SM (each holds all 512 TMEM columns while
// it runs).
constexpr size_t kSmemMin = 116 * 1024, kSmemMax = 227 * 1024;
template <int KD, int S, bool ICVT>
constexpr size_t gemm_smem()
{
    if constexpr (KD == 64) return Shape64<S>::kSmem;
    else return GemmShape<KD, S, ICVT>::kSmem;
}

template <int KD, int S, bool ICVT>
constexpr auto gemm_kernel()
{
    static_assert(gemm_smem<KD, S, ICVT>() >= kSmemMin && gemm_smem<KD, S, ICVT>() <= kSmemMax, "one tensor CTA per SM");
    if constexpr (KD == 64) return k_gemm64<S, ICVT>;
    else return k_split_gemm<KD, S, ICVT>;
}

template <int KD, int S, bool ICVT>
cudaError_t prepare_gemm()
{
    return cudaFuncSetAttribute(gemm_kernel<KD, S, ICVT>(), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                int(gemm_smem<KD, S, ICVT>()));
}

}  // namespace

cudaError_t split_prepare()
{
    cudaError_t e = cudaSuccess;
    for (auto f : {prepare_gemm<256, kSplitSlices, false>, prepare_gemm<256, kSplitSlices, true>,
                   prepare_gemm<64, kSplitSlices, false>, prepare_gemm<64, kSplitSlices, true>,
                   prepare_gemm<256, kWideSlices, false>, prepare_gemm<144, kWideSlices, false>,
                   prepare_gemm<64, kWideSlices, false>})
        if (e == cudaSuccess) e = f();
    // the digit kernels run before and beside the tensor launches: the
    // largest shared-memory carveout (see fp64_prepare)
    for (const void *k : {(const void *)k_split_vec<kSplitSlices>, (const void *)k_split_vec<kWideSlices>,
                          (const void *)k_split_exp<kSplitSlices>, (const void *)k_split_exp<kWideSlices>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    int dev = 0;
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_sms, cudaDevAttrMultiProcessorCount, dev);
    return e;
}

int split_sm_count() { return g_sms > 0 ? g_sms : 152; }

SplitGemm gemm_group_v(const SplitTables &T, const SplitTree &s, int dir, const SplitTile *tiles, const SplitCol *cols,
                       int n, const double *vin, double scale)
{
    SplitGemm g;
    g.tiles = tiles; g.cols = cols; g.ntiles = n;
    g.ops = T.ops[0][dir]; g.op_exp = T.op_exp[0][dir];
    g.dig = s.vdig; g.dexp = s.vexp;
    g.opf = T.opf[0][dir];
    g.src0 = vin; g.cs0 = T.vscale[dir];
    g.scale = scale;
    g.kvalid = T.np;
    return g;
}

SplitGemm gemm_group_e(const SplitTables &T, const SplitTree &s, int dir, const SplitTile *tiles, const SplitCol *cols,
                       int n, const double2 *ea, const double2 *eb, int64_t nbox, int P1, double scale)
{
    SplitGemm g;
    g.tiles = tiles; g.cols = cols; g.ntiles = n;
    g.ops = T.ops[1][dir]; g.op_exp = T.op_exp[1][dir];
    g.dig = s.edig; g.dexp = s.eexp;
    g.opf = T.opf[1][dir];
    g.src0 = reinterpret_cast<const double *>(ea); g.cs0 = T.escale[dir];
    g.src1 = reinterpret_cast<const double *>(eb); g.cs1 = T.escale[dir] + kSplitKE;
    g.nsplit = nbox;
    g.scale = scale;
    g.kvalid = 2 * P1;
    return g;
}

namespace {

// Columns of the segments (blockIdx.y), one entry per thread.
__global__ void __launch_bounds__(256) k_make_cols(const __grid_constant__ ColLists cl)
{
    const ColSeg &s = cl.seg[blockIdx.y];
    const bool adj = s.dir == 1;
    // the leaf whose list holds entry e: the last with ptr[leaf] <= e
    auto owner = [&](const int32_t *ptr, int e) {
        int64_t lo = 0, hi = cl.nleaf - 1;
        while (lo < hi) {
            const int64_t mid = (lo + hi + 1) >> 1;
            if (ptr[mid] <= e) lo = mid; else hi = mid - 1;
        }
        return int(lo);
    };
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < s.n; i += int64_t(gridDim.x) * blockDim.x) {
        const int e = s.perm[i];
        int vec = e, shift = 0, inv = 0;   // power-of-two factor r^2 / r_0^2, or the factor 1/alpha0
        int64_t at = e;
        switch (s.kind) {
        case ColKind::Near:
            vec = cl.near_src[e];
            shift = -2 * cl.leaf_level[adj ? owner(cl.near_ptr, e) : vec];
            break;
        case ColKind::LeafA:
            if (adj) inv = 1; else shift = -2 * cl.leaf_level[e];
            at = cl.leaf_box[e];
            break;
        case ColKind::X:
            vec = cl.x_src[e];
            if (adj) inv = 1; else shift = -2 * (cl.box_level[cl.x_box[e]] - 1);
            break;
        case ColKind::L2P:
            vec = cl.leaf_box[e];
            if (adj) shift = -2 * cl.leaf_level[e];
            break;
        case ColKind::W:
            vec = cl.w_src[e];
            if (adj) shift = -2 * cl.leaf_level[owner(cl.w_ptr, e)];
            break;
        case ColKind::V:
            vec = cl.v_src[e];
            inv = adj;
            break;
        }
        SplitCol c;
        c.vec = int32_t(s.vec0 + vec);
        c.ctl = shift * 2 + inv;
        c.out = s.out + at * s.stride;
        s.cols[i] = c;
    }
}

}  // namespace

cudaError_t launch_make_cols(const ColLists &cl, cudaStream_t st)
{
    int64_t n = 0;
    for (int i = 0; i < cl.nseg; i++) n = std::max(n, cl.seg[i].n);
    if (n <= 0) return cudaSuccess;
    k_make_cols<<<dim3(unsigned(std::min<int64_t>((n + 255) / 256, 152 * 4)), unsigned(cl.nseg)), 256, 0, st>>>(cl);
    return cudaGetLastError();
}

cudaError_t launch_split_digits_vec(const SplitTables &T, int dir, int64_t nleaf, const double *v, double scale,
                                    uint16_t *dig, int32_t *dexp, cudaStream_t st, const uint8_t *active)
{
    if (nleaf <= 0) return cudaSuccess;
    const int grid = int(std::min<int64_t>(nleaf, 152 * 16)), nth = (T.kv / 2 + 31) / 32 * 32;
    if (T.slices == kWideSlices)
        return launch_pdl(k_split_vec<kWideSlices>, grid, nth, 0, st, nleaf, v, scale, T.vscale[dir], dig, dexp, active,
                          T.np, T.kv);
    return launch_pdl(k_split_vec<kSplitSlices>, grid, nth, 0, st, nleaf, v, scale, (const double *)nullptr, dig, dexp,
                      active, T.np, T.kv);
}

cudaError_t launch_split_digits_exp(const SplitTables &T, int dir, int64_t i0, int64_t i1, int64_t nbox,
                                    const double2 *ea, const double2 *eb, int P1, double scale, uint16_t *dig,
                                    int32_t *dexp, cudaStream_t st)
{
    if (i1 <= i0) return cudaSuccess;
    const int grid = int(std::min<int64_t>((i1 - i0 + 7) / 8, 152 * 16));
    return launch_pdl(T.slices == kWideSlices ? k_split_exp<kWideSlices> : k_split_exp<kSplitSlices>, grid, 256, 0, st,
                      i0, i1, nbox, reinterpret_cast<const double *>(ea), reinterpret_cast<const double *>(eb), 2 * P1,
                      scale, T.escale[dir], dig, dexp);
}

cudaError_t launch_split_gemm(const SplitTables &T, const SplitGemm &g, int kd, double inv_alpha0, int32_t *err,
                              cudaStream_t st, bool intcvt)
{
    if (g.ntiles <= 0) return cudaSuccess;
    const int sms = g_sms > 0 ? g_sms : 152;
    const int grid = std::min(g.ntiles, g.max_ctas > 0 ? std::min(g.max_ctas, sms) : sms);
    int ie = 0;
    const int inv_alpha_exp = std::frexp(inv_alpha0, &ie) == 0.5 ? ie - 1 : kNoExp;
#define BC_GEMM(KD, S, IC)                                                                                       \
    launch_pdl(gemm_kernel<KD, S, IC>(), grid, kGemmThreads, gemm_smem<KD, S, IC>(), st, g, inv_alpha0,            \
               inv_alpha_exp, err, T.wait_limit, T.withhold_copy)
    if (T.slices == kWideSlices) {
        if (kd == 256) return BC_GEMM(256, kWideSlices, false);
        if (kd == 144) return BC_GEMM(144, kWideSlices, false);
        return BC_GEMM(64, kWideSlices, false);
    }
    if (kd == 256) return intcvt ? BC_GEMM(256, kSplitSlices, true) : BC_GEMM(256, kSplitSlices, false);
    return intcvt ? BC_GEMM(64, kSplitSlices, true) : BC_GEMM(64, kSplitSlices, false);
#undef BC_GEMM
}

}  // namespace bc
