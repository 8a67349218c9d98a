// FMM evaluation of the glue layer potential at every leaf node of a tree.
//
// The glue step of the solver (Sec. 3.4) patches the bulk and strip
// solutions together with v_glue = S[sigma] - D[tau] on the fictitious curve,
// a single-layer and a double-layer Laplace potential with Phi = (1/2pi)
// log(1/|x - y|); discretised on the curve's quadrature nodes y_j (weights
// w_j, unit normals n_j) with q_j = w_j sigma_j and m_j = w_j tau_j n_j:
//
//   u(x) = -(1/2pi) sum_j [ q_j log|x - y_j| + Re(m_j / (x - y_j)) ]
//
// (points as complex numbers; Re(m / (x - y)) = m.(x - y)/|x - y|^2).  The
// sources are point charges and dipoles; the far field runs through the same
// expansions, lists and level passes as the volume potential (multipoles in
// the scaled form of the leaf-to-expansion step, M2M, M2L, L2L), with these
// point-source steps around them:
//   P2M  (leaf box of centre c, half-side r, eta = (y - c)/r):
//        M_0 = sum c_q,  M_k = sum [ -c_q eta^k / k + (c_m / r) eta^(k-1) ]
//   P2L  (X list: source leaf c, target box b one level finer, e = (c_b - c_c)/r_c,
//        w = e - eta, the target's own coordinate rho = (x - c_b)/r_b):
//        L_0 = sum [ c_q log|w| + (c_m / r_c) / w ]     (c_q log r_c: downward pass)
//        L_l = sum (-1)^l (2w)^-l [ -c_q / l + (c_m / r_c) / w ]
//   M2P  (W list) and L2P as for the volume potential, near field direct;
// with c_q = -q / (2 pi), c_m = -m / (2 pi).  A source that coincides with a
// target node contributes nothing.  FP64 accuracy throughout: the near sums'
// logarithm and reciprocal in fixed point, the L2P on the volume apply's group-E
// tensor tiles over the same locals (7 digits in the FP64 mode, 5 in the split one).
// 17,584 leaves, 4,096 nodes, FP64: 1.86 -> 1.63 ms by the L2P; 0.74 with the near
// sums, level passes and P2M as they are now.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "bc_internal.h"

namespace bc {
namespace {

constexpr double kInvTwoPi = 0.159154943091895335768883763372514362;

__device__ __forceinline__ double2 cmul(double2 a, double2 b)
{
    return make_double2(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cinv(double2 a)
{
    const double d = 1.0 / fma(a.x, a.x, a.y * a.y);
    return make_double2(a.x * d, -a.y * d);
}
// ---------------------------------------------------------------------------
// log x and 1/x for the direct near sums: a table-driven logarithm after Tang (ACM
// TOMS 16, 1990) in fixed point.  An FP64 operation holds a sub-partition's FP64
// pipe for 64 cycles per warp, 30 of them per (node, source) pair bound the sums
// (13 for the logarithm, 8 for the reciprocal); integer and FP32 operations take 1 or
// 2 cycles, and ten FP64 operations per pair are left (17,584 leaves, 4,096 sources:
// leaf output 1160 -> 408 us).  With
// x = 2^e m, m in [1, 2), and j the top kLogBits bits of m's fraction, c_j is
// 1 / (1 + (j + 1/2) / 2^kLogBits) rounded to 11 bits, so that m c_j is an exact 64-bit
// integer and r = m c_j - 1 an exact multiple of 2^-63, |r| < 7.4e-4; then
//     log x = e ln 2 - log c_j + log1p(r),  log1p(r) = r - r^2/2 + r^3 (1/3 - r/4 + r^2/5),
//     1/x   = 2^-e c_j / (1 + r),           1/(1+r)  = 1 - r + r^2 + r^3 (-1 + r - r^2),
// the linear and square terms as 64-bit integers (r^2 to 2^-62), the cubic ones, below
// 4e-10, in FP32 (2e-17), the series cut below 2e-19.  Errors before the last rounding:
// logarithm 2^-53 absolute (also next to x = 1, where the rounding of x, a squared
// distance, alone makes as much; relative accuracy there, in FP64, made a layer of 40,000
// sources in 16 leaves 10% slower), reciprocal 2^-54 relative.  Valid for normal x with 1/x
// normal (|e| <= 1021), which the near sums' squared distances meet.  Table:
// g_logtab[j] = (c_j 2^11 - 1024) in 11 bits, -log c_j in units of 2^-53 in 53 bits (set by
// layer_log_init).
// ---------------------------------------------------------------------------
constexpr int kLogBits = 10, kLogN = 1 << kLogBits;
__device__ unsigned long long g_logtab[kLogN];

// m 2^ex, m > 0 and the result normal, rounded to nearest by integer operations.
__device__ __forceinline__ long long int_bits(unsigned long long m, int ex)
{
    const int lz = __clzll(static_cast<long long>(m));
    m <<= lz;   // leading one at bit 63: it adds one to the exponent field
    return (static_cast<long long>(63 - lz + ex + 1022) << 52) + static_cast<long long>(m >> 11) +
           static_cast<long long>((m >> 10) & 1);
}

__device__ __forceinline__ void log_inv(double x, const unsigned long long *__restrict__ tab, double &lg, double &inv)
{
    constexpr long long kLn2 = 6243314768165359ll;   // ln 2 in units of 2^-53, and the next 32 bits
    constexpr unsigned kLn2Lo = 897137782u;
    const long long bits = __double_as_longlong(x);
    const int e = int(bits >> 52) - 1023;   // x > 0
    const unsigned long long tw = tab[int(bits >> (52 - kLogBits)) & (kLogN - 1)];
    const unsigned c = 1024u + unsigned(tw >> 53);
    const unsigned long long m = (bits & 0x000FFFFFFFFFFFFFll) | 0x0010000000000000ll;
    const long long r = static_cast<long long>(m * c - (1ull << 63));   // units 2^-63
    // r^2 in units of 2^-82, from r = 2^22 rh + rl
    const int rh = int(r >> 22), rl = int(r) & 0x3FFFFF;
    const long long w = static_cast<long long>(rh) * rh + ((static_cast<long long>(rh) * rl) >> 21);
    // the cubic terms in units of 2^-61
    const float rf = float(rh) * 0x1p-41f, r3 = rf * rf * (rf * 0x1p61f);
    const int cl = __float2int_rn(r3 * fmaf(rf, fmaf(rf, 0.2f, -0.25f), 1.0f / 3.0f));
    const int ci = __float2int_rn(r3 * fmaf(rf, 1.0f - rf, -1.0f));
    const long long l1 = r - (w >> 20) + 4ll * cl;
    const long long l = static_cast<long long>(tw & ((1ull << 53) - 1)) + ((l1 + 512) >> 10) + e * kLn2 +
                        ((static_cast<long long>(e) * kLn2Lo) >> 32);
    const long long lb = int_bits(static_cast<unsigned long long>(l < 0 ? -l : l), -53);
    lg = l ? __longlong_as_double(lb | (l & (1ll << 63))) : 0.0;
    const unsigned long long s = (1ull << 63) - r + (w >> 19) + 4ll * ci;   // 1 / (1 + r), units 2^-63
    const unsigned cw = c << 20;
    inv = __longlong_as_double(int_bits((s >> 32) * cw + __umulhi(unsigned(s), cw), -62 - e));   // from units 2^-62
}

__global__ void k_log_inv_check(const double *__restrict__ x, int64_t n, double *__restrict__ lg,
                                double *__restrict__ inv)
{
    __shared__ unsigned long long tab[kLogN];
    for (int i = threadIdx.x; i < kLogN; i += blockDim.x) tab[i] = g_logtab[i];
    __syncthreads();
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        double a, b;
        log_inv(x[i], tab, a, b);
        lg[i] = a;
        inv[i] = b;
    }
}

struct BoxGeom {
    double cx, cy, r;
};
__device__ __forceinline__ BoxGeom box_geom(int b, const int32_t *box_level, const int32_t *box_ix,
                                            const int32_t *box_iy, double x0, double y0, double L)
{
    const double h = ldexp(L, -box_level[b]);
    return {x0 + (box_ix[b] + 0.5) * h, y0 + (box_iy[b] + 0.5) * h, 0.5 * h};
}

// the strengths in sorted order, scaled by -1/(2 pi)
__global__ void k_layer_gather(int64_t n, const int32_t *__restrict__ perm, const double *__restrict__ q,
                               const double *__restrict__ m, double *__restrict__ cq, double2 *__restrict__ cm)
{
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t j = perm[i];
        cq[i] = -kInvTwoPi * q[j];
        cm[i] = make_double2(-kInvTwoPi * m[2 * j], -kInvTwoPi * m[2 * j + 1]);
    }
}

// Sum over the warp of each of 32 coefficients, lane k ends with coefficient k: the
// lanes of each half hand the other half its coefficients, 62 additions in all (a
// butterfly of each coefficient takes 310).
__device__ __forceinline__ double2 warp_sums(double2 (&acc)[32], int lane)
{
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const bool up = lane & h;   // keeps the upper half
#pragma unroll
        for (int i = 0; i < h; i++) {
            const double2 keep = up ? acc[i + h] : acc[i], give = up ? acc[i] : acc[i + h];
            acc[i].x = keep.x + __shfl_xor_sync(0xffffffffu, give.x, h);
            acc[i].y = keep.y + __shfl_xor_sync(0xffffffffu, give.y, h);
        }
    }
    return acc[0];
}

// e^n, 0 <= n < 32, n per lane (repeated squaring).
__device__ __forceinline__ double2 cpow(double2 e, int n)
{
    double2 r = n & 1 ? e : make_double2(1.0, 0.0);
#pragma unroll
    for (int b = 1; b < 5; b++) {
        e = make_double2(fma(e.x, e.x, -e.y * e.y), (e.x + e.x) * e.y);
        if (n >> b & 1) r = cmul(r, e);
    }
    return r;
}

// P2M: a cluster of four blocks (16 warps on four SMs) per leaf with sources; the
// warps' partial sums meet in distributed shared memory.  A curve's sources crowd in a
// few leaves, whose chains of FP64 instructions, 64 cycles of a sub-partition's pipe
// each, set the time.
//   Up to kP2MFew sources: lane k is coefficient k, a warp takes every 16th source and
//   its lanes form their powers of eta by repeated squaring, about 50 FP64 instructions
//   per source (at most eight sources per warp).
//   More: lane s takes sources s, s + 512, ..., carries the power up the coefficients,
//   about 310 instructions per source of a lane, then 62 for the sums.
// 4,096 sources in 17,584 leaves: one warp per leaf, the second form alone with 680
// instructions, 62 us; kP2MFew = 16: 51, 128: 32 to 36.
constexpr int kP2MFew = 128, kLayerCluster = 4;

// The sums of the cluster's 16 warps (part: this block's four) to out[0..P1); sum
// alternates between two buffers from call to call.
__device__ __forceinline__ void cluster_sum_store(const double2 (&part)[4][32], double2 *sum, int P1,
                                                  double2 *__restrict__ out)
{
    auto cluster = cooperative_groups::this_cluster();
    __syncthreads();
    const int k = threadIdx.x;
    if (k < P1)
        sum[k] = make_double2((part[0][k].x + part[1][k].x) + (part[2][k].x + part[3][k].x),
                              (part[0][k].y + part[1][k].y) + (part[2][k].y + part[3][k].y));
    cluster.sync();
    if (cluster.block_rank() == 0 && k < P1) {
        const double2 a = sum[k], b = cluster.map_shared_rank(sum, 1)[k], c = cluster.map_shared_rank(sum, 2)[k],
                      d = cluster.map_shared_rank(sum, 3)[k];
        out[k] = make_double2((a.x + b.x) + (c.x + d.x), (a.y + b.y) + (c.y + d.y));
    }
}

// P2M.  Every leaf box is written (zero without sources: the climb reads all
// children).  P1 <= 32.
__global__ void __cluster_dims__(kLayerCluster, 1, 1) __launch_bounds__(128)
k_layer_p2m(int64_t nleaf, const int32_t *__restrict__ src_ptr, const double2 *__restrict__ sxy,
            const double *__restrict__ cq, const double2 *__restrict__ cm, const int32_t *__restrict__ leaf_box,
            const int32_t *__restrict__ box_level, const int32_t *__restrict__ box_ix,
            const int32_t *__restrict__ box_iy, double x0, double y0, double L, int P1, double2 *__restrict__ ex)
{
    __shared__ double2 part[4][32], sum[2][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int rank = blockIdx.x % kLayerCluster, cid = blockIdx.x / kLayerCluster, ncl = gridDim.x / kLayerCluster;
    int par = 0;
    const double ik = lane ? -1.0 / double(lane) : 0.0;
    for (int64_t base = cid; base < nleaf; base += 32 * int64_t(ncl)) {   // 32 leaves at a time
        const int64_t cand = base + lane * int64_t(ncl);
        const bool in = cand < nleaf;
        const int cb = in ? leaf_box[cand] : 0, cj0 = in ? src_ptr[cand] : 0, cj1 = in ? src_ptr[cand + 1] : 0;
        const unsigned some = __ballot_sync(0xffffffffu, cj1 > cj0), any = __ballot_sync(0xffffffffu, in);
        // most leaves: no source, no sums to form
        for (int q = rank * 4 + w; q < 32; q += 4 * kLayerCluster)
            if ((any & ~some) >> q & 1) {
                const int64_t b = __shfl_sync(0xffffffffu, cb, q);
                if (lane < P1) ex[b * P1 + lane] = make_double2(0.0, 0.0);
            }
        for (unsigned todo = some; todo; todo &= todo - 1) {   // uniform over the cluster
        const int q = __ffs(todo) - 1;
        const int b = __shfl_sync(0xffffffffu, cb, q), j0 = __shfl_sync(0xffffffffu, cj0, q),
                  j1 = __shfl_sync(0xffffffffu, cj1, q);
        const BoxGeom g = box_geom(b, box_level, box_ix, box_iy, x0, y0, L);
        const double ir = 1.0 / g.r;
        if (j1 - j0 <= kP2MFew) {
            double2 acc = make_double2(0.0, 0.0);
            for (int j = j0 + 4 * rank + w; j < j1; j += 4 * kLayerCluster) {
                const double2 y = sxy[j];
                const double2 eta = make_double2((y.x - g.cx) * ir, (y.y - g.cy) * ir);
                const double c = cq[j], ck = c * ik;
                // (c_m / r - (c_q / k) eta) eta^(k-1)
                const double2 t = make_double2(fma(ck, eta.x, cm[j].x * ir), fma(ck, eta.y, cm[j].y * ir));
                const double2 pw = cpow(eta, lane ? lane - 1 : 0);
                if (lane == 0) {
                    acc.x += c;
                } else {
                    acc.x = fma(pw.x, t.x, fma(-pw.y, t.y, acc.x));
                    acc.y = fma(pw.x, t.y, fma(pw.y, t.x, acc.y));
                }
            }
            part[w][lane] = acc;
        } else {
            double2 acc[32];
#pragma unroll
            for (int k = 0; k < 32; k++) acc[k] = make_double2(0.0, 0.0);
            for (int j = j0 + 128 * rank + int(threadIdx.x); j < j1; j += 128 * kLayerCluster) {
                const double2 y = sxy[j];
                const double2 eta = make_double2((y.x - g.cx) * ir, (y.y - g.cy) * ir);
                const double c = cq[j];
                const double2 cmr = make_double2(cm[j].x * ir, cm[j].y * ir);   // c_m / r
                acc[0].x += c;
                double2 pw = make_double2(1.0, 0.0);   // eta^(k-1)
#pragma unroll
                for (int k = 1; k < 32; k++) {
                    if (k < P1) {
                        const double ck = c * (-1.0 / double(k));
                        const double2 t = make_double2(fma(ck, eta.x, cmr.x), fma(ck, eta.y, cmr.y));
                        acc[k].x = fma(pw.x, t.x, fma(-pw.y, t.y, acc[k].x));
                        acc[k].y = fma(pw.x, t.y, fma(pw.y, t.x, acc[k].y));
                        pw = cmul(pw, eta);
                    }
                }
            }
            part[w][lane] = j0 + 128 * rank + 32 * w < j1 ? warp_sums(acc, lane) : acc[0];
        }
        cluster_sum_store(part, sum[par], P1, ex + int64_t(b) * P1);
        par ^= 1;
        }
    }
    cooperative_groups::this_cluster().sync();   // the last sums have been read
}

// P2L of the X list: one warp per entry, lane s the sources s, s + 32, ... of
// the source leaf; each lane carries t^l = (-1/(2w))^l up the coefficients,
// then the warp sums each coefficient.  P1 <= 32.  (Entries of 65 to 128 sources as
// a rule: four blocks per entry, as for P2M, repeat the log and the division and took
// 70 us instead of 43 for 288 entries; an FP64 butterfly of every coefficient made it 60.)
__global__ void __launch_bounds__(128)
k_layer_p2l(int64_t nx, const int32_t *__restrict__ x_box, const int32_t *__restrict__ x_src,
            const int32_t *__restrict__ src_ptr, const double2 *__restrict__ sxy, const double *__restrict__ cq,
            const double2 *__restrict__ cm, const int32_t *__restrict__ leaf_box,
            const int32_t *__restrict__ box_level, const int32_t *__restrict__ box_ix,
            const int32_t *__restrict__ box_iy, double x0, double y0, double L, int P1, double2 *__restrict__ PX)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = int64_t(gridDim.x) * (blockDim.x >> 5);
    for (int64_t x = blockIdx.x * int64_t(blockDim.x >> 5) + (threadIdx.x >> 5); x < nx; x += nw) {
        const int leaf = x_src[x];
        const BoxGeom gc = box_geom(leaf_box[leaf], box_level, box_ix, box_iy, x0, y0, L);
        const BoxGeom gb = box_geom(x_box[x], box_level, box_ix, box_iy, x0, y0, L);
        const double ir = 1.0 / gc.r;
        const double2 e = make_double2((gb.cx - gc.cx) * ir, (gb.cy - gc.cy) * ir);
        double2 acc[32];
#pragma unroll
        for (int l = 0; l < 32; l++) acc[l] = make_double2(0.0, 0.0);
        for (int j = src_ptr[leaf] + lane; j < src_ptr[leaf + 1]; j += 32) {
            const double2 y = sxy[j];
            const double2 w = make_double2(e.x - (y.x - gc.cx) * ir, e.y - (y.y - gc.cy) * ir);
            const double2 iw = cinv(w);
            const double2 dm = cmul(make_double2(cm[j].x * ir, cm[j].y * ir), iw);   // (c_m / r_c) / w
            const double c = cq[j];
            acc[0].x += fma(c, 0.5 * log(fma(w.x, w.x, w.y * w.y)), dm.x);
            acc[0].y += dm.y;
            const double2 t = make_double2(-0.5 * iw.x, -0.5 * iw.y);   // -1 / (2w)
            double2 pw = make_double2(1.0, 0.0);
#pragma unroll
            for (int l = 1; l < 32; l++) {
                if (l < P1) {
                    pw = cmul(pw, t);
                    const double vx = fma(c, -1.0 / double(l), dm.x);
                    acc[l].x = fma(pw.x, vx, fma(-pw.y, dm.y, acc[l].x));
                    acc[l].y = fma(pw.x, dm.y, fma(pw.y, vx, acc[l].y));
                }
            }
        }
        const double2 s = warp_sums(acc, lane);
        if (lane < P1) PX[x * P1 + lane] = s;
    }
}

// Leaf output: one block of NP threads per target leaf, thread j its node.
// u = L2P of the leaf's local expansion (levels >= 2; PE: its row from the
// tensor-core tiles, else in FP64 here) + the W list's
// multipoles at the nodes (M2P, with the log r term of the target level) +
// the direct sum over the sources of the leaf's near leaves.
constexpr int kSrcChunk = 128;
__global__ void __launch_bounds__(256)
k_layer_out(int64_t nleaf, const int32_t *__restrict__ order, const int32_t *__restrict__ leaf_box,
            const int32_t *__restrict__ box_level, const int32_t *__restrict__ box_ix,
            const int32_t *__restrict__ box_iy, double x0, double y0, double L, const int32_t *__restrict__ w_ptr,
            const int32_t *__restrict__ w_src, const int32_t *__restrict__ w_code,
            const int32_t *__restrict__ n_ptr, const int32_t *__restrict__ n_src,
            const int32_t *__restrict__ src_ptr, const double2 *__restrict__ sxy, const double *__restrict__ cq,
            const double2 *__restrict__ cm, const double2 *__restrict__ OpE, const double2 *__restrict__ OpW,
            const double2 *__restrict__ loc, const double2 *__restrict__ mul, const double *__restrict__ lvtab,
            int p, int P1, double *__restrict__ u, const double *__restrict__ PE)
{
    const int NP = p * p, j = threadIdx.x;
    __shared__ double2 se[32];
    __shared__ double2 s_xy[kSrcChunk], s_m[kSrcChunk];
    __shared__ double s_q[kSrcChunk];
    __shared__ unsigned long long s_log[kLogN];
    for (int i = j; i < kLogN; i += blockDim.x) s_log[i] = g_logtab[i];   // read after the first barrier below
    const double pi = 3.14159265358979323846;
    const double xj = -cos((2.0 * (j % p) + 1.0) * pi / (2.0 * p)), yj = -cos((2.0 * (j / p) + 1.0) * pi / (2.0 * p));
    for (int64_t li = blockIdx.x; li < nleaf; li += gridDim.x) {
        const int o = order[li];
        const int b = leaf_box[o];
        const int lvo = box_level[b];
        const BoxGeom g = box_geom(b, box_level, box_ix, box_iy, x0, y0, L);
        const double zx = g.cx + g.r * xj, zy = g.cy + g.r * yj;
        double acc = 0.0;
        if (lvo >= 2 && PE) {
            acc = PE[int64_t(o) * NP + j];   // the L2P from the tensor cores
        } else if (lvo >= 2) {
            __syncthreads();
            for (int i = j; i < P1; i += blockDim.x) se[i] = loc[int64_t(b) * P1 + i];
            __syncthreads();
            double a1 = 0.0;
            int l = 0;
            for (; l + 1 < P1; l += 2) {
                const double2 op0 = OpE[l * NP + j], c0 = se[l], op1 = OpE[(l + 1) * NP + j], c1 = se[l + 1];
                acc = fma(op0.x, c0.x, fma(-op0.y, c0.y, acc));
                a1 = fma(op1.x, c1.x, fma(-op1.y, c1.y, a1));
            }
            if (l < P1) {
                const double2 op = OpE[l * NP + j], c = se[l];
                acc = fma(op.x, c.x, fma(-op.y, c.y, acc));
            }
            acc += a1;
        }
        double lw = 0.0;
        for (int e = w_ptr[o]; e < w_ptr[o + 1]; e++) {
            const double2 *op = OpW + size_t(w_code[e]) * P1 * NP;
            __syncthreads();
            for (int i = j; i < P1; i += blockDim.x) se[i] = mul[int64_t(w_src[e]) * P1 + i];
            __syncthreads();
            for (int k = 0; k < P1; k++) {
                const double2 opk = op[k * NP + j], c = se[k];
                acc = fma(opk.x, c.x, fma(-opk.y, c.y, acc));
            }
            lw += se[0].x;
        }
        acc = fma(lvtab[kLvTab + lvo], lw, acc);
        // near field, sources staged in chunks
        double near = 0.0;
        for (int e = n_ptr[o]; e < n_ptr[o + 1]; e++) {
            const int s = n_src[e];
            for (int c0 = src_ptr[s]; c0 < src_ptr[s + 1]; c0 += kSrcChunk) {
                const int cnt = min(kSrcChunk, src_ptr[s + 1] - c0);
                __syncthreads();
                for (int i = j; i < cnt; i += blockDim.x) {
                    s_xy[i] = sxy[c0 + i];
                    s_q[i] = 0.5 * cq[c0 + i];   // c_q log|x - y| = (c_q / 2) log r^2
                    s_m[i] = cm[c0 + i];
                }
                __syncthreads();
                for (int i = 0; i < cnt; i++) {
                    const double dx = zx - s_xy[i].x, dy = zy - s_xy[i].y;
                    const double r2 = fma(dx, dx, dy * dy);
                    // r2 > 0, as integers (no sign bit; NaN is left out, as by the comparison)
                    if (static_cast<unsigned long long>(__double_as_longlong(r2)) - 1 < 0x7FF0000000000000ull) {
                        double lg, ir2;
                        log_inv(r2, s_log, lg, ir2);
                        near = fma(s_q[i], lg, near);
                        near = fma(fma(s_m[i].x, dx, s_m[i].y * dy), ir2, near);
                    }
                }
            }
        }
        u[int64_t(o) * NP + j] = acc + near;
    }
}

inline int grid_cap(int64_t n, int cap) { return int(n < cap ? (n > 0 ? n : 1) : cap); }

}  // namespace

cudaError_t layer_log_init()
{
    // c_j to 11 bits, -log c_j from the host's extended-precision logarithm (once per
    // process: half a millisecond where that is done in software)
    struct Table {
        unsigned long long t[kLogN];
        Table()
        {
            for (int j = 0; j < kLogN; j++) {
                const double c = std::nearbyint(2048.0 / (1.0 + (j + 0.5) / kLogN));
                const long double l = -logl(static_cast<long double>(c) / 2048.0L);
                t[j] = static_cast<unsigned long long>(c - 1024.0) << 53 |
                       static_cast<unsigned long long>(l * 9007199254740992.0L + 0.5L);
            }
        }
    };
    static const Table tab;
    return cudaMemcpyToSymbol(g_logtab, tab.t, sizeof tab.t);
}

cudaError_t launch_log_inv_check(const double *x, int64_t n, double *lg, double *inv, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    const int grid = int(std::min<int64_t>((n + 255) / 256, 152 * 8));
    k_log_inv_check<<<grid, 256, 0, st>>>(x, n, lg, inv);
    return cudaGetLastError();
}

cudaError_t launch_layer(const PassArgs &a, const HostTree &h, const DevTree &d, const DevTables &tb,
                         const LayerDev &ly, const double *q, const double *m, double *u, cudaStream_t st,
                         const SplitLaunch *split)
{
    cudaError_t e;
    const int P1 = a.P1;
    if (ly.n > 0) {
        k_layer_gather<<<grid_cap((ly.n + 255) / 256, 152 * 8), 256, 0, st>>>(ly.n, ly.perm, q, m, ly.cq, ly.cm);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    k_layer_p2m<<<kLayerCluster * grid_cap(a.nleaf, 152 * 4), 128, 0, st>>>(
        a.nleaf, ly.src_ptr, ly.sxy, ly.cq, ly.cm, d.leaf_box, d.box_level, d.box_ix, d.box_iy, h.x0, h.y0, h.L, P1,
        d.expA);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (ly.nx > 0) {
        k_layer_p2l<<<grid_cap((ly.nx + 3) / 4, 152 * 8), 128, 0, st>>>(
            ly.nx, ly.x_box, ly.x_src, ly.src_ptr, ly.sxy, ly.cq, ly.cm, d.leaf_box, d.box_level, d.box_ix, d.box_iy,
            h.x0, h.y0, h.L, P1, ly.PX);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    FarLists fl;
    fl.v_ptr = ly.v_ptr; fl.v_src = ly.v_src; fl.v_code = ly.v_code;
    fl.x_ptr = ly.x_ptr; fl.x_src = ly.x_src; fl.PX = ly.PX;
    fl.live = ly.live;
    if ((e = launch_far_points(a, h, d, tb, fl, st)) != cudaSuccess) return e;
    const double *PE = nullptr;
    if (split) {
        // L2P of every leaf at level >= 2 on the tensor cores: digits of the
        // locals (expB, the forward apply's second array), then the forward
        // group-E tiles that evaluate them at the leaf nodes, into PE
        const SplitTables *sT = split->tables;
        const SplitTree *sp = split->tree;
        const int64_t nbox = a.nbox;
        e = launch_split_digits_exp(*sT, 0, nbox, 2 * nbox, nbox, d.expA, d.expB, P1, 1.0, sp->edig, sp->eexp, st);
        if (e != cudaSuccess) return e;
        e = launch_split_gemm(*sT, gemm_group_e(*sT, *sp, 0, sp->tE, sp->cE[0], sp->ntL, d.expA, d.expB, nbox, P1,
                                                1.0),
                              kSplitKE, 1.0 / (a.half_L * a.half_L), sp->err, st);
        if (e != cudaSuccess) return e;
        PE = sp->PE;
    }
    k_layer_out<<<grid_cap(a.nleaf, 152 * 8), a.NP, 0, st>>>(
        a.nleaf, ly.order, d.leaf_box, d.box_level, d.box_ix, d.box_iy, h.x0, h.y0, h.L, ly.w_ptr, ly.w_src,
        ly.w_code, ly.n_ptr, ly.n_src, ly.src_ptr, ly.sxy, ly.cq, ly.cm, tb.fwd.e, tb.fwd.w, d.expB, d.expA, d.lvtab,
        a.p, P1, u, PE);
    return cudaGetLastError();
}

}  // namespace bc
