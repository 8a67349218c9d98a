// Strip solve (Sec. 3.3), blocks above 32 x 32 (the paper's elements of 16 x 24
// = 384 nodes): one system on the whole GPU in one cooperative launch.  The
// elimination is that of kernels_strip.cu (block LU, the corners as a border):
//
//   D_k = A_k - C_k H_{k-1},  [H_k | G_k] = D_k^-1 [B_k | (b_k | E_k) - C_k G_{k-1}],   k < N - 1,
//   X_k = G_k - H_k X_{k+1},  then the border system S x_{N-1} = s and x_k = Y_k - Z_k x_{N-1}.
//
// The chain over the elements, and inside each the chain over its panels of 16
// columns, bounds the solve: the FP64 work of the paper's strip (34 GFLOP) takes
// 27 ms of the whole GPU's FP64 pipes, but a 16-column panel of 384 rows 17 us of
// one SM's.  So one CTA (the panel CTA) does nothing but factor panels, one
// inverts their upper diagonal blocks, and the others (workers) own columns: column c of D_k and of B_k (then H_k) belongs to
// worker c mod NW, the right-hand columns are dealt the other way round.  A
// worker keeps its columns in shared memory from element to element, and every
// step is local to a column: the products C_k H, the panels' row exchanges and
// updates, the back substitution.  What CTAs exchange goes through L2 with
// counters: a worker delivers a column to the panel's store F when all earlier
// panels have been applied to it; the panel CTA publishes each factored panel.
// While the next panel is not there, a worker goes on with its background: the
// products C_k G and the panels' updates of B_k and the right-hand columns, which
// may lag (F keeps all panels of an element).  F is doubled by the parity of
// the element.
// Every wait is bounded by progress: it gives up after kPollLimit polls during which
// no worker finished an element of the backward sweep (the only phase that a wait
// spans whole, and one as long as the strip).  A wait that runs out raises the abort
// word, at which all CTAs leave, the workers with NaN in the solution; the status
// word then says 2.
// The paper's strip (N = 56, m = 384, r = 1): 216 ms as some 8,000 launches (panel,
// exchange, triangular solve and DGEMM kernels, recorded again for new arguments;
// 170 ms replayed), 55 ms so: per element 0.87 ms, of which the 24 panels take 19 us
// each on average and 5 us more from one's publication to the next one's columns,
// the back substitution 0.15 ms, the products for D 0.08 ms; the backward sweep
// 0.11 ms per element.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "bc_internal.h"

namespace bc {
namespace {

constexpr int kW = 16;         // panel width
constexpr int kMaxM = 448;
// columns of a kind per worker: three and four for m = 448, r = 32 on 150 workers,
// four of each from 120 workers on
constexpr int kMaxD = 4, kMaxR = 4;
constexpr int kPollLimit = 1 << 22;   // polls of several hundred cycles: a second or two

// counters in the workspace (zeroed before the launch), 64 bytes apart
// (kCtrDone: one per parity of the element; kCtrBeat: elements that the workers have
// finished in the backward sweep)
enum { kCtrPanel = 0, kCtrCols = 16, kCtrInv = 32, kCtrDone = 48, kCtrGrid = 80, kCtrAbort = 96, kCtrBeat = 112, kCtrWords = 128 };

struct LargeArgs {
    int64_t N;
    int m, r, R, np, nw;       // R = r + m; panels; workers
    const double *A, *B, *C, *b;
    double *x;
    double *H, *G;             // [N-1][m columns][m rows], [N-1][R columns][m rows]
    double *F;                 // [2][m columns][m rows]: L below, U on and above the diagonal
    double *Linv, *Uinv;       // [2][np][16][16] inverses of the panels' diagonal blocks
    int32_t *perm;             // [2][np][m] row (within the panel's rows) that ends at each position
    uint32_t *ctr;
    int32_t *status;
    int polls;                 // polls of a wait without progress
    int withhold;              // diagnostics: the panel CTA factors nothing (the first wait for a panel runs out)
    int stall_ns;              // diagnostics: workers without a matrix column wait so long before each background panel
};

__device__ __forceinline__ uint32_t ctr_load(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void ctr_add(uint32_t *p, uint32_t n)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(n) : "memory");
}

// Whether a wait goes on after its poll `it` (reset where the backward sweep has moved).
__device__ __forceinline__ bool keep_waiting(const LargeArgs &a, int &it, uint32_t &beat)
{
    if (++it >= a.polls) {
        const uint32_t b = ctr_load(a.ctr + kCtrBeat);
        if (b == beat) return false;
        beat = b;
        it = 0;
    }
    return (it & 63) != 63 || !ctr_load(a.ctr + kCtrAbort);
}

// Thread 0 waits until *p >= want; all threads of the CTA get the outcome.
__device__ bool cta_wait(const LargeArgs &a, int word, uint32_t want, int *s_ok)
{
    if (threadIdx.x == 0) {
        int ok = 0, it = 0;
        uint32_t beat = ctr_load(a.ctr + kCtrBeat);
        do ok = ctr_load(a.ctr + word) >= want;
        while (!ok && keep_waiting(a, it, beat));
        if (!ok) atomicExch(a.ctr + kCtrAbort, 1u);
        *s_ok = ok;
    }
    __syncthreads();
    const bool ok = *s_ok != 0;
    __syncthreads();
    return ok;
}

// The CTA's global writes so far, then n more on the counter.
__device__ __forceinline__ void cta_signal(const LargeArgs &a, int word, uint32_t n)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        ctr_add(a.ctr + word, n);
    }
}

__device__ bool grid_barrier(const LargeArgs &a, uint32_t &phase, int *s_ok)
{
    cta_signal(a, kCtrGrid, 1);
    phase++;
    return cta_wait(a, kCtrGrid, phase * uint32_t(a.nw + 2), s_ok);
}

// ---------------------------------------------------------------------------
// The panel CTA.  Thread t of the row warps owns row t of the panel's rows [16p,
// m) in registers; rows are never moved, each thread carries its row's position
// (pivoting exchanges positions).  Per column: each thread updates its next
// column, every warp finds its candidate (redux on the magnitude's two words,
// lowest position on a tie) and leaves its key; after a barrier all know the
// pivot, whose thread takes the reciprocal while all finish their rows, and
// passes its row through shared memory.  One warp forms the inverse of the unit
// lower diagonal block on the side, a row per column.  What counts is the number
// of FP64 instructions of any width: each holds a sub-partition's pipe for 64 to
// 76 cycles, dependent or not (384 rows: 12 warps x 152, 17 us per panel).
// ---------------------------------------------------------------------------
struct PanelShared {
    double row[2][kW + 2];     // the pivot row from the pivot's column on; [16]: its reciprocal pivot
    uint32_t hi[2][16];
    int pos[2][16];
    int who[2];                // the pivot row's thread
    double li[kW][kW + 1];     // the unit lower inverse
};

// 1/d by one cubic (Halley) step from an FP32 reciprocal of the leading 24 bits:
// three FP64 instructions; within an ulp or so.  Zero and non-finite d give 0
// (such a pivot is flagged and eliminates nothing); the ends of the exponent
// range take the division.
__device__ __forceinline__ double pivot_reciprocal(double d)
{
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(d));
    const int e = int((bits >> 52) & 0x7FF);
    if (e < 2 || e > 2040) return d != 0.0 && isfinite(d) ? 1.0 / d : 0.0;
    const double m = __longlong_as_double(static_cast<long long>((bits & 0x000FFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
    const float r = __frcp_rn(__uint_as_float(0x3F800000u | unsigned((bits >> 29) & 0x7FFFFFu)));   // in (1/2, 1]
    const unsigned rb = __float_as_uint(r);
    const double x0 = __longlong_as_double((static_cast<long long>(rb & 0x7FFFFFu) << 29) |
                                           (static_cast<long long>(int(rb >> 23) - 127 + 1023) << 52));
    const double t = fma(-m, x0, 1.0);
    const double x = fma(x0, fma(t, t, t), x0);   // 1/m
    const long long xb = __double_as_longlong(x) + (static_cast<long long>(1023 - e) << 52);
    return __longlong_as_double(xb | static_cast<long long>(bits & 0x8000000000000000ull));
}

// warps that hold rows; the warp of the lower inverse sits on sub-partition 3, the
// last one that the row warps (0, 1, 2, ...) fill
__host__ __device__ __forceinline__ int row_warps(int m) { return (m + 31) / 32; }
__host__ __device__ __forceinline__ int inverse_warp(int m) { return row_warps(m) | 3; }

// Ls: [16][m] shared, the multipliers by thread.  After each column a row's
// registers move up by one.
template <bool FULL>   // a panel of 16 columns (the loop unrolled)
__device__ __forceinline__ void panel_factor(const LargeArgs &a, double *F, double *Linv, int32_t *perm, int p, PanelShared &S, double *Ls,
                             int *bad)
{
    const int m = a.m, j0 = p * kW, rows = m - j0, jb = FULL ? kW : min(kW, rows);
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, nrw = row_warps(m);
    const bool in = w < nrw && t < rows, inverse = w == inverse_warp(m);
    double v[kW];   // columns j, j + 1, ... of the row
#pragma unroll
    for (int j = 0; j < kW; j++) v[j] = in && j < jb ? __ldcg(&F[size_t(j0 + j) * m + j0 + t]) : 0.0;
    int pos = in ? t : 1 << 20;
    // The largest magnitude by its upper 32 bits (sign cleared), the lowest position
    // among equals: the pivot is within 2^-20 of the largest entry.  (All upper words
    // zero: by the lower ones.)  A NaN sorts above every number.
    // Candidates of column j into slot j & 1:
    auto candidate = [&](int j, double x) {
        const bool act = in && pos >= j;
        const unsigned hi = act ? unsigned(__double2hiint(x)) & 0x7FFFFFFFu : 0u;
        unsigned mh = __reduce_max_sync(0xffffffffu, hi), key = hi;
        if (mh == 0u) {   // zeros and subnormal numbers (uniform)
            key = act ? unsigned(__double2loint(x)) >> 12 : 0u;   // below every other upper word
            mh = __reduce_max_sync(0xffffffffu, key);
        }
        const unsigned mp = __reduce_min_sync(0xffffffffu, act && key == mh ? unsigned(pos) : 0xffffffffu);
        if (lane == 0) {
            S.hi[j & 1][w] = mh;
            S.pos[j & 1][w] = int(mp);   // -1: no active row
        }
    };
    // the pivot of column j over the warps' candidates (its position)
    auto pivot = [&](int j) -> int {
        const int q = lane < nrw ? lane : 0, cp = S.pos[j & 1][q];
        const unsigned hi = S.hi[j & 1][q];
        const bool cw = lane < nrw && cp >= 0;
        const unsigned mh = __reduce_max_sync(0xffffffffu, cw ? hi : 0u);
        return int(__reduce_min_sync(0xffffffffu, cw && hi == mh ? unsigned(cp) : 0xffffffffu));
    };
    auto publish = [&](double *row, const double *from, double inv, int j) {
#pragma unroll
        for (int c = 0; c < kW; c += 2) *reinterpret_cast<double2 *>(row + c) = make_double2(from[c], c + 1 < kW ? from[c + 1] : 0.0);
        row[kW] = inv;
        S.who[j & 1] = t;
        if (!(from[0] != 0.0 && isfinite(from[0]))) *bad = 1;
    };
    if (w < nrw) candidate(0, v[0]);
    __syncthreads();
    int P = pivot(0);
    if (in && pos == P) publish(S.row[0], v, pivot_reciprocal(v[0]), 0);
    __syncthreads();
#pragma unroll(FULL ? kW : 1)
    for (int j = 0; j < jb; j++) {
        const double *row = S.row[j & 1];
        const int left = jb - j;   // columns from j on
        if (in) {   // exchange of positions j and P
            if (pos == P) pos = j;
            else if (pos == j) pos = P;
        }
        const bool below = in && pos > j;
        double l = 0.0;
        if (below) {
            l = v[0] * row[kW];
            Ls[j * m + t] = l;
            if (left > 1) v[1] = fma(-l, row[1], v[1]);
        }
        if (w < nrw && left > 1) candidate(j + 1, v[1]);
        __syncthreads();   // keys of column j + 1
        if (left > 1) P = pivot(j + 1);
        const bool next = in && left > 1 && pos == P;
        double inv = 0.0;
        if (next) inv = pivot_reciprocal(v[1]);
        if (below) {
#pragma unroll
            for (int c = 2; c < kW; c++)
                if (c < left) v[c] = fma(-l, row[c], v[c]);
        }
#pragma unroll
        for (int c = 0; c + 1 < kW; c++) v[c] = v[c + 1];
        if (next) publish(S.row[(j + 1) & 1], v, inv, j + 1);   // the next pivot's thread
        if (inverse) {
            if (lane < left) F[size_t(j0 + j + lane) * m + j0 + j] = row[lane];   // row j of U
            // row j of the unit lower inverse, e_j - sum_{i<j} l_ji (row i):
            // even terms on the first half of the warp, odd ones on the second
            const int h = lane >> 4, c = lane & 15, who = S.who[j & 1];
            double s = h == 0 && c == j ? 1.0 : 0.0;
            for (int i = h; i < j; i += 2) s = fma(-Ls[i * m + who], S.li[i][c], s);
            s += __shfl_xor_sync(0xffffffffu, s, 16);
            if (h == 0) S.li[j][c] = s;
        }
        __syncthreads();   // the next pivot row in place, this one read
    }
    if (in) {
        for (int j = 0; j < min(pos, jb); j++) F[size_t(j0 + j) * m + j0 + pos] = Ls[j * m + t];
        perm[pos] = t;
    }
    if (inverse)
        for (int q = lane; q < kW * kW; q += 32) Linv[q] = q / kW < jb ? S.li[q / kW][q % kW] : 0.0;
}

__device__ void panel_cta(const LargeArgs &a, double *Ls)
{
    __shared__ PanelShared S;
    __shared__ int s_ok, s_bad;
    if (threadIdx.x == 0) s_bad = 0;
    __syncthreads();
    uint32_t phase = 0;
    const int64_t Nt = a.N - 1;
    bool ok = true;
    for (int64_t e = 0; e <= Nt && ok; e++) {
        if (e == Nt && Nt > 0) ok = grid_barrier(a, phase, &s_ok) && grid_barrier(a, phase, &s_ok);
        const int par = int(e & 1);
        double *F = a.F + size_t(par) * a.m * a.m, *Li = a.Linv + size_t(par) * a.np * kW * kW;
        int32_t *pm = a.perm + size_t(par) * a.np * a.m;
        for (int p = 0; p < a.np && ok; p++) {
            ok = cta_wait(a, kCtrCols, uint32_t(e * a.m + min(a.m, (p + 1) * kW)), &s_ok);
            if (!ok) break;
            if (a.withhold) continue;   // diagnostics: the waits for this panel run out
            if ((p + 1) * kW <= a.m) panel_factor<true>(a, F, Li + p * kW * kW, pm + size_t(p) * a.m, p, S, Ls, &s_bad);
            else panel_factor<false>(a, F, Li + p * kW * kW, pm + size_t(p) * a.m, p, S, Ls, &s_bad);
            cta_signal(a, kCtrPanel, 1);
        }
    }
    if (ok) ok = grid_barrier(a, phase, &s_ok);
    if (threadIdx.x == 0) *a.status = !ok || ctr_load(a.ctr + kCtrAbort) ? 2 : s_bad ? 1 : 0;
}

// The helper CTA: the inverse of each published panel's upper diagonal block
// (for the back substitution), off the panel CTA's FP64 pipe.  Lane c of its
// first warp has column c, from the last row up.
__device__ void helper_cta(const LargeArgs &a)
{
    __shared__ double U[kW][kW + 1];
    __shared__ int s_ok;
    const int lane = threadIdx.x & 31, m = a.m;
    uint32_t phase = 0;
    const int64_t Nt = a.N - 1;
    bool ok = true;
    for (int64_t e = 0; e <= Nt && ok; e++) {
        if (e == Nt && Nt > 0) ok = grid_barrier(a, phase, &s_ok) && grid_barrier(a, phase, &s_ok);
        const double *F = a.F + size_t(e & 1) * m * m;
        for (int p = 0; p < a.np && ok; p++) {
            ok = cta_wait(a, kCtrPanel, uint32_t(e * a.np + p + 1), &s_ok);
            if (!ok) break;
            const int j0 = p * kW, jb = min(kW, m - j0);
            for (int q = threadIdx.x; q < kW * kW; q += blockDim.x) {
                const int c = q / kW, i = q % kW;
                U[i][c] = i < jb && c < jb ? __ldcg(&F[size_t(j0 + c) * m + j0 + i]) : 0.0;
            }
            __syncthreads();
            double *Uinv = a.Uinv + (size_t(e & 1) * a.np + p) * kW * kW;
            if (threadIdx.x < 32) {
                double x[kW];
#pragma unroll
                for (int i = kW - 1; i >= 0; i--) {
                    double s = lane == i ? 1.0 : 0.0;
#pragma unroll
                    for (int q = i + 1; q < kW; q++) s = fma(-U[i][q], x[q], s);
                    const double d = U[i][i];   // zero past a short panel's columns
                    x[i] = d != 0.0 && isfinite(d) ? s / d : 0.0;
                    if (lane < kW) Uinv[i * kW + lane] = x[i];
                }
            }
            cta_signal(a, kCtrInv, 1);
            __syncthreads();
        }
    }
    if (ok) grid_barrier(a, phase, &s_ok);
}

// ---------------------------------------------------------------------------
// Workers.  Thread t is row t of every column (the warps past row m - 1 only help
// with copies).  Columns lie one after another in shared memory, m entries each:
//   D [nD] | R0 [nR] | H [nD] | R1 [nR]
// (R0 and R1 take turns as this element's right-hand columns and the previous
// one's; H, B until it is solved for, is next to both, so that the background's
// columns are always one range.)  Functions are compiled for the exact number of
// columns.
// ---------------------------------------------------------------------------
struct WorkShared {
    double inv[kW * kW];
    double a[kMaxD + kMaxR][kW], u[kW][kMaxD + kMaxR];
    int ok;
    uint32_t seen;
};

template <class F>
__device__ __forceinline__ void with_count(int n, F &&f)   // f of an integral constant
{
    static_assert(kMaxD + kMaxR == 8, "cases below");
    switch (n) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    default: break;
    }
}

// Sixteen entries of row t of the row-major block M from column c0 (zero past
// the last).  A thread reads whole 128-byte lines of its row, so the block goes
// through L1 once, without staging and barriers.
__device__ __forceinline__ void load_row16(double (&v)[kW], const double *M, int m, int t, int c0)
{
    const double *row = M + size_t(t) * m + c0;
    if (t < m && c0 + kW <= m) {
        if (((reinterpret_cast<uintptr_t>(row) | (m & 1 ? 8 : 0)) & 15) == 0) {
#pragma unroll
            for (int j = 0; j < kW; j += 2) {
                const double2 x = *reinterpret_cast<const double2 *>(row + j);
                v[j] = x.x;
                v[j + 1] = x.y;
            }
        } else {
#pragma unroll
            for (int j = 0; j < kW; j++) v[j] = row[j];
        }
    } else {
#pragma unroll
        for (int j = 0; j < kW; j++) v[j] = t < m && c0 + j < m ? row[j] : 0.0;
    }
}

// acc[c] += v . in[c][c0 ..], columns in[c] at in + c m; sums are formed from zero
// and taken off once: a chain that starts from a column's value would round at
// the magnitude of a diagonal entry each time
template <int NC>
__device__ __forceinline__ void dot16(double (&acc)[NC], const double (&v)[kW], const double *in, int m, int c0)
{
    const int w = min(kW, m - c0);
#pragma unroll
    for (int j = 0; j < kW; j++)
        if (j < w) {
#pragma unroll
            for (int c = 0; c < NC; c++) acc[c] = fma(v[j], in[c * m + c0 + j], acc[c]);
        }
}

// out[c] -= M in[c], c < NC, for a row-major block M (each thread its row)
template <int NC>
__device__ void block_product(double *out, const double *in, const double *M, int m)
{
    const int t = threadIdx.x;
    double acc[NC], v[kW], vn[kW];
#pragma unroll
    for (int c = 0; c < NC; c++) acc[c] = 0.0;
    load_row16(v, M, m, t, 0);
    for (int c0 = 0; c0 < m; c0 += kW) {
        load_row16(vn, M, c0 + kW < m ? m : 0, t, c0 + kW);
        if (t < m) dot16<NC>(acc, v, in, m, c0);
#pragma unroll
        for (int j = 0; j < kW; j++) v[j] = vn[j];
    }
    if (t < m) {
#pragma unroll
        for (int c = 0; c < NC; c++) out[c * m + t] -= acc[c];
    }
}

// S.u[j][c] = sum_k inv[j][k] S.a[c][k], the triangular solve with a panel's
// diagonal block by its inverse (whose other triangle is zero), one warp per
// column: lanes 0-15 the even terms of row j = lane, lanes 16-31 the odd ones
__device__ __forceinline__ void diag_product(WorkShared &S, int nc, int jb)
{
    const int lane = threadIdx.x & 31, j = lane & 15, h = lane >> 4;
    for (int c = threadIdx.x >> 5; c < nc; c += blockDim.x >> 5) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < kW; k += 2)
            if (k + h < jb) s = fma(S.inv[j * kW + k + h], S.a[c][k + h], s);
        s += __shfl_xor_sync(0xffffffffu, s, 16);
        if (h == 0) S.u[j][c] = s;
    }
}

// sum_j l[j] u[j][c]
template <int NC>
__device__ __forceinline__ void row_sums(double (&acc)[NC], const double (&l)[kW], const WorkShared &S)
{
#pragma unroll
    for (int c = 0; c < NC; c++) acc[c] = 0.0;
#pragma unroll
    for (int j = 0; j < kW; j++)
#pragma unroll
        for (int c = 0; c < NC; c++) acc[c] = fma(l[j], S.u[j][c], acc[c]);
}

// panel p applied to NC columns at col: rows permuted, u = Linv a on the panel's
// rows, rows below minus L u
template <int NC>
__device__ void apply_panel(const LargeArgs &a, const double *F, const double *Linv, const int32_t *perm, int p, double *col,
                            WorkShared &S)
{
    const int m = a.m, j0 = p * kW, rows = m - j0, jb = min(kW, rows), t = threadIdx.x;
    const bool in = t < rows;
    const int src = in ? __ldcg(&perm[t]) : 0;
    double l[kW];
#pragma unroll
    for (int j = 0; j < kW; j++) l[j] = j < jb && in && t >= jb ? __ldcg(&F[size_t(j0 + j) * m + j0 + t]) : 0.0;
    for (int q = t; q < kW * kW; q += blockDim.x) S.inv[q] = __ldcg(&Linv[q]);
    double v[NC];
#pragma unroll
    for (int c = 0; c < NC; c++) {
        v[c] = in ? col[c * m + j0 + src] : 0.0;
        if (t < kW) S.a[c][t] = v[c];
    }
    __syncthreads();
    diag_product(S, NC, jb);
    __syncthreads();
    if (t < jb) {
#pragma unroll
        for (int c = 0; c < NC; c++) col[c * m + j0 + t] = S.u[t][c];
    } else if (in) {
        double acc[NC];
        row_sums<NC>(acc, l, S);
#pragma unroll
        for (int c = 0; c < NC; c++) col[c * m + j0 + t] = v[c] - acc[c];
    }
    __syncthreads();
}

// back substitution with U of F on NC columns at col; the next panel's entries
// are fetched while this one is worked on
template <int NC>
__device__ void back_substitute(const LargeArgs &a, const double *F, const double *Uinv, double *col, WorkShared &S)
{
    const int m = a.m, t = threadIdx.x;
    constexpr int kVI = 2;   // entries of the inverse per thread (blockDim >= 128)
    double l[kW], ln[kW], vi[kVI];
    auto fetch = [&](int p, double (&d)[kW]) {
        const int j0 = p * kW, jb = min(kW, m - j0);
#pragma unroll
        for (int j = 0; j < kW; j++) d[j] = j < jb && t < j0 ? __ldcg(&F[size_t(j0 + j) * m + t]) : 0.0;
#pragma unroll
        for (int q = 0; q < kVI; q++) {
            const int i = t + q * int(blockDim.x);
            vi[q] = i < kW * kW ? __ldcg(&Uinv[p * kW * kW + i]) : 0.0;
        }
    };
    fetch(a.np - 1, ln);
    for (int p = a.np - 1; p >= 0; p--) {
        const int j0 = p * kW, jb = min(kW, m - j0);
#pragma unroll
        for (int j = 0; j < kW; j++) l[j] = ln[j];
#pragma unroll
        for (int q = 0; q < kVI; q++) {
            const int i = t + q * int(blockDim.x);
            if (i < kW * kW) S.inv[i] = vi[q];
        }
        if (t >= j0 && t < j0 + jb) {
#pragma unroll
            for (int c = 0; c < NC; c++) S.a[c][t - j0] = col[c * m + t];
        }
        __syncthreads();
        if (p > 0) fetch(p - 1, ln);
        diag_product(S, NC, jb);
        __syncthreads();
        if (t < j0) {   // (a thread reads and writes its own rows of the columns only)
            double acc[NC];
            row_sums<NC>(acc, l, S);
#pragma unroll
            for (int c = 0; c < NC; c++) col[c * m + t] -= acc[c];
        } else if (t < j0 + jb) {
#pragma unroll
            for (int c = 0; c < NC; c++) col[c * m + t] = S.u[t - j0][c];
        }
        __syncthreads();   // S.u and S.inv read
    }
}

// false: a wait ran out
__device__ bool worker_cta(const LargeArgs &a, double *sh)
{
    __shared__ WorkShared S;
    const int m = a.m, r = a.r, R = a.R, np = a.np, t = threadIdx.x, w = int(blockIdx.x) - 2;
    const int64_t Nt = a.N - 1;
    const size_t mm = size_t(m) * m;
    // columns: D / B column w + i nw; right-hand column (nw - 1 - w) + i nw
    const int wr = a.nw - 1 - w;
    const int nD = w < m ? (m - w + a.nw - 1) / a.nw : 0, nR = wr < R ? (R - wr + a.nw - 1) / a.nw : 0;
    double *const D = sh, *const R0 = D + nD * m, *const Hc = R0 + nR * m, *const R1 = Hc + nD * m;
    uint32_t phase = 0;
    bool ok = true;
    int cur = 0;   // this element's right-hand columns: R0 (0) or R1 (1)

    auto rhs = [&](int64_t e, int q, int k) -> double {   // row k of right-hand column q of element e < N - 1
        if (q < r) return a.b[(size_t(e) * m + k) * r + q];
        double v = 0.0;
        if (e == 0) v += a.C[size_t(k) * m + (q - r)];
        if (e == Nt - 1) v += a.B[e * mm + size_t(k) * m + (q - r)];
        return v;
    };
    // LU of one element: D delivered panel by panel, the nbg background columns at
    // bg following; Cm: the C block still to be applied to the right-hand columns
    // `now` with the previous element's `prev` (null: none)
    auto factor = [&](int64_t e, double *bg, int nbg, const double *Cm, double *now, const double *prev) -> bool {
        const int par = int(e & 1);
        double *F = a.F + size_t(par) * mm;
        const double *Li = a.Linv + size_t(par) * np * kW * kW;
        const int32_t *pm = a.perm + size_t(par) * np * m;
        // F of this parity was last read in element e - 2, which every worker has to
        // have left: each adds one per element to its parity's count.  (One count for
        // both would not do: a worker without a matrix column holds up no panel, so it
        // may lag while the others' counts run ahead.)
        uint32_t *const done = a.ctr + kCtrDone + 16 * par;
        if (e >= 2 && !cta_wait(a, int(done - a.ctr), uint32_t((e / 2) * a.nw), &S.ok)) return false;
        auto panel_of = [&](int i) { return (w + i * a.nw) / kW; };   // of own D column i
        auto deliver = [&](int p) {   // own columns of panel p into F
            int n = 0;
            for (int i = 0; i < nD; i++) {
                if (panel_of(i) != p) continue;
                for (int k = t; k < m; k += blockDim.x) F[size_t(w + i * a.nw) * m + k] = D[i * m + k];
                n++;
            }
            if (n) cta_signal(a, kCtrCols, uint32_t(n));   // uniform
        };
        deliver(0);
        int pD = 0, pB = 0, tile = 0, idle = 0, first = 0;   // first: own D columns before it are delivered
        while (first < nD && panel_of(first) == 0) first++;
        const int ntile = Cm ? np : 0;
        const int pDend = nD ? panel_of(nD - 1) : 0;   // panels that change own D columns
        while (pD < pDend || pB < np) {
            if (t == 0) S.seen = ctr_load(a.ctr + kCtrPanel);
            __syncthreads();
            const int avail = int(S.seen - uint32_t(e * np));
            __syncthreads();
            // an own column is next on the critical path: nothing else is begun
            const bool urgent = pD < pDend && panel_of(first) == pD + 1;
            if (pD < pDend && pD < avail) {
                // first the columns of the next panel, then the later ones
                int last = first;
                while (last < nD && panel_of(last) == pD + 1) last++;
                const double *Lp = Li + pD * kW * kW;
                const int32_t *pp = pm + size_t(pD) * m;
                if (last > first) {
                    with_count(last - first, [&](auto n) { apply_panel<decltype(n)::value>(a, F, Lp, pp, pD, D + first * m, S); });
                    deliver(pD + 1);
                }
                if (last < nD)
                    with_count(nD - last, [&](auto n) { apply_panel<decltype(n)::value>(a, F, Lp, pp, pD, D + last * m, S); });
                first = last;
                pD++;
                idle = 0;
            } else if (tile < ntile && !urgent) {
                with_count(nR, [&](auto n) {   // the running sums stay in `now`, which then becomes rhs - sum
                    constexpr int NC = decltype(n)::value;
                    double acc[NC], v[kW];
                    load_row16(v, Cm, m, t, tile * kW);
                    if (t < m) {
#pragma unroll
                        for (int c = 0; c < NC; c++) acc[c] = tile > 0 ? now[c * m + t] : 0.0;
                        dot16<NC>(acc, v, prev, m, tile * kW);
#pragma unroll
                        for (int c = 0; c < NC; c++)
                            now[c * m + t] = tile + 1 < ntile ? acc[c] : rhs(e, wr + c * a.nw, t) - acc[c];
                    }
                });
                tile++;
                __syncthreads();
            } else if (pB < np && pB < avail && tile >= ntile && !urgent) {
                if (a.stall_ns > 0 && nD == 0) __nanosleep(a.stall_ns);
                with_count(nbg, [&](auto n) {
                    apply_panel<decltype(n)::value>(a, F, Li + pB * kW * kW, pm + size_t(pB) * m, pB, bg, S);
                });
                pB++;
                idle = 0;
            } else {
                if (t == 0) {   // (no backward sweep runs beside a factorization: nothing resets this one)
                    S.ok = ++idle < a.polls && ((idle & 63) != 63 || !ctr_load(a.ctr + kCtrAbort));
                    if (!S.ok) atomicExch(a.ctr + kCtrAbort, 1u);
                }
                __syncthreads();
                const bool go = S.ok != 0;
                __syncthreads();
                if (!go) return false;
            }
        }
        if (!cta_wait(a, kCtrInv, uint32_t((e + 1) * np), &S.ok)) return false;
        with_count(nbg, [&](auto n) {
            back_substitute<decltype(n)::value>(a, F, a.Uinv + size_t(par) * np * kW * kW, bg, S);
        });
        cta_signal(a, int(done - a.ctr), 1);
        return true;
    };

    // ---- forward over T'
    for (int64_t e = 0; e < Nt && ok; e++) {
        double *now = cur ? R1 : R0, *prev = cur ? R0 : R1;
        for (int i = 0; i < nD; i++)
            for (int k = t; k < m; k += blockDim.x) D[i * m + k] = a.A[e * mm + size_t(k) * m + w + i * a.nw];
        for (int i = 0; i < nR && e == 0; i++)   // later elements: with the last tile of C G
            for (int k = t; k < m; k += blockDim.x) now[i * m + k] = rhs(0, wr + i * a.nw, k);
        __syncthreads();
        if (e > 0) with_count(nD, [&](auto n) { block_product<decltype(n)::value>(D, Hc, a.C + e * mm, m); });
        __syncthreads();
        const int nB = e < Nt - 1 ? nD : 0;
        for (int i = 0; i < nB; i++)
            for (int k = t; k < m; k += blockDim.x) Hc[i * m + k] = a.B[e * mm + size_t(k) * m + w + i * a.nw];
        __syncthreads();
        // background: R0 | H or H | R1
        ok = factor(e, cur ? (nB ? Hc : R1) : R0, nB + nR, e > 0 && nR ? a.C + e * mm : nullptr, now, prev);
        if (!ok) break;
        for (int i = 0; i < nB; i++)
            for (int k = t; k < m; k += blockDim.x) a.H[e * mm + size_t(w + i * a.nw) * m + k] = Hc[i * m + k];
        for (int i = 0; i < nR; i++)
            for (int k = t; k < m; k += blockDim.x) a.G[(size_t(e) * R + wr + i * a.nw) * m + k] = now[i * m + k];
        cur ^= 1;
    }
    if (!ok) return false;
    if (Nt > 0) {
        if (!grid_barrier(a, phase, &S.ok)) return false;   // every H is written
        // ---- backward: X_k = G_k - H_k X_{k+1}, thread t row t; sixteen columns
        // of H_k at a time, the next sixteen on their way
        for (int64_t k = Nt - 2; k >= 0; k--) {
            const double *Hk = a.H + k * mm, *X = cur ? R0 : R1;   // X_{k+1}: the last written
            double *Y = cur ? R1 : R0;
            with_count(nR, [&](auto n) {
                constexpr int NC = decltype(n)::value;
                if (t >= m) return;
                double acc[NC], h[kW], hn[kW];
#pragma unroll
                for (int c = 0; c < NC; c++) acc[c] = 0.0;
#pragma unroll
                for (int j = 0; j < kW; j++) h[j] = j < m ? __ldcg(&Hk[size_t(j) * m + t]) : 0.0;
                for (int q = 0; q < m; q += kW) {
#pragma unroll
                    for (int j = 0; j < kW; j++) hn[j] = q + kW + j < m ? __ldcg(&Hk[size_t(q + kW + j) * m + t]) : 0.0;
                    dot16<NC>(acc, h, X, m, q);
#pragma unroll
                    for (int j = 0; j < kW; j++) h[j] = hn[j];
                }
#pragma unroll
                for (int c = 0; c < NC; c++) {
                    double *g = &a.G[(size_t(k) * R + wr + c * a.nw) * m + t];
                    Y[c * m + t] = *g - acc[c];
                    *g = Y[c * m + t];
                }
            });
            cur ^= 1;
            __syncthreads();
            if (t == 0) asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(a.ctr + kCtrBeat) : "memory");
        }
        if (!grid_barrier(a, phase, &S.ok)) return false;   // every X is written
    }
    // ---- border: S = A - B Z_0 - C Z_{N-2} (N = 1: A + B + C) in D, s likewise in
    // R0 (own right-hand columns below r); H and R1 hold the columns of Z and Y
    const double *An = a.A + Nt * mm, *Bn = a.B + Nt * mm, *Cn = a.C + Nt * mm;
    int nS = 0;
    while (nS < nR && wr + nS * a.nw < r) nS++;
    for (int i = 0; i < nD; i++)
        for (int k = t; k < m; k += blockDim.x) {
            const size_t at = size_t(k) * m + w + i * a.nw;
            D[i * m + k] = Nt == 0 ? An[at] + Bn[at] + Cn[at] : An[at];
        }
    for (int i = 0; i < nS; i++)
        for (int k = t; k < m; k += blockDim.x) R0[i * m + k] = a.b[(size_t(Nt) * m + k) * r + wr + i * a.nw];
    __syncthreads();
    for (int side = 0; side < 2 && Nt > 0; side++) {
        const double *Gk = a.G + (side ? size_t(Nt - 1) : 0) * R * m, *Mk = side ? Cn : Bn;
        for (int i = 0; i < nD; i++)
            for (int k = t; k < m; k += blockDim.x) Hc[i * m + k] = __ldcg(&Gk[size_t(r + w + i * a.nw) * m + k]);
        for (int i = 0; i < nS; i++)
            for (int k = t; k < m; k += blockDim.x) R1[i * m + k] = __ldcg(&Gk[size_t(wr + i * a.nw) * m + k]);
        __syncthreads();
        with_count(nD, [&](auto n) { block_product<decltype(n)::value>(D, Hc, Mk, m); });
        with_count(nS, [&](auto n) { block_product<decltype(n)::value>(R0, R1, Mk, m); });
        __syncthreads();
    }
    ok = factor(Nt, R0, nS, nullptr, nullptr, nullptr);
    if (!ok) return false;
    for (int i = 0; i < nS; i++)
        for (int k = t; k < m; k += blockDim.x) a.x[(size_t(Nt) * m + k) * r + wr + i * a.nw] = R0[i * m + k];
    if (!grid_barrier(a, phase, &S.ok)) return false;   // x_{N-1} is written
    // ---- x_k = Y_k - Z_k x_{N-1}: element and right-hand side per pass, thread t row t
    for (int64_t job = w; job < Nt * r; job += a.nw) {
        const int64_t k = job / r;
        const int c = int(job - k * r);
        const double *Gk = a.G + size_t(k) * R * m;
        for (int q = t; q < m; q += blockDim.x) sh[q] = __ldcg(&a.x[(size_t(Nt) * m + q) * r + c]);
        __syncthreads();
        if (t < m) {
            double s[1] = {0.0}, h[kW];
            for (int q = 0; q < m; q += kW) {
#pragma unroll
                for (int j = 0; j < kW; j++) h[j] = q + j < m ? __ldcg(&Gk[size_t(r + q + j) * m + t]) : 0.0;
                dot16<1>(s, h, sh, m, q);
            }
            a.x[(size_t(k) * m + t) * r + c] = __ldcg(&Gk[size_t(c) * m + t]) - s[0];
        }
        __syncthreads();
    }
    return true;
}

__global__ void __launch_bounds__(512, 1) k_strip_large(const __grid_constant__ LargeArgs a)
{
    extern __shared__ double sh[];
    if (blockIdx.x == 0) panel_cta(a, sh);
    else if (blockIdx.x == 1) helper_cta(a);
    else if (!worker_cta(a, sh)) {
        // nothing of an unfinished solution passes for one
        const int64_t n = a.N * a.m * a.r;
        for (int64_t i = (int64_t(blockIdx.x) - 2) * blockDim.x + threadIdx.x; i < n; i += int64_t(a.nw) * blockDim.x)
            a.x[i] = nan("");
    }
}

int strip_panels(int m) { return (m + kW - 1) / kW; }

// What a launch may ask for.  The limit belongs to the kernel, not to the launch, so
// every call sets this one: a smaller one would fail another thread's launch.
constexpr size_t kMaxSmem = 200 * 1024;
size_t large_smem(int m, int r, int nw)
{
    const size_t nD = size_t(m + nw - 1) / nw, nR = size_t(m + r + nw - 1) / nw;
    return sizeof(double) * std::max<size_t>(2 * nD + 2 * nR, kW) * m;   // a worker's columns; the panel's multipliers
}

}  // namespace

// H, G, F, the diagonal blocks' inverses, row orders and counters
size_t strip_large_work_doubles(int64_t N, int m, int r)
{
    const size_t nt = size_t(std::max<int64_t>(N - 1, 1)), R = size_t(r) + m, np = strip_panels(m);
    return nt * (size_t(m) * m + size_t(m) * R) + 2 * size_t(m) * m + 4 * np * kW * kW + np * m + kCtrWords / 2 + 2;
}

cudaError_t launch_strip_large(int64_t N, int m, int r, const double *A, const double *B, const double *C, const double *b,
                               double *x, double *work, int32_t *status, cudaStream_t st, const bc_strip_debug &dbg)
{
    if (m > kMaxM) return cudaErrorInvalidValue;
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    LargeArgs a{};
    a.N = N; a.m = m; a.r = r; a.R = r + m;
    a.np = strip_panels(m);
    // one CTA per SM; no more workers than there are columns of the larger kind
    a.nw = std::min(sms - 2, m + r);
    if (dbg.max_blocks > 0) a.nw = std::min(a.nw, dbg.max_blocks - 2);
    const int nD = (m + a.nw - 1) / std::max(a.nw, 1), nR = (a.R + a.nw - 1) / std::max(a.nw, 1);
    const size_t smem = large_smem(m, r, std::max(a.nw, 1));
    if (a.nw < kW || nD > kMaxD || nR > kMaxR || smem > kMaxSmem) return cudaErrorNotSupported;
    a.A = A; a.B = B; a.C = C; a.b = b; a.x = x;
    const size_t nt = size_t(std::max<int64_t>(N - 1, 1));
    double *w = work;
    a.H = w; w += nt * size_t(m) * m;
    a.G = w; w += nt * size_t(m) * a.R;
    a.F = w; w += 2 * size_t(m) * m;
    a.Linv = w; w += 2 * size_t(a.np) * kW * kW;
    a.Uinv = w; w += 2 * size_t(a.np) * kW * kW;
    a.perm = reinterpret_cast<int32_t *>(w); w += size_t(a.np) * m;
    a.ctr = reinterpret_cast<uint32_t *>(w); w += kCtrWords / 2;
    a.status = status ? status : reinterpret_cast<int32_t *>(w);
    a.polls = dbg.wait_polls > 0 ? dbg.wait_polls : kPollLimit;
    a.withhold = dbg.withhold_panels;
    a.stall_ns = dbg.stall_ns;
    e = cudaMemsetAsync(a.ctr, 0, kCtrWords * sizeof(uint32_t), st);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_strip_large, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMaxSmem));
    if (e != cudaSuccess) return e;
    void *args[] = {&a};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_strip_large), dim3(unsigned(a.nw + 2)),
                                       dim3(unsigned(32 * (inverse_warp(m) + 1))), args, smem, st);
}

}  // namespace bc
