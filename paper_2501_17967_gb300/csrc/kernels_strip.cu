// Strip solve (Sec. 3.3): the multidomain collocation system of the strip
// couples each element only to its neighbours around the closed strip, so it
// is block tridiagonal with two corner blocks:
//
//   C[k] x[k-1] + A[k] x[k] + B[k] x[k+1] = b[k],   k = 0..N-1, indices mod N.
//
// Solved by block LU with the corners as a border (the rank-m form of the
// paper's Woodbury correction): x_{N-1} is eliminated last.  The first N - 1
// block rows form a tridiagonal T' whose right-hand side also carries the
// border column E (C_0 in row 0, B_{N-2} in row N-2: they couple to x_{N-1}),
// so m columns ride through the sweep beside the r right-hand sides:
//   D_0 = A_0; D_k = A_k - C_k H_{k-1};
//   [H_k | g_k] = D_k^-1 [B_k | (b_k | E_k) - C_k g_{k-1}]      (R = r + m columns in g)
//   X_{N-2} = g_{N-2}, X_k = g_k - H_k X_{k+1}                  (X = [Y | Z])
//   S = A_{N-1} - B_{N-1} Z_0 - C_{N-1} Z_{N-2},  S x_{N-1} = b_{N-1} - B_{N-1} Y_0 - C_{N-1} Y_{N-2}
//   x_k = Y_k - Z_k x_{N-1}.
// Every D_k and S are factored by LU with partial pivoting.
//
// Blocks up to 32 x 32 (interface-sized blocks): one CTA of 1 to 8 warps per
// system, many systems at once; the blocks of the current step live in shared
// memory, H_k and X_k in a global workspace.  Larger blocks (the paper's
// elements of 16 x 24 nodes): kernels_strip_large.cu.
// FP64.
#include <cuda_runtime.h>

#include <algorithm>

#include "bc_internal.h"

namespace bc {
namespace {

// ---------------------------------------------------------------------------
// Small blocks.  The step is a chain of short FP64 phases on one SM: at m = 17,
// r = 1 about 22,000 FMAs, each 32 of which hold a sub-partition's FP64 pipe
// for 64 cycles, so a phase should fill whole warps and wait little.
//  * Phases run over flattened (row, column) lists, so that no lane idles at the
//    ends of short rows; the list is walked without divisions.
//  * Elimination scales the pivot row (unit upper factor), so that neither the
//    update nor the back substitution divides; warp 0 updates the next pivot
//    column first and searches it (one element per lane, reduced by redux) and
//    takes the reciprocal while the other warps update the rest, of which it
//    gets a share shortened by that work.
//  * The next element's blocks are copied (cp.async) while this one is solved.
// 608 systems, N = 256, m = 17, r = 1: 34.5 ms with one warp per system, divisions
// in the index arithmetic and 2m border columns; 12.7 ms so (the FP64 pipe alone
// would take 9).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void strip_copy8(double *dst, const double *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void strip_copy_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Position t of a list with `cols` columns per row, advanced without divisions.
struct Walk {
    int i, c, cols;
    __device__ __forceinline__ Walk(int t, int n) : i(t / n), c(t - (t / n) * n), cols(n) {}
    __device__ __forceinline__ void step(int d)
    {
        c += d;
        while (c >= cols) {
            c -= cols;
            i++;
        }
    }
};

constexpr int kMaxM = 32, kMaxR = 32;   // largest block and number of right-hand sides

struct StripPivot {
    int row, bad;
    double inv;
};

// Warp 0: the pivot of column j (rows j .. m-1, one per lane; v: the lane's
// entry) and its reciprocal.  A NaN sorts above every number; a zero or
// non-finite pivot is flagged and eliminates nothing.
__device__ __forceinline__ void strip_pivot(double v, int j, int m, StripPivot *pv)
{
    const int lane = threadIdx.x & 31;
    const bool in = lane >= j && lane < m;
    const unsigned long long key = static_cast<unsigned long long>(__double_as_longlong(v)) & 0x7FFFFFFFFFFFFFFFull;
    const unsigned hi = in ? unsigned(key >> 32) : 0u;
    const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
    const bool c1 = in && hi == mh;
    const unsigned ml = __reduce_max_sync(0xffffffffu, c1 ? unsigned(key) : 0u);
    const int p = __ffs(__ballot_sync(0xffffffffu, c1 && unsigned(key) == ml)) - 1;
    const double d = __shfl_sync(0xffffffffu, v, p);
    const bool good = d != 0.0 && isfinite(d);
    const double inv = good ? 1.0 / d : 0.0;
    if (lane == 0) {
        pv->row = p;
        pv->inv = inv;
        if (!good) pv->bad = 1;
    }
}

// M [m][W] (shared): columns [0, m) factored with partial pivoting, columns
// [m, W) become M[:, 0:m]^-1 times themselves.  All threads; ends with a barrier.
__device__ void strip_lu_solve(double *M, int m, int W, StripPivot *pv)
{
    const int tid = threadIdx.x, nt = blockDim.x, w = tid >> 5, lane = tid & 31, nw = nt >> 5;
    if (w == 0) strip_pivot(lane < m ? M[lane * W] : 0.0, 0, m, pv);
    __syncthreads();
    for (int j = 0; j < m; j++) {
        // exchange rows j and p, row j scaled
        const int p = pv->row;
        const double inv = pv->inv;
        for (int c = j + tid; c < W; c += nt) {
            const double v = M[p * W + c];
            if (p != j) M[p * W + c] = M[j * W + c];
            M[j * W + c] = v * inv;
        }
        __syncthreads();
        const int rows = m - 1 - j, cols = W - j - 2;
        if (rows > 0) {
            const double *Lj = M + (j + 1) * W + j, *Uj = M + j * W;
            if (w == 0) {   // the next pivot column
                double v = 0.0;
                if (lane > j && lane < m) {
                    v = fma(-M[lane * W + j], Uj[j + 1], M[lane * W + j + 1]);
                    M[lane * W + j + 1] = v;
                }
                strip_pivot(v, j + 1, m, pv);
            }
            // columns j + 2 .. W - 1: warp 0's search counts as 14 rounds
            const int n = rows * cols, Q = (n + 31) >> 5;
            const int q0 = nw == 1 ? Q : max(0, (Q - 14 * (nw - 1)) / nw);
            const int lo = w == 0 ? lane : q0 * 32 + (w - 1) * 32 + lane, hi = w == 0 ? min(n, q0 * 32) : n;
            const int d = w == 0 ? 32 : 32 * (nw - 1);
            Walk k(lo, cols);
            int t = lo;
            for (; t + 3 * d < hi; t += 4 * d) {   // four independent updates in flight
                double *q[4];
                double l[4], u[4], x[4];
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    q[e] = M + (j + 1 + k.i) * W + j + 2 + k.c;
                    l[e] = Lj[k.i * W];
                    u[e] = Uj[j + 2 + k.c];
                    x[e] = *q[e];
                    k.step(d);
                }
#pragma unroll
                for (int e = 0; e < 4; e++) *q[e] = fma(-l[e], u[e], x[e]);
            }
            for (; t < hi; t += d) {
                double *q = M + (j + 1 + k.i) * W + j + 2 + k.c;
                *q = fma(-Lj[k.i * W], Uj[j + 2 + k.c], *q);
                k.step(d);
            }
        }
        __syncthreads();
    }
    // back substitution with the unit upper factor
    const int R = W - m;
    for (int i = m - 1; i > 0; i--) {
        Walk k(tid, R);
        for (int t = tid; t < i * R; t += nt) {
            double *q = M + k.i * W + m + k.c;
            *q = fma(-M[k.i * W + i], M[i * W + m + k.c], *q);
            k.step(nt);
        }
        __syncthreads();
    }
}

// out[i][c] -= sum_t P[i][t] Q[t][c], i < m, c < nc; column c of the output at
// c (c < m0) or c + shift; four outputs per thread in flight.
__device__ __forceinline__ void strip_sub_mm(double *out, int lo, int m0, int shift, const double *P, const double *Q,
                                             int lq, int m, int nc)
{
    const int nt = blockDim.x, n = m * nc;
    Walk k(threadIdx.x, nc);
    for (int t0 = threadIdx.x; t0 < n; t0 += 4 * nt) {
        double *o[4];
        const double *p[4], *q[4];
        double s[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
            const bool in = t0 + e * nt < n;   // past the end: repeats the first, not stored
            const int i = in ? k.i : 0, c = in ? k.c : 0;
            o[e] = in ? out + i * lo + (c < m0 ? c : c + shift) : nullptr;
            p[e] = P + i * m;
            q[e] = Q + c;
            s[e] = in ? *o[e] : 0.0;
            k.step(nt);
        }
        const int live = min(4, (n - t0 + nt - 1) / nt);
        if (live == 4) {
            for (int t = 0; t < m; t++)
#pragma unroll
                for (int e = 0; e < 4; e++) s[e] = fma(-p[e][t], q[e][t * lq], s[e]);
        } else {
            for (int t = 0; t < m; t++)
#pragma unroll
                for (int e = 0; e < 3; e++)
                    if (e < live) s[e] = fma(-p[e][t], q[e][t * lq], s[e]);
        }
#pragma unroll
        for (int e = 0; e < 4; e++)
            if (o[e]) *o[e] = s[e];
    }
}

__global__ void __launch_bounds__(256)
k_strip_small(int64_t N, int m, int r, const double *__restrict__ A, const double *__restrict__ B,
              const double *__restrict__ C, const double *__restrict__ b, double *__restrict__ x,
              double *__restrict__ work, int32_t *__restrict__ status)
{
    extern __shared__ double sh[];
    __shared__ StripPivot pv;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int R = r + m, W = 2 * m + R;   // columns: D | B, H | b, Y | E, Z
    const int64_t s = blockIdx.x, Nt = N - 1;
    const int mm = m * m, mR = m * R;
    const double *As = A + s * N * mm, *Bs = B + s * N * mm, *Cs = C + s * N * mm, *bs = b + s * N * m * r;
    double *xs = x + s * N * m * r;
    double *Hs = work + s * N * (mm + mR), *Gs = Hs + N * mm;   // [N][m][m], [N][m][R]
    double *aug[2] = {sh, sh + m * W}, *third = sh + 2 * m * W;   // third: m (m + R)
    if (tid == 0) pv.bad = 0;
    // element k into aug[k & 1] and its C block into third[(k & 1) mm]
    auto fetch = [&](int64_t k) {
        double *M = aug[k & 1], *sC = third + (k & 1) * mm;
        Walk q(tid, W);
        for (int t = tid; t < m * W; t += nt) {
            const int i = q.i, c = q.c;
            if (c < m) strip_copy8(M + t, As + k * mm + i * m + c);
            else if (c < 2 * m) {
                if (k < Nt - 1) strip_copy8(M + t, Bs + k * mm + i * m + (c - m));
                else M[t] = 0.0;
            } else if (c < 2 * m + r) strip_copy8(M + t, bs + (k * m + i) * r + (c - 2 * m));
            else {
                const int e = i * m + (c - 2 * m - r);
                double v = 0.0;
                if (k == 0) v += Cs[e];
                if (k == Nt - 1) v += Bs[k * mm + e];
                M[t] = v;
            }
            q.step(nt);
        }
        if (k > 0)
            for (int t = tid; t < mm; t += nt) strip_copy8(sC + t, Cs + k * mm + t);
    };
    // ---- forward sweep
    if (Nt > 0) fetch(0);
    for (int64_t k = 0; k < Nt; k++) {
        strip_copy_wait();
        __syncthreads();
        double *M = aug[k & 1], *prev = aug[(k + 1) & 1];
        if (k > 0) {   // D = A - C H_{k-1}, rhs - C g_{k-1}
            strip_sub_mm(M, W, m, m, third + (k & 1) * mm, prev + m, W, m, m + R);
            __syncthreads();
        }
        if (k + 1 < Nt) fetch(k + 1);
        strip_lu_solve(M, m, W, &pv);
        Walk q(tid, m + R);
        for (int t = tid; t < m * (m + R); t += nt) {
            const double v = M[q.i * W + m + q.c];
            if (q.c < m) Hs[k * mm + q.i * m + q.c] = v;
            else Gs[k * mR + q.i * R + (q.c - m)] = v;
            q.step(nt);
        }
    }
    // ---- backward sweep: X_k = g_k - H_k X_{k+1} over g; three buffers of
    // [H | g] in turn: X_{k+1}, element k, element k - 1 on its way
    double *X = aug[(Nt + 1) & 1] + 2 * m;   // X_{N-2}, leading dimension W
    int ldx = W;
    if (Nt > 1) {
        double *buf[3] = {aug[Nt & 1], third, aug[(Nt + 1) & 1]};
        __syncthreads();
        auto fetch_back = [&](int64_t k, double *M) {
            for (int t = tid; t < mm; t += nt) strip_copy8(M + t, Hs + k * mm + t);
            for (int t = tid; t < mR; t += nt) strip_copy8(M + mm + t, Gs + k * mR + t);
        };
        fetch_back(Nt - 2, buf[0]);
        int at = 0;
        for (int64_t k = Nt - 2; k >= 0; k--) {
            strip_copy_wait();
            __syncthreads();   // element k is here, X_{k+1} complete
            double *M = buf[at];
            if (k > 0) fetch_back(k - 1, buf[(at + 1) % 3]);
            strip_sub_mm(M + mm, R, R, 0, M, X, ldx, m, R);
            __syncthreads();
            for (int t = tid; t < mR; t += nt) Gs[k * mR + t] = M[mm + t];
            X = M + mm;
            ldx = R;
            at = (at + 1) % 3;
        }
    }
    __syncthreads();
    // ---- border: [S | s], leading dimension m + r, in a buffer that X is not in
    double *S = (X >= aug[0] && X < aug[0] + m * W) ? aug[1] : aug[0];
    const int ldS = m + r;
    const double *An = As + Nt * mm, *Bn = Bs + Nt * mm, *Cn = Cs + Nt * mm;
    for (int t = tid; t < m * ldS; t += nt) {
        const int i = t / ldS, c = t % ldS;
        double v = c < m ? An[i * m + c] : bs[(Nt * m + i) * r + (c - m)];
        if (Nt == 0) {
            if (c < m) v += Bn[i * m + c] + Cn[i * m + c];
        } else {
            const int g = c < m ? r + c : c - m;   // column of [Y | Z]
            const double *Gl = Gs + (Nt - 1) * mR;
            for (int q = 0; q < m; q++) v = fma(-Bn[i * m + q], X[q * ldx + g], v);
            for (int q = 0; q < m; q++) v = fma(-Cn[i * m + q], Gl[q * R + g], v);
        }
        S[t] = v;
    }
    __syncthreads();
    strip_lu_solve(S, m, ldS, &pv);
    // ---- x_{N-1} from the border, x_k = Y_k - Z_k x_{N-1}
    for (int t = tid; t < m * r; t += nt) xs[Nt * m * r + t] = S[(t / r) * ldS + m + t % r];
    for (int64_t t = tid; t < Nt * m * r; t += nt) {
        const int64_t row = t / r;
        const int c = int(t - row * r);
        const double *g = Gs + row * R;
        double v = g[c], v1 = 0.0;
        int q = 0;
        for (; q + 1 < m; q += 2) {
            v = fma(-g[r + q], S[q * ldS + m + c], v);
            v1 = fma(-g[r + q + 1], S[(q + 1) * ldS + m + c], v1);
        }
        if (q < m) v = fma(-g[r + q], S[q * ldS + m + c], v);
        xs[t] = v + v1;
    }
    if (status && tid == 0) status[s] = pv.bad;
}

}  // namespace

// two augmented blocks and a third buffer of [H | g] (or two C blocks)
size_t strip_smem_bytes(int m, int r)
{
    const size_t R = size_t(r) + m, W = 2 * size_t(m) + R;
    return sizeof(double) * (2 * m * W + m * (m + R));
}

size_t strip_work_doubles(int64_t N, int m, int r) { return size_t(N) * (size_t(m) * m + size_t(m) * (r + m)); }

cudaError_t launch_strip(int64_t nsys, int64_t N, int m, int r, const double *A, const double *B, const double *C,
                         const double *b, double *x, double *work, int32_t *status, cudaStream_t st)
{
    const size_t sm = strip_smem_bytes(m, r);
    // the limit of the largest shape in every call: it belongs to the kernel, and a
    // smaller one would fail another thread's launch
    const cudaError_t ce = cudaFuncSetAttribute(k_strip_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                int(strip_smem_bytes(kMaxM, kMaxR)));
    if (ce != cudaSuccess) return ce;
    // Warps per system, by the entries of the augmented block and the systems an
    // SM gets.  Measured (ms at 1 / 2 / 4 / 8 warps): m = 8, 608 systems 4.8 / 3.9 /
    // 4.3 / 8.7; m = 17, 608 systems 21.7 / 16.0 / 12.7 / 20.1, one system 21.2 / 14.2 /
    // 9.3 / 8.4; m = 32, 600 systems 54 / 31 / 21 / 17; m = 3, 3 systems 1.2 / 1.4 / 1.7 / 2.5.
    const int e = m * (3 * m + r);
    const bool many = nsys > 2 * 152;
    const int nw = e < 128 ? 1 : e < 400 ? (many ? 2 : 4) : many && e < 2200 ? 4 : 8;
    k_strip_small<<<dim3(unsigned(nsys)), 32 * nw, sm, st>>>(N, m, r, A, B, C, b, x, work, status);
    return cudaGetLastError();
}

}  // namespace bc
