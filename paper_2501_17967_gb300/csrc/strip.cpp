// C ABI of the strip solve (include/boxcode.h, bc_strip_*): argument checks and
// the launches, one thread block per system for blocks up to 32 x 32
// (kernels_strip.cu), one cooperative launch per system for larger ones
// (kernels_strip_large.cu).
#include <algorithm>
#include <cstdint>

#include "bc_internal.h"

namespace bc {
namespace {

bool strip_on_device(const void *p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

constexpr int kSmallM = 32;     // blocks up to this size: one thread block per system
constexpr int kLargeM = 448;    // one panel row per thread of the panel block

bool strip_shape_ok(int64_t nsys, int64_t N, int m, int r)
{
    return nsys >= 0 && nsys <= INT32_MAX && N >= 1 && m >= 1 && m <= kLargeM && r >= 1 && r <= 32 &&
           (m <= kSmallM || N * int64_t(m) <= INT32_MAX / 4);
}

// doubles of scratch: small blocks, per system; large blocks, one system's
// arrays (systems run one after another)
size_t strip_scratch_doubles(int64_t nsys, int64_t N, int m, int r)
{
    return m <= kSmallM ? size_t(nsys) * strip_work_doubles(N, m, r) : strip_large_work_doubles(N, m, r);
}

bc_status strip_solve(int64_t nsys, int64_t N, int m, int r, const double *A, const double *B, const double *C,
                      const double *b, double *x, void *work, int32_t *status, const bc_strip_debug &dbg, void *stream)
{
    if (!strip_shape_ok(nsys, N, m, r)) {
        set_error("bc_strip_solve: need nsys >= 0, N >= 1, 1 <= m <= 448, 1 <= r <= 32");
        return BC_ERR_ARG;
    }
    if (nsys == 0) return BC_OK;
    if (!A || !B || !C || !b || !x || !work) { set_error("bc_strip_solve: NULL argument"); return BC_ERR_ARG; }
    for (const void *p : {(const void *)A, (const void *)B, (const void *)C, (const void *)b, (const void *)x,
                          (const void *)work})
        if (!strip_on_device(p)) { set_error("bc_strip_solve: every array must be device memory"); return BC_ERR_ARG; }
    if (status && !strip_on_device(status)) { set_error("bc_strip_solve: status must be device memory"); return BC_ERR_ARG; }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double *wk = static_cast<double *>(work);
    cudaError_t e = cudaSuccess;
    if (m <= kSmallM) {
        e = launch_strip(nsys, N, m, r, A, B, C, b, x, wk, status, st);
    } else {
        const size_t mm = size_t(m) * m;
        for (int64_t s = 0; s < nsys && e == cudaSuccess; s++)
            e = launch_strip_large(N, m, r, A + s * N * mm, B + s * N * mm, C + s * N * mm, b + s * N * m * r,
                                   x + s * N * m * r, wk, status ? status + s : nullptr, st, dbg);
    }
    if (e == cudaErrorNotSupported) {
        set_error("bc_strip_solve: blocks of m = %d with r = %d need more SMs than there are (122 for every m and r)", m, r);
        return BC_ERR_UNSUPPORTED;
    }
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("bc_strip_solve: %s (%s)", cudaGetErrorName(e), cudaGetErrorString(e));
        return BC_ERR_CUDA;
    }
    return BC_OK;
}

}  // namespace
}  // namespace bc

using namespace bc;

bc_status bc_strip_workspace(int64_t nsys, int64_t N, int m, int r, int64_t *bytes)
{
    if (!bytes || !strip_shape_ok(nsys, N, m, r)) {
        set_error("bc_strip_workspace: need nsys >= 0, N >= 1, 1 <= m <= 448, 1 <= r <= 32");
        return BC_ERR_ARG;
    }
    *bytes = int64_t(sizeof(double) * strip_scratch_doubles(nsys, N, m, r));
    return BC_OK;
}

bc_status bc_strip_solve(int64_t nsys, int64_t N, int m, int r, const double *A, const double *B, const double *C,
                         const double *b, double *x, void *work, int32_t *status, void *stream)
{
    return strip_solve(nsys, N, m, r, A, B, C, b, x, work, status, bc_strip_debug{}, stream);
}

bc_status bc_debug_strip_solve(int64_t nsys, int64_t N, int m, int r, const double *A, const double *B,
                               const double *C, const double *b, double *x, void *work, int32_t *status,
                               const bc_strip_debug *debug, void *stream)
{
    if (!debug || debug->wait_polls < 0 || debug->wait_polls > (1 << 22) || debug->stall_ns < 0 || debug->stall_ns > 1000000 || debug->max_blocks < 0) {
        set_error("bc_debug_strip_solve: need wait_polls in [0, 2^22], stall_ns in [0, 1000000], max_blocks >= 0");
        return BC_ERR_ARG;
    }
    return strip_solve(nsys, N, m, r, A, B, C, b, x, work, status, *debug, stream);
}
