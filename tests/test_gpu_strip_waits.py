"""The waits of the large-block strip solve (one cooperative launch whose blocks exchange columns through counters)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2501_17967_gb300 as bc  # noqa: E402

pytestmark = pytest.mark.gpu


def system(nsys, N, m, r, seed=1):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(seed)
    A = rng.standard_normal((nsys, N, m, m)) + 4.0 * m * np.eye(m)
    B, C = rng.standard_normal((2, nsys, N, m, m))
    return [torch.from_numpy(t).cuda() for t in (A, B, C, rng.standard_normal((nsys, N, m, r)))]


def debug_solve(A, B, C, b, **debug):
    """bc_debug_strip_solve: x (zeros where nothing was written) and the status words."""
    nsys, N, m, r = b.shape
    x, status = torch.zeros_like(b), torch.full((nsys,), 7, dtype=torch.int32, device="cuda")
    work = bc.strip_workspace(nsys, N, m, r, "cuda")
    ptr = [ctypes.c_void_p(t.data_ptr()) for t in (A, B, C, b, x, work, status)]
    bc._check(bc._load().bc_debug_strip_solve(nsys, N, m, r, *ptr, ctypes.byref(bc._StripDebug(**debug)), None))
    torch.cuda.synchronize()
    return x, status.cpu().tolist()


# blocks without a matrix column: 32 of 72, 1 of 34, 16 of 150 (m = 134)
@pytest.mark.parametrize("N,m,r", [(7, 40, 32), (6, 33, 1), (5, 134, 32)])
def test_blocks_without_a_matrix_column_may_lag(N, m, r):
    """The factored panels of an element stay until every block has applied them."""
    args = system(1, N, m, r)
    want = bc.strip_solve(*args)
    x, status = debug_solve(*args, stall_ns=300000)
    assert status == [0] and torch.equal(x, want)
