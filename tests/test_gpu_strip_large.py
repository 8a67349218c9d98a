"""The large-block strip solve at the edges of its tiling: a short last panel (m not a multiple of 16), one to fourteen row
warps, workers with no or several columns, every N at which its phases differ (1, 2, 3), many right-hand sides, rows that
force off-diagonal pivots, and a singular system; against numpy's dense solve.  Bar: 1e-12 relative max-norm, as for the
other well-conditioned strips."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2501_17967_gb300 as bc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys,N,m,r", [(1, 1, 33, 1), (2, 2, 48, 3), (1, 3, 47, 32), (1, 4, 65, 2), (1, 3, 150, 1), (1, 2, 151, 1),
                                        (1, 3, 200, 31), (1, 2, 301, 1), (1, 3, 448, 32), (1, 1, 447, 5)])
def test_large_blocks(nsys, N, m, r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(1000 * N + 10 * m + r)
    A = rng.standard_normal((nsys, N, m, m)) + 4.0 * m * np.eye(m)[rng.permutation(m)]
    B, C = rng.standard_normal((2, nsys, N, m, m))
    b = rng.standard_normal((nsys, N, m, r))
    args = [torch.from_numpy(t).cuda() for t in (A, B, C, b)]
    x, status = bc.strip_solve(*args, return_status=True)
    again = bc.strip_solve(*args)
    assert torch.equal(x, again)      # no race decides a result
    x = x.cpu().numpy()
    assert not status.any()
    for s in range(nsys):
        M = np.zeros((N * m, N * m))
        for k in range(N):
            for blk, j in ((A, k), (B, (k + 1) % N), (C, (k - 1) % N)):
                M[k * m:(k + 1) * m, j * m:(j + 1) * m] += blk[s, k]
        ref = np.linalg.solve(M, b[s].reshape(N * m, r)).reshape(N, m, r)
        assert np.abs(x[s] - ref).max() <= 1e-12 * np.abs(ref).max()


def test_singular_and_capture():
    """A zero block is reported and the next solve is sound; a solve may be recorded into a graph."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(9)
    m = 40
    A = rng.standard_normal((1, 3, m, m)) + 3.0 * m * np.eye(m)
    B, C = rng.standard_normal((2, 1, 3, m, m))
    args = [torch.from_numpy(t).cuda() for t in (A, B, C, rng.standard_normal((1, 3, m, 1)))]
    want = bc.strip_solve(*args)
    zero = [args[0].clone()] + args[1:]
    zero[0][0, 0] = 0.0
    _, status = bc.strip_solve(*zero, return_status=True)
    assert status.cpu().tolist() == [1]
    out, work, st = torch.zeros_like(want), bc.strip_workspace(1, 3, m, 1, "cuda"), torch.full((1,), 7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bc.strip_solve(*args, out=out, work=work, status=st)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want) and int(st) == 0
