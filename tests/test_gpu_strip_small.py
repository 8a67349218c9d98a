"""The small-block strip solve at the edges of its launch rule and of its buffers, against numpy's dense solve.

Warps per system change with m (3 m + r) (128, 400, 2200) and the number of systems; three buffers go round in the
backward sweep (N = 1 .. 6); the diagonal blocks are row-permuted, so that every pivot is off the diagonal.  Bar: 1e-12
relative max-norm, as for the other well-conditioned strips."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2501_17967_gb300 as bc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nsys,N,m,r", [(2, 1, 32, 32), (2, 2, 32, 32), (3, 3, 6, 1), (3, 4, 7, 1), (2, 5, 11, 2), (2, 6, 12, 5),
                                        (320, 4, 11, 1), (320, 3, 17, 3), (320, 2, 27, 1), (320, 3, 32, 1), (1, 6, 31, 7), (4, 5, 2, 9)])
def test_small_blocks(nsys, N, m, r):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(1000 * N + 10 * m + r)
    A = rng.standard_normal((nsys, N, m, m)) + 4.0 * m * np.eye(m)[rng.permutation(m)]
    B, C = rng.standard_normal((2, nsys, N, m, m))
    b = rng.standard_normal((nsys, N, m, r))
    x, status = bc.strip_solve(*(torch.from_numpy(t).cuda() for t in (A, B, C, b)), return_status=True)
    x = x.cpu().numpy()
    assert not status.any()
    for s in {0, nsys // 2, nsys - 1}:
        M = np.zeros((N * m, N * m))
        for k in range(N):
            for blk, j in ((A, k), (B, (k + 1) % N), (C, (k - 1) % N)):
                M[k * m:(k + 1) * m, j * m:(j + 1) * m] += blk[s, k]
        ref = np.linalg.solve(M, b[s].reshape(N * m, r)).reshape(N, m, r)
        assert np.abs(x[s] - ref).max() <= 1e-12 * np.abs(ref).max()
