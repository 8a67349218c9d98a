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


@pytest.mark.parametrize("N,m,r", [(1, 40, 2), (3, 48, 1), (2, 150, 3)])
def test_a_wait_that_runs_out(N, m, r):
    """A panel that never comes: every block leaves, the status says 2, no number passes for a solution, and the next
    solve is sound."""
    args = system(2, N, m, r)
    x, status = debug_solve(*args, wait_polls=2000, withhold_panels=1)
    assert status == [2, 2] and torch.isnan(x).all()
    want, st = bc.strip_solve(*args, return_status=True)
    assert st.cpu().tolist() == [0, 0] and torch.isfinite(want).all()


def test_a_long_strip_outlasts_the_polls():
    """The panel block waits through the whole backward sweep: a limit that covers some hundred elements (4,000 polls of
    about 0.4 us) does not end a sweep of 6,000 (10 us or so each, as long as the sweep moves)."""
    args = system(1, 6000, 33, 1)
    want = bc.strip_solve(*args)
    x, status = debug_solve(*args, wait_polls=4000)
    assert status == [0] and torch.equal(x, want)


@pytest.mark.parametrize("big,small", [((1, 3, 448, 32), (1, 3, 33, 1)), ((2, 3, 32, 32), (2, 3, 30, 1))])
def test_shapes_from_two_threads(big, small):
    """Solves that want much and little shared memory, from two threads at once: every launch is accepted."""
    import threading
    args = [system(*s) for s in (big, small)]
    want = [bc.strip_solve(*a) for a in args]
    torch.cuda.synchronize()
    failed = []

    def work(i):
        try:
            st, out = torch.cuda.Stream(), torch.empty_like(want[i])
            mem = bc.strip_workspace(*args[i][3].shape, "cuda")
            status = torch.zeros(len(out), dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            for _ in range(300):
                bc.strip_solve(*args[i], out=out, work=mem, status=status, stream=st)
            st.synchronize()
            assert torch.equal(out, want[i])
        except Exception as e:
            failed.append(e)

    th = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not failed, failed


def test_memory_of_a_solve_on_another_stream():
    """What strip_solve allocates for itself is not handed out again while the solve runs on the caller's stream."""
    args = system(1, 8, 100, 1)
    want = bc.strip_solve(*args)
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    for _ in range(20):
        out = torch.empty_like(want)
        x, status = bc.strip_solve(*args, out=out, stream=st, return_status=True)
        junk = [torch.full((n,), float("nan"), device="cuda", dtype=torch.float64) for n in (64, 1 << 12, 1 << 16, 1 << 18)]
        del junk
        st.synchronize()
        assert torch.equal(x, want) and status.cpu().tolist() == [0]


@pytest.mark.parametrize("blocks,m,r", [(148, 448, 32), (148, 439, 1), (122, 448, 32), (132, 391, 5)])
def test_the_whole_range_on_fewer_blocks(blocks, m, r):
    """Four columns of a kind per block, as on a part with fewer SMs: every documented shape from 122 blocks on."""
    args = system(1, 3, m, r)
    want = bc.strip_solve(*args)
    x, status = debug_solve(*args, max_blocks=blocks)
    assert status == [0] and (x - want).abs().max() <= 1e-12 * want.abs().max()
    with pytest.raises(bc.BoxCodeError) as e:
        debug_solve(*args, max_blocks=80)
    assert e.value.status == -6
