"""The FP64 mode's 7-digit tensor-core products against the FP64 kernels.

bc_apply (FP64) forms its operator products from 56-bit digits on the tensor
cores; bc_apply_noalloc runs the same operator on the FP64 kernels, so the two
are compared directly.  Bar: a chain of K <= 256 FP64 additions rounds at most
K 2^-53 = 2.8e-14 of the sum of its magnitudes, and a node adds up about forty
such products of which the largest dominate; 1e-13 of max |u| is the bar the
FP64 kernels are held to among themselves.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2501_17967_gb300 as bc  # noqa: E402
from paper_2501_17967_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu
BAR = 1e-13


@pytest.fixture(autouse=True)
def need_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def kernels(tree, x, adjoint):
    out = torch.empty_like(x)
    bc._check(bc._load().bc_apply_noalloc(tree.ctx.handle, tree.handle, ctypes.c_void_p(x.data_ptr()),
                                          ctypes.c_void_p(out.data_ptr()), int(adjoint), None))
    return out


def digits(tree, x, adjoint):
    return bc.apply_adjoint(tree, x) if adjoint else bc.apply(tree, x)


def make(p, nterms, kappa=0.7, max_level=6):
    ctx = bc.Context(p=p, nterms=nterms, device=0)
    tree = bc.Tree(ctx, *synth.geometric_leaves(synth.gaussians(4, 5, wlog10=(-2.0, -0.8)), kappa=kappa, max_level=max_level))
    gen = torch.Generator(device="cuda").manual_seed(p)
    x = torch.randn(tree.nleaf, p, p, generator=gen, device="cuda", dtype=torch.float64)
    return tree, x


def relerr(a, b):
    return ((a - b).abs().max() / b.abs().max()).item()


# inner dimension of the tiles: p^2 padded to 64 (p <= 8), 144 (p <= 12) or 256;
# rows: one 128-row job (p <= 11), two of which the second is short (12..15) or full (16)
@pytest.mark.parametrize("p,nterms", [(4, 4), (5, 32), (8, 24), (9, 17), (11, 30), (12, 31), (13, 8), (16, 30), (16, 32)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_orders(p, nterms, adjoint):
    tree, x = make(p, nterms)
    err = relerr(digits(tree, x, adjoint), kernels(tree, x, adjoint))
    print(f"p {p} nterms {nterms} leaves {tree.nleaf}: {err:.1e}")
    assert err <= BAR


# list lengths at the edges of a 32-column tile: 1, 4, 16, 64 leaves and a few more
@pytest.mark.parametrize("level", [0, 1, 2, 3])
@pytest.mark.parametrize("adjoint", [False, True])
def test_small_trees(level, adjoint):
    ctx = bc.Context(p=16, nterms=30, device=0)
    tree = bc.Tree(ctx, *synth.uniform_leaves(level))
    x = torch.randn(tree.nleaf, 16, 16, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(level))
    assert relerr(digits(tree, x, adjoint), kernels(tree, x, adjoint)) <= BAR


# one node of each leaf carries everything (a corner node: the smallest weight),
# leaves of very different magnitude, and the ends of the exponent range
@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("kind", ["corner", "spread", "large", "small"])
def test_magnitudes(kind, adjoint):
    tree, x = make(16, 30)
    if kind == "corner":
        x[:, 1:] *= 2.0 ** -60
        x[:, :, 1:] *= 2.0 ** -60
    elif kind == "spread":
        x *= 2.0 ** torch.linspace(-200, 200, tree.nleaf, device="cuda", dtype=torch.float64).round()[:, None, None]
    else:
        x *= 2.0 ** (900 if kind == "large" else -960)
    u, v = digits(tree, x, adjoint), kernels(tree, x, adjoint)
    assert torch.isfinite(u).all() and relerr(u, v) <= BAR
    if kind == "spread":   # leaf by leaf near the small end too
        err = ((u - v).abs().amax((1, 2)) / v.abs().amax((1, 2))).max().item()
        assert err <= BAR


@pytest.mark.parametrize("p", [8, 12, 16])
@pytest.mark.parametrize("adjoint", [False, True])
def test_results_about_the_end_of_the_normal_range(p, adjoint):
    """Products of which some entries are subnormal (a leaf's rows carry its r^2, higher coefficients are smaller):
    lanes of one epilogue warp scale their results in different ways.  The level passes lose bits there too, in
    either path: the bar is BAR above twice what the FP64 kernels lose on the same input."""
    tree, x = make(p, 24)
    u1 = kernels(tree, x, adjoint)
    top = u1.abs().max().item()
    scale = 2.0 ** (-1015 - round(np.log2(top)))
    u, v = digits(tree, x * scale, adjoint), kernels(tree, x * scale, adjoint)
    assert (u / scale - u1).abs().max().item() <= BAR * top + 2.0 * (v / scale - u1).abs().max().item()


@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_values(bad, adjoint):
    """A leaf with an infinity or a NaN has no digits: its products are formed in FP64."""
    tree, x = make(16, 24, max_level=5)
    x[3, 4, 5] = bad
    u, v = digits(tree, x, adjoint), kernels(tree, x, adjoint)
    assert torch.equal(torch.isfinite(u), torch.isfinite(v))
    assert not torch.isfinite(u).all()
    bc._check(bc._load().bc_sync(tree.ctx.handle, None))
    x[3, 4, 5] = 1.0       # nothing of it stays behind
    assert relerr(digits(tree, x, adjoint), kernels(tree, x, adjoint)) <= BAR


def test_zero_input():
    tree, x = make(12, 24, max_level=4)
    assert not digits(tree, torch.zeros_like(x), False).any()


def test_first_apply_inside_a_capture():
    """The first apply of a tree may be recorded into a graph; the replay serves new values."""
    tree, x = make(16, 24, max_level=5)
    want, y = kernels(tree, x, False), torch.zeros_like(x)
    src = torch.zeros_like(x)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bc.apply(tree, src, out=y)
    src.copy_(x)
    g.replay()
    torch.cuda.synchronize()
    assert relerr(y, want) <= BAR


@pytest.mark.parametrize("first", ["fp64", "split", "layer"])
def test_first_use_of_the_tiles_later_in_a_capture(first):
    """The 7-digit tiles of a tree made while its internal stream is part of the capture, by an earlier apply (of
    the all-tensor mode, which does not use them)."""
    tree, x = make(16, 24, max_level=5)
    y, z, src = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
    bc.apply(tree, x, out=y, precision=bc.SPLIT_BF16_ALL)
    if first == "split":       # the 5-digit tiles exist, the 7-digit M2L's do not
        fn = lambda t, v, out: bc.apply(t, v, out=out, precision=bc.SPLIT_BF16)   # noqa: E731
    elif first == "layer":
        curve = np.stack([0.5 * np.cos(np.arange(100)), 0.5 * np.sin(np.arange(100))], 1)
        m = torch.zeros(100, 2, device="cuda", dtype=torch.float64)
        fn = lambda t, v, out: layers[id(t)].apply(v.reshape(-1)[:100], m, out=out.reshape(-1))   # noqa: E731
        layers = {id(tree): bc.Layer(tree, curve)}
    else:
        fn = lambda t, v, out: bc.apply(t, v, out=out)   # noqa: E731
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bc.apply(tree, src, out=y, precision=bc.SPLIT_BF16_ALL)
        fn(tree, src, z)
    src.copy_(x)
    g.replay()
    torch.cuda.synchronize()
    want = torch.empty_like(x)
    assert torch.equal(y, bc.apply(tree, x, precision=bc.SPLIT_BF16_ALL))
    fn(tree, x, want)
    assert torch.equal(z, want)
    if first == "fp64":        # by the digits, not by the kernels that serve where they do not fit
        assert not torch.equal(z, kernels(tree, x, False)) and relerr(z, kernels(tree, x, False)) <= BAR


def test_trees_on_their_own_streams():
    """Applies of different trees of one context, from several threads and streams at once."""
    import threading
    ctx = bc.Context(p=16, nterms=24, device=0)
    leaves = synth.geometric_leaves(synth.gaussians(4, 9, wlog10=(-2.0, -0.8)), kappa=0.7, max_level=6)
    trees = [bc.Tree(ctx, *leaves) for _ in range(3)]
    xs = [torch.randn(t.nleaf, 16, 16, device="cuda", dtype=torch.float64) for t in trees]
    want = [bc.apply(t, x) for t, x in zip(trees, xs)]
    outs = [torch.empty_like(x) for x in xs]
    torch.cuda.synchronize()

    def work(i):
        st = torch.cuda.Stream()
        for _ in range(20):
            bc.apply(trees[i], xs[i], out=outs[i], stream=st)
        st.synchronize()

    th = [threading.Thread(target=work, args=(i,)) for i in range(3)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for w, o in zip(want, outs):
        assert torch.equal(w, o)
    assert np.isfinite(relerr(outs[0], want[0]))


# 256 nodes of at most 64 a leaf: the FP64 kernels serve; above, or with larger leaves, the digits
@pytest.mark.parametrize("p,level,native", [(4, 0, True), (4, 1, True), (4, 2, True), (5, 1, True), (5, 2, False), (8, 0, True),
                                            (8, 1, True), (9, 0, False), (9, 1, False), (16, 0, False), (4, 3, False)])
def test_small_trees_of_small_orders(p, level, native):
    tree = bc.Tree(bc.Context(p=p, nterms=20, device=0), *synth.uniform_leaves(level))
    x = torch.randn(tree.nleaf, p, p, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(p))
    for adjoint in (False, True):
        u, v = digits(tree, x, adjoint), kernels(tree, x, adjoint)
        assert torch.equal(u, v) if native else relerr(u, v) <= BAR
    x[0, 0, 0] = float("inf")
    assert torch.equal(torch.isfinite(digits(tree, x, False)), torch.isfinite(kernels(tree, x, False)))
    batch = bc.Batch(tree.ctx, [tree, tree])     # the union may be above the line where its trees are not
    xs = [torch.randn_like(x) for _ in range(2)]
    outs = [torch.empty_like(x) for _ in range(2)]
    batch.run(xs, outs)
    for a, u in zip(xs, outs):
        assert relerr(u, kernels(tree, a, False)) <= BAR


@pytest.mark.parametrize("p", [7, 16])
def test_native_fp64_on_request(p):
    """fp64_native: BC_FP64 on the FP64 kernels alone, bit for bit bc_apply_noalloc, without the tiles' memory."""
    tree, x = make(p, 30)
    tree.ctx.set_option("fp64_native", 1)
    for adjoint in (False, True):
        assert torch.equal(digits(tree, x, adjoint), kernels(tree, x, adjoint))
    batch = bc.Batch(tree.ctx, [tree, tree])
    outs = [torch.empty_like(x) for _ in range(2)]
    batch.run([x, x], outs)
    assert torch.equal(outs[0], kernels(tree, x, False)) and torch.equal(outs[1], outs[0])
    curve = np.stack([0.5 * np.cos(np.arange(200)), 0.5 * np.sin(np.arange(200))], 1)
    layer, q, m = bc.Layer(tree, curve), x.reshape(-1)[:200], x.reshape(-1)[200:600].reshape(200, 2)
    native = layer.apply(q, m)
    batch.close()
    split = bc.apply(tree, x, precision=bc.SPLIT_BF16) if p == 16 else None   # its M2L follows: no 7-digit tiles
    free = torch.cuda.mem_get_info()[0]
    tree.ctx.set_option("fp64_native", 0)
    if p == 16:
        assert relerr(bc.apply(tree, x, precision=bc.SPLIT_BF16), split) <= 1e-10
        assert torch.cuda.mem_get_info()[0] < free
    u = digits(tree, x, False)
    assert not torch.equal(u, kernels(tree, x, False)) and relerr(u, kernels(tree, x, False)) <= BAR
    assert relerr(layer.apply(q, m), native) <= BAR
    with pytest.raises(bc.BoxCodeError):
        tree.ctx.set_option("fp64_native", 2)


@pytest.mark.parametrize("order", [("split", "fp64"), ("fp64", "split"), ("split", "all", "fp64"), ("all", "layer", "split", "fp64")])
def test_parts_of_the_tiles_in_any_order(order):
    """A tree sets up its tiles as its calls need them (the split mode the M2L's part of the 7-digit ones only): every
    order of first use gives what a fresh tree gives."""
    curve = np.stack([0.5 * np.cos(np.arange(300)), 0.5 * np.sin(np.arange(300))], 1)

    def run(tree, x, what):
        if what == "layer":
            return bc.Layer(tree, curve).apply(x.reshape(-1)[:300], x.reshape(-1)[300:900].reshape(300, 2))
        prec = {"fp64": bc.FP64, "split": bc.SPLIT_BF16, "all": bc.SPLIT_BF16_ALL}[what]
        return torch.cat([bc.apply(tree, x, precision=prec), bc.apply_adjoint(tree, x, precision=prec)])

    tree, x = make(16, 24, max_level=5)
    for what in order + order:
        fresh, _ = make(16, 24, max_level=5)
        assert torch.equal(run(tree, x, what), run(fresh, x, what)), what
    bc._check(bc._load().bc_sync(tree.ctx.handle, None))
