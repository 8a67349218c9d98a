"""Value and gradient off the grid at every order class of the kernel (p <= 8, 12, 16), against the Chebyshev
series of the leaf interpolant in numpy: random points, points on nodes, leaf edges and the root's corners.

Bars: the basis values are sums of products of rounded factors, a few p units in the last place times the Lebesgue
constant (below 3 for p <= 16): 1e-13 of max |u|; a derivative is at most p^2 / r times that (Markov).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2501_17967_gb300 as bc  # noqa: E402
from paper_2501_17967_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [4, 7, 8, 9, 12, 13, 16])
def test_points_against_chebyshev_series(p):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = bc.Context(p=p, nterms=8, device=0)
    lv, ix, iy = synth.uniform_leaves(2)
    tree = bc.Tree(ctx, lv, ix, iy)
    rng = np.random.default_rng(p)
    u = rng.standard_normal((16, p, p))
    nodes = tree.nodes().reshape(-1, 2)
    edges = np.stack(np.meshgrid(np.linspace(-1, 1, 9), np.linspace(-1, 1, 9)), -1).reshape(-1, 2)
    xy = np.concatenate([rng.uniform(-1, 1, (701, 2)), nodes, edges, nodes[:40] + 1e-14])
    c = np.minimum(((xy + 1) * 2).astype(int), 3)
    leaf = c[:, 1] * 4 + c[:, 0]
    t = (xy - (-1 + (2 * c + 1) * 0.25)) / 0.25
    x = -np.cos((2 * np.arange(p) + 1) * np.pi / (2 * p))
    M = np.linalg.inv(np.polynomial.chebyshev.chebvander(x, p - 1))
    D = np.polynomial.chebyshev.chebder(np.eye(p))          # [p - 1, p]
    coef = np.einsum("ai,nij,bj->nab", M, u, M)[leaf]
    T = [np.polynomial.chebyshev.chebvander(t[:, d], p - 1) for d in (0, 1)]
    dT = [np.polynomial.chebyshev.chebvander(t[:, d], p - 2) @ D for d in (0, 1)]
    want = np.einsum("na,nab,nb->n", T[1], coef, T[0])
    wgrad = np.stack([np.einsum("na,nab,nb->n", T[1], coef, dT[0]), np.einsum("na,nab,nb->n", dT[1], coef, T[0])], 1) / 0.25
    ud, xd = torch.from_numpy(u).cuda(), torch.from_numpy(xy).cuda()
    val, grad = bc.eval_points_grad(tree, ud, xd)
    only = bc.eval_points(tree, ud, xd)
    big = np.abs(u).max()
    assert torch.equal(val, only)
    assert np.abs(val.cpu().numpy() - want).max() <= 1e-13 * big * 9
    assert np.abs(grad.cpu().numpy() - wgrad).max() <= 1e-13 * big * 9 * p * p / 0.25
