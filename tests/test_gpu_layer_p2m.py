"""Sources of one leaf to its multipole: the two forms of the leaf step (coefficients
over the lanes, sources over the lanes) and the split of the sources over 16 warps, at
the source counts where either changes.  All sources sit in one corner of one leaf;
reference: the direct sum at every node of the other leaves.  Bar: the truncation bound
of the expansions, 1e-10 of max |u| at 30 terms (point sources at a box's corner
converge like 0.55^P)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2501_17967_gb300 as bc  # noqa: E402
from paper_2501_17967_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 16, 17, 127, 128, 129, 512, 513, 700])
def test_source_counts(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = bc.Context(p=16, nterms=30, device=0)
    tree = bc.Tree(ctx, *synth.uniform_leaves(3))
    rng = np.random.default_rng(n)
    src = np.array([-0.99, -0.74]) + rng.uniform(0.0, 0.23, (n, 2))   # inside the leaf [-1, -0.75] x [-0.75, -0.5]
    q, m = rng.standard_normal(n), 0.1 * rng.standard_normal((n, 2))
    u = bc.Layer(tree, src).apply(torch.from_numpy(q).cuda(), torch.from_numpy(m).cuda()).cpu().numpy().reshape(-1, 256)
    nodes = oracle.leaf_nodes(synth.leaf_geometry(*(np.asarray(a) for a in tree.leaves())), 16)
    ref = oracle.layer(src, q, m, nodes.reshape(-1, 2)).reshape(-1, 256)
    far = np.abs(nodes - src.mean(0)).max(axis=(1, 2)) > 0.5   # by expansions: two leaves and more away
    err = np.abs(u[far] - ref[far]).max() / np.abs(ref[far]).max()
    print(f"{n} sources, {far.sum()} leaves: {err:.1e}")
    assert far.sum() >= 40 and err <= 1e-10


# the L2P's tiles made by the layer itself, and the tree's after an apply: same products
@pytest.mark.parametrize("level", [0, 1, 3])
def test_before_and_after_an_apply(level):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ctx = bc.Context(p=16, nterms=30, device=0)
    tree = bc.Tree(ctx, *synth.uniform_leaves(level))
    rng = np.random.default_rng(3)
    layer = bc.Layer(tree, rng.uniform(-0.9, 0.9, (40, 2)))
    q, m = torch.from_numpy(rng.standard_normal(40)).cuda(), torch.from_numpy(rng.standard_normal((40, 2))).cuda()
    before = layer.apply(q, m)
    bc.apply(tree, torch.ones(tree.nleaf, 16, 16, device="cuda", dtype=torch.float64))
    assert torch.equal(before, layer.apply(q, m))
