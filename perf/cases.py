"""Performance cases of the box code: what a user's program has it do, over the range of sizes it is used at.

A case is a dict with a "kind":
  apply   v_bulk on one adaptive quadtree: u = A f and h = A^T g (or one of them), in one of the precision modes
  grad    the differentiable apply: forward, and the gradient of a loss through autograd
  trunc   the same applies on a truncated tree (a domain with discarded leaves)
  batch   many trees of one order in one batched run, both directions
  layer   the glue layer potential of a closed curve at every leaf node
  points  value and gradient of v_bulk off the grid
  strip   the strip's block-tridiagonal systems with periodic corners

Trees are refined here, by the paper's resolution criterion (Alg. 2) and a 2:1 balance, from Gaussian-sum densities whose
centres and widths belong to the case; the seed of `prepare` draws the amplitudes, so that one case always has the same leaves.
"""
import functools
import math

import numpy as np
import torch

import paper_2501_17967_gb300 as bc

PRECISION = {"fp64": bc.FP64, "split": bc.SPLIT_BF16, "split_all": bc.SPLIT_BF16_ALL}
DEV = "cuda"


def listed():
    return [
        # the smallest call: one apply of a coarse uniform tree, default order, terms and precision (latency of the passes)
        {"name": "apply-fp64-64", "kind": "apply", "p": 16, "nterms": 30, "precision": "fp64", "dirs": "f", "uniform": 3},
        # an ordinary solve's tree in the default precision, forward and adjoint (one step of an optimisation over f)
        {"name": "apply-fp64-700", "kind": "apply", "p": 16, "nterms": 30, "precision": "fp64", "dirs": "fa", "gaussians": 9,
         "wmin": -2.7, "tree_seed": 1},
        # the benchmark's 200-Gaussian density (widths 1e-4 .. 1e-1), default precision
        {"name": "apply-fp64-17k", "kind": "apply", "p": 16, "nterms": 30, "precision": "fp64", "dirs": "fa", "gaussians": 200,
         "wmin": -4.0, "tree_seed": 2},
        # the same in the benchmark's precision and order
        {"name": "apply-split-17k", "kind": "apply", "p": 16, "nterms": 24, "precision": "split", "dirs": "fa", "gaussians": 200,
         "wmin": -4.0, "tree_seed": 2},
        # an ordinary tree in the all-tensor mode
        {"name": "apply-split_all-700", "kind": "apply", "p": 16, "nterms": 24, "precision": "split_all", "dirs": "fa",
         "gaussians": 9, "wmin": -2.7, "tree_seed": 1},
        # gradients with respect to the density through autograd, many leaves
        {"name": "grad-split-28k", "kind": "grad", "p": 16, "nterms": 24, "precision": "split", "uniform": 7},
        # a domain: the star-shaped boundary, leaves outside it discarded
        {"name": "trunc-split-4k", "kind": "trunc", "p": 16, "nterms": 24, "precision": "split", "dirs": "fa", "gaussians": 20,
         "wmin": -3.0, "tree_seed": 1},
        # a batch of small trees of a lower order in the default precision
        {"name": "batch-fp64-12", "kind": "batch", "p": 12, "nterms": 30, "precision": "fp64", "trees": 12, "gaussians": 5,
         "wmin": -2.0, "tree_seed": 1000},
        # the glue potential of 4096 curve nodes on the large tree, default precision
        {"name": "layer-fp64-4096", "kind": "layer", "p": 16, "nterms": 30, "precision": "fp64", "gaussians": 200, "wmin": -4.0,
         "tree_seed": 2, "panels": 256},
        # v_bulk and its gradient at the curve's nodes (the jumps of the glue step) and as many again as a plot takes
        {"name": "points-100k", "kind": "points", "p": 16, "n": 100003, "gaussians": 20, "wmin": -3.0, "tree_seed": 1},
        # the paper's strip: 56 elements of 16 x 24 nodes
        {"name": "strip-56x384", "kind": "strip", "nsys": 1, "N": 56, "m": 384, "r": 1},
        # many small strips at once
        {"name": "strip-608x256x17", "kind": "strip", "nsys": 608, "N": 256, "m": 17, "r": 1},
    ]


def draw(rng):
    def logint(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["apply", "apply", "apply", "apply", "grad", "batch", "layer", "points", "strip", "strip"])
    seed = rng.randrange(1 << 20)
    if kind == "strip":
        if rng.random() < 0.5:
            m = rng.randint(2, 32)
            N = logint(2, 256)
            nsys = logint(1, max(1, int(608 * 256 * 17 ** 3 / (N * m ** 3))) if m > 3 else 2000)
            return {"kind": "strip", "nsys": min(nsys, 2000), "N": N, "m": m, "r": rng.choice([1, 1, 1, 2, 3])}
        m = rng.randint(33, 448)
        N = logint(2, max(3, min(200, int(56 * 384 * 384 / (m * m)))))
        return {"kind": "strip", "nsys": 1, "N": min(N, 56 * 384 // m), "m": m, "r": rng.choice([1, 1, 2, 5])}
    n = logint(1, 200)
    wmin = rng.uniform(-4.0, -1.2)
    if kind == "points":
        return {"kind": "points", "p": rng.choice([16, 16, 12, 8, 11]), "n": logint(100, 400000), "gaussians": min(n, 40),
                "wmin": max(wmin, -3.0), "tree_seed": seed}
    if kind == "layer":
        return {"kind": "layer", "p": 16, "nterms": 30, "precision": rng.choice(["fp64", "split"]), "gaussians": n, "wmin": wmin,
                "tree_seed": seed, "panels": logint(8, 256)}
    precision = rng.choice(["fp64", "fp64", "split", "split", "split_all"])
    p = rng.choice([16, 16, 12, 8]) if precision != "fp64" else rng.choice([16, 16, 12, 8, rng.randint(5, 15)])
    nterms = rng.choice([30, 30, 24, rng.randint(18, 32)])
    if kind == "batch":
        return {"kind": "batch", "p": p, "nterms": nterms, "precision": precision, "trees": rng.randint(2, 8 if p < 12 else 16),
                "gaussians": rng.randint(3, 8), "wmin": max(wmin, -2.0), "tree_seed": seed}
    if p < 16:
        n, wmin = min(n, 30), max(wmin, -2.5)
    case = {"kind": kind, "p": p, "nterms": nterms, "precision": precision, "gaussians": n, "wmin": wmin, "tree_seed": seed}
    if kind == "apply":
        case["dirs"] = rng.choice(["f", "a", "fa"])
    return case


# ---------------------------------------------------------------------------
# Densities, trees, curves
# ---------------------------------------------------------------------------
class Density:
    """sum_k a_k exp(-|x - c_k|^2 / (2 w_k^2)); centres and widths from the case, amplitudes from the seed."""

    def __init__(self, n, wmin, tree_seed, seed=None):
        r = np.random.default_rng(tree_seed)
        c = r.uniform(-0.5, 0.5, (n, 2))
        w = 10.0 ** r.uniform(wmin, -1.0, n)
        a = np.random.default_rng([7, seed]).standard_normal(n) if seed is not None else np.ones(n)
        self.c, self.w, self.a = (torch.tensor(v, device=DEV) for v in (c, w, a))

    def __call__(self, xy):
        out = torch.zeros(xy.shape[:-1], dtype=torch.float64, device=xy.device)
        for c, w, a in zip(self.c, self.w, self.a):
            out += a * torch.exp((xy - c).square().sum(-1) / (-2.0 * w * w))
        return out


def chebyshev(p):
    return -np.cos((2 * np.arange(p) + 1) * np.pi / (2 * p))


def cheb_matrix(p):
    """[p, p]: node values -> Chebyshev coefficients."""
    th = np.arccos(chebyshev(p))
    m = 2.0 / p * np.cos(np.outer(np.arange(p), th))
    m[0] *= 0.5
    return m


def leaf_nodes(lv, ix, iy, p):
    """[nleaf, p*p, 2] node coordinates (x fastest), on the GPU."""
    r = 1.0 / 2.0 ** lv.astype(np.float64)
    x = torch.tensor(chebyshev(p), device=DEV)
    cx, cy, r = (torch.tensor(v, device=DEV) for v in (-1 + (2 * ix + 1) * r, -1 + (2 * iy + 1) * r, r))
    X = cx[:, None, None] + r[:, None, None] * x[None, None, :].expand(1, p, p)
    Y = cy[:, None, None] + r[:, None, None] * x[None, :, None].expand(1, p, p)
    return torch.stack([X, Y], -1).reshape(len(lv), p * p, 2)


def refine(p, density, curve=None, max_level=16):
    """Leaves of Alg. 2 (function-resolution criterion) with a 2:1 balance; near a curve, boxes of half-side at most 1/32."""
    eps = max(1e-11, 10.0 ** -p)
    M = torch.tensor(cheb_matrix(p), device=DEV)
    tail = torch.zeros(p, p, dtype=torch.bool, device=DEV)
    tail[p - 2:] = True
    tail[:, p - 2:] = True
    inner = []          # keys iy * 2^lv + ix of the split boxes of each level
    ix = iy = np.zeros(1, np.int64)
    centre, width = density.c.cpu().numpy(), density.w.cpu().numpy()
    for lv in range(max_level):
        split = np.zeros(len(ix), bool)
        for s in range(0, len(ix), 4096):
            v = density(leaf_nodes(np.full(len(ix[s:s + 4096]), lv), ix[s:s + 4096], iy[s:s + 4096], p)).reshape(-1, p, p)
            coef = torch.einsum("ai,nij,bj->nab", M, v, M).abs()
            split[s:s + 4096] = (coef[:, tail].amax(1) > eps).cpu().numpy()
        # a box that its nodes say nothing about: one that holds the centre of a far narrower Gaussian, or a piece of the curve
        for at in (centre[width < 0.5 ** lv], curve if curve is not None and lv < 5 else centre[:0]):
            at = np.clip(((at + 1) / 2 * 2 ** lv).astype(np.int64), 0, 2 ** lv - 1)
            split |= np.isin(iy * 2 ** lv + ix, at[:, 1] * 2 ** lv + at[:, 0])
        inner.append(np.unique(iy[split] * 2 ** lv + ix[split]))
        if not split.any():
            break
        ix, iy = children(ix[split], iy[split])
    return balance(inner)


def children(ix, iy):
    q = np.arange(4)
    return (2 * ix[:, None] + (q & 1)).ravel(), (2 * iy[:, None] + (q >> 1)).ravel()


def balance(inner):
    """(level, ix, iy) of the leaves: touching leaves differ by at most one level."""
    inner = [np.asarray(k, np.int64) for k in inner if len(k)]
    for lv in range(len(inner), 1, -1):     # boxes of level lv are children of inner[lv - 1]
        n = 1 << (lv - 1)
        bx, by = children(inner[lv - 1] % n, inner[lv - 1] // n)
        need = []
        for dx in (-1, 0, 1):
            for dy in (-1, 0, 1):
                x, y = bx + dx, by + dy
                ok = (x >= 0) & (y >= 0) & (x < 2 * n) & (y < 2 * n)
                need.append((y[ok] >> 2) * (n >> 1) + (x[ok] >> 2))
        inner[lv - 2] = np.unique(np.concatenate([inner[lv - 2]] + need))
    out = []
    bx = by = np.zeros(1, np.int64)
    for lv in range(len(inner) + 1):
        cut = np.isin(by * (1 << lv) + bx, inner[lv]) if lv < len(inner) else np.zeros(len(bx), bool)
        out.append((np.full(int((~cut).sum()), lv), bx[~cut], by[~cut]))
        bx, by = children(bx[cut], by[cut])
    return tuple(np.concatenate(v).astype(np.int32) for v in zip(*out))


def curve(panels, q=16, k=5):
    """Gauss-Legendre panels on a star-shaped closed curve: nodes, weights, outward normals, parameter."""
    g, gw = np.polynomial.legendre.leggauss(q)
    h = 2 * math.pi / panels
    t = ((np.arange(panels)[:, None] + 0.5) * h + 0.5 * h * g).ravel()
    r, dr = 0.72 + 0.1 * np.cos(k * t), -0.1 * k * np.sin(k * t)
    xy = np.stack([r * np.cos(t), r * np.sin(t)], 1)
    d = np.stack([dr * np.cos(t) - r * np.sin(t), dr * np.sin(t) + r * np.cos(t)], 1)
    speed = np.linalg.norm(d, axis=1)
    return xy, np.tile(0.5 * h * gw, panels) * speed, np.stack([d[:, 1], -d[:, 0]], 1) / speed[:, None], t


@functools.lru_cache(maxsize=64)
def tree_leaves(p, uniform, gaussians, wmin, tree_seed, panels):
    if uniform is not None:
        n = 1 << uniform
        iy, ix = np.divmod(np.arange(n * n), n)
        if uniform < 5:
            return np.full(n * n, uniform, np.int32), ix.astype(np.int32), iy.astype(np.int32)
        low = (ix < n // 2) & (iy < n // 2)     # one quadrant a level finer
        cx, cy = children(ix[low], iy[low])
        return tuple(np.concatenate(v).astype(np.int32) for v in ((np.full((~low).sum(), uniform), np.full(len(cx), uniform + 1)),
                                                                  (ix[~low], cx), (iy[~low], cy)))
    return refine(p, Density(gaussians, wmin, tree_seed), curve(panels)[0] if panels else None)


def leaves_of(case, k=0):
    return tree_leaves(case["p"], case.get("uniform"), case.get("gaussians"), case.get("wmin"), case.get("tree_seed", 0) + k,
                       case.get("panels"))


def density_of(case, seed, k=0):
    if "uniform" in case:
        return Density(6, -1.5, 3, seed)
    return Density(case["gaussians"], case["wmin"], case["tree_seed"] + k, seed)


@functools.lru_cache(maxsize=None)
def context(p, nterms):
    """A program's one context of an order."""
    return bc.Context(p=p, nterms=nterms)


def generator(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(1000003 * k + seed)


# ---------------------------------------------------------------------------
# prepare, run, work
# ---------------------------------------------------------------------------
def tree_inputs(case, seed, leaves, k=0):
    """Leaf values of the density, and the adjoint's right-hand side."""
    p = case["p"]
    f = density_of(case, seed, k)(leaf_nodes(*leaves, p)).reshape(-1, p, p)
    return f, torch.randn(f.shape, dtype=torch.float64, device=DEV, generator=generator(seed, k + 1))


def layer_inputs(case, seed):
    xy, w, nrm, t = curve(case["panels"])
    r = np.random.default_rng([11, seed])
    mode = np.arange(1, 9)
    sigma, tau = ((r.standard_normal(8) / mode) @ np.cos(np.outer(mode, t) + r.uniform(0, 6.28, (8, 1))) for _ in range(2))
    return xy, torch.tensor(w * sigma, device=DEV), torch.tensor((w * tau)[:, None] * nrm, device=DEV)


def point_inputs(case, seed, leaves):
    p, g = case["p"], generator(seed, 2)
    a = torch.randn(3, 4, dtype=torch.float64, device=DEV, generator=g)
    xy = leaf_nodes(*leaves, p)
    u = sum(c[0] * torch.sin(3 * c[1] * xy[..., 0] + 3 * c[2] * xy[..., 1] + c[3]) for c in a)
    pts = 2 * torch.rand(case["n"], 2, dtype=torch.float64, device=DEV, generator=g) - 1
    return u.contiguous(), pts


def strip_inputs(case, seed):
    g = generator(seed, 3)
    nsys, N, m, r = case["nsys"], case["N"], case["m"], case["r"]
    A, B, C = (torch.randn(nsys, N, m, m, dtype=torch.float64, device=DEV, generator=g) for _ in range(3))
    A += 3.0 * m * torch.eye(m, dtype=torch.float64, device=DEV)
    return A, B, C, torch.randn(nsys, N, m, r, dtype=torch.float64, device=DEV, generator=g)


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "precision": PRECISION[case.get("precision", "fp64")], "dirs": case.get("dirs", "fa")}
    if kind == "strip":
        s["in"] = strip_inputs(case, seed)
        A, b = s["in"][0], s["in"][3]
        s["work"] = bc.strip_workspace(A.shape[0], A.shape[1], A.shape[2], b.shape[3], DEV)
        return s
    ctx = context(case["p"], case.get("nterms", 30))
    if kind == "batch":
        s["trees"], s["f"], s["g"] = [], [], []
        for k in range(case["trees"]):
            leaves = leaves_of(case, k)
            f, g = tree_inputs(case, seed, leaves, k)
            s["trees"].append(bc.Tree(ctx, *leaves))
            s["f"].append(f)
            s["g"].append(g)
        s["batch"] = bc.Batch(ctx, s["trees"])
        return s
    if kind == "trunc":
        t = 2 * math.pi * np.arange(600) / 600
        d = np.stack([np.cos(t), np.sin(t)], 1)
        r = (0.8 + 0.1 * np.cos(5 * t))[:, None]
        shape = Density(case["gaussians"], case["wmin"], case["tree_seed"])
        s["tree"] = bc.Tree.refine_truncated(ctx, lambda xy: shape(torch.tensor(xy, device=DEV)).cpu().numpy(), r * d,
                                             (r - 0.08) * d, eps=1e-11, max_level=16)
        mask = torch.tensor(s["tree"].node_mask(), device=DEV).reshape(-1, case["p"], case["p"])
        s["f"], s["g"] = (v * mask for v in tree_inputs(case, seed, s["tree"].leaves()))
        return s
    leaves = leaves_of(case)
    s["tree"] = bc.Tree(ctx, *leaves)
    if kind == "layer":
        xy, s["q"], s["m"] = layer_inputs(case, seed)
        s["layer"] = bc.Layer(s["tree"], xy)
    elif kind == "points":
        s["u"], s["xy"] = point_inputs(case, seed, leaves)
    else:
        s["f"], s["g"] = tree_inputs(case, seed, leaves)
    return s


def run(s):
    kind, prec = s["kind"], s["precision"]
    if kind == "strip":
        return bc.strip_solve(*s["in"], work=s["work"], return_status=True)
    if kind == "layer":
        return s["layer"].apply(s["q"], s["m"], precision=prec)
    if kind == "points":
        return bc.eval_points_grad(s["tree"], s["u"], s["xy"])
    if kind == "batch":
        us, hs = [torch.empty_like(f) for f in s["f"]], [torch.empty_like(g) for g in s["g"]]
        s["batch"].run(s["f"], us, precision=prec)
        s["batch"].run(s["g"], hs, precision=prec, adjoint=True)
        return us + hs
    if kind == "grad":
        f = s["f"].detach().requires_grad_(True)
        u = bc.BoxCodeApply.apply(f, s["tree"], prec)
        u.backward(s["g"])
        return u.detach(), f.grad
    out = []
    if "f" in s["dirs"]:
        out.append(bc.apply(s["tree"], s["f"], precision=prec))
    if "a" in s["dirs"]:
        out.append(bc.apply_adjoint(s["tree"], s["g"], precision=prec))
    return out


def work(case):
    """Inputs and outputs once; flops: each leaf's products with itself and its eight neighbours (the near field)."""
    kind = case["kind"]
    if kind == "strip":
        nsys, N, m, r = case["nsys"], case["N"], case["m"], case["r"]
        return {"bytes": 8.0 * nsys * N * (3 * m * m + 2 * m * r), "flops": float(nsys * N) * m * m * (14 * m / 3 + 6 * (r + m))}
    NP = case["p"] ** 2
    if kind == "trunc":
        nleaf = 4441    # of the star-shaped domain's tree
    else:
        nleaf = sum(len(leaves_of(case, k)[0]) for k in range(case.get("trees", 1)))
    if kind == "points":
        return {"bytes": 8.0 * (min(nleaf, case["n"]) * NP + 5 * case["n"]), "flops": 8.0 * NP * case["n"]}
    if kind == "layer":
        n = 16 * case["panels"]
        return {"bytes": 8.0 * (nleaf * NP + 5 * n), "flops": 4.0 * case["nterms"] * nleaf * NP}
    d = len(case.get("dirs", "fa"))
    return {"bytes": 16.0 * nleaf * NP * d, "flops": 18.0 * nleaf * NP * NP * d}


# ---------------------------------------------------------------------------
# The same in 64 bits by direct quadrature and plain elimination
# ---------------------------------------------------------------------------
def lagrange(p, y):
    """[..., p]: the Lagrange basis of the Chebyshev nodes at y."""
    k = torch.arange(p, device=DEV, dtype=torch.float64)
    T = torch.cos(k * torch.arccos(y.clamp(-1, 1))[..., None])
    return T @ torch.tensor(cheb_matrix(p), device=DEV)


def gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.tensor(x, device=DEV), torch.tensor(w, device=DEV)


def graded(p, x, levels=24, n=20):
    """1-D rule on [-1, 1] graded towards clip(x) (x: [m]): points [m, q] and weights times the Lagrange basis [m, q, p]."""
    g, w = gauss(n)
    c = x.clamp(-1, 1)
    edge = torch.cat([torch.zeros(1, dtype=torch.float64, device=DEV), 2.0 ** torch.arange(-levels, 1, device=DEV, dtype=torch.float64)])
    mid, half = (edge[1:] + edge[:-1]) / 2, (edge[1:] - edge[:-1]) / 2
    s = (mid[:, None] + half[:, None] * g).ravel()
    ws = (half[:, None] * w).ravel()
    up, lo = (1 - c)[:, None], (1 + c)[:, None]
    y = torch.cat([c[:, None] + up * s, c[:, None] - lo * s], 1)
    return y, torch.cat([up * ws, lo * ws], 1)[..., None] * lagrange(p, y)


@functools.lru_cache(maxsize=256)
def near_block(p, gx, gy, rho):
    """[p*p targets, p*p]: int log|x_i - y| L_k(y) dy over [-1, 1]^2 for x_i = g + rho * node."""
    t = torch.tensor(chebyshev(p), device=DEV)
    X, Y = gx + rho * t, gy + rho * t
    (yx, wx), (yy, wy) = graded(p, X), graded(p, Y)
    rows = []
    for j in range(p):
        d2 = (X[:, None, None] - yx[:, None, :]).square() + (Y[j] - yy[j])[None, :, None].square()
        rows.append(torch.einsum("iab,ak,ibl->ikl", 0.5 * torch.log(d2), wy[j], wx).reshape(p, p * p))
    return torch.cat(rows, 0)


def exact_apply(case, leaves, f, g):
    """(A f, A^T g) by quadrature leaf pair by leaf pair: graded rules for touching leaves, 24 or p + 8 Gauss points beyond."""
    p, NP = case["p"], case["p"] ** 2
    lv, ix, iy = (v.astype(np.int64) for v in leaves)
    n = len(lv)
    r = 1.0 / 2.0 ** lv
    cx, cy = -1 + (2 * ix + 1) * r, -1 + (2 * iy + 1) * r
    xy = leaf_nodes(*leaves, p)
    f, g = f.reshape(n, NP), g.reshape(n, NP)
    u, h = torch.zeros_like(f), torch.zeros_like(f)
    dist = np.maximum(abs(cx[:, None] - cx), abs(cy[:, None] - cy))     # [target, source]
    touch = dist < (r[:, None] + r) * (1 + 1e-9)
    close = (dist < 9 * r + r[:, None]) & ~touch
    rd = torch.tensor(r, device=DEV)
    rules = []
    for q in (24, max(p - 1, 8)):
        x, w = gauss(q)
        up = torch.einsum("a,b,ak,bl->abkl", w, w, lagrange(p, x), lagrange(p, x)).reshape(q * q, NP)
        pts = torch.stack(torch.meshgrid(x, x, indexing="ij")[::-1], -1).reshape(-1, 2)
        c = torch.tensor(np.stack([cx, cy], 1), device=DEV)
        rules.append((c[:, None] + rd[:, None, None] * pts, (f @ up.T) * rd[:, None] ** 2, torch.zeros(n, q * q, dtype=torch.float64, device=DEV), up))
    wsum = rules[0][3].sum(0)      # integrals of the basis
    for t in range(n):
        for (pts, rho, hq, _), sel in zip(rules, (close[t], ~close[t] & ~touch[t])):
            src = torch.tensor(np.nonzero(sel)[0], device=DEV)
            for s in src.split(4096) if len(src) else ():
                y = pts[s].reshape(-1, 2)
                lg = 0.5 * torch.log((xy[t, :, None, 0] - y[:, 0]).square() + (xy[t, :, None, 1] - y[:, 1]).square())
                u[t] += lg @ rho[s].reshape(-1)
                hq[s] += (g[t] @ lg).reshape(len(s), -1)
        for s in np.nonzero(touch[t])[0]:
            T = near_block(p, float((cx[t] - cx[s]) / r[s]), float((cy[t] - cy[s]) / r[s]), float(r[t] / r[s]))
            T = r[s] ** 2 * (T + math.log(r[s]) * wsum)
            u[t] += T @ f[s]
            h[s] += g[t] @ T
    for _, _, hq, up in rules:
        h += rd[:, None] ** 2 * (hq @ up)
    return u.reshape(n, p, p) / (2 * math.pi), h.reshape(n, p, p) / (2 * math.pi)


def exact_layer(case, seed, leaves):
    xy, q, m = layer_inputs(case, seed)
    y, x = torch.tensor(xy, device=DEV), leaf_nodes(*leaves, case["p"]).reshape(-1, 2)
    out = torch.empty(len(x), dtype=torch.float64, device=DEV)
    for s in range(0, len(x), 32768):
        dx, dy = x[s:s + 32768, None, 0] - y[:, 0], x[s:s + 32768, None, 1] - y[:, 1]
        d2 = dx * dx + dy * dy
        out[s:s + 32768] = 0.5 * (torch.log(d2) @ q) + (dx / d2) @ m[:, 0] + (dy / d2) @ m[:, 1]
    return out / (-2 * math.pi)


def exact_points(case, seed, leaves):
    p = case["p"]
    u, pts = point_inputs(case, seed, leaves)
    lv, ix, iy = (v.astype(np.int64) for v in leaves)
    at, where = pts.cpu().numpy(), np.full(len(pts), -1)
    for l in np.unique(lv):
        sel = np.nonzero(lv == l)[0]
        key = iy[sel] * (1 << l) + ix[sel]
        order = np.argsort(key)
        c = np.minimum(((at + 1) / 2 * (1 << l)).astype(np.int64), (1 << l) - 1)
        want = c[:, 1] * (1 << l) + c[:, 0]
        pos = np.minimum(np.searchsorted(key[order], want), len(key) - 1)
        hit = key[order][pos] == want
        where[hit] = sel[order][pos[hit]]
    r = 1.0 / 2.0 ** lv[where]
    x = torch.tensor((at[:, 0] - (-1 + (2 * ix[where] + 1) * r)) / r, device=DEV)
    y = torch.tensor((at[:, 1] - (-1 + (2 * iy[where] + 1) * r)) / r, device=DEV)
    M = torch.tensor(cheb_matrix(p), device=DEV)
    coef = torch.einsum("ai,nij,bj->nab", M, u.reshape(-1, p, p), M)[torch.tensor(where, device=DEV)]    # [n, y, x]

    def basis(t):
        T, D = [torch.ones_like(t), t], [torch.zeros_like(t), torch.ones_like(t)]
        for _ in range(2, p):
            T.append(2 * t * T[-1] - T[-2])
            D.append(2 * T[-2] + 2 * t * D[-1] - D[-2])
        return torch.stack(T[:p], 1), torch.stack(D[:p], 1)

    (Tx, Dx), (Ty, Dy) = basis(x), basis(y)
    rr = torch.tensor(r, device=DEV)
    val = torch.einsum("na,nab,nb->n", Ty, coef, Tx)
    return val, torch.stack([torch.einsum("na,nab,nb->n", Ty, coef, Dx) / rr, torch.einsum("na,nab,nb->n", Dy, coef, Tx) / rr], 1)


def exact_strip(case, seed):
    A, B, C, b = strip_inputs(case, seed)
    N, m, r = case["N"], case["m"], case["r"]
    if N < 3:
        D = torch.zeros(len(A), N * m, N * m, dtype=torch.float64, device=DEV)
        for k in range(N):
            for blk, j in ((A, k), (B, (k + 1) % N), (C, (k - 1) % N)):
                D[:, k * m:(k + 1) * m, j * m:(j + 1) * m] += blk[:, k]
        return torch.linalg.solve(D, b.reshape(len(b), N * m, r)).reshape(b.shape), None
    # the corner blocks as a border: block N - 1 last
    lus, H = [], []
    for k in range(N - 1):
        D = A[:, k] - (C[:, k] @ H[-1] if k else 0)
        lus.append(torch.linalg.lu_factor(D))
        H.append(torch.linalg.lu_solve(*lus[-1], B[:, k]))

    def inner(rhs):
        g = []
        for k in range(N - 1):
            g.append(torch.linalg.lu_solve(*lus[k], rhs[:, k] - (C[:, k] @ g[-1] if k else 0)))
        for k in range(N - 3, -1, -1):
            g[k] = g[k] - H[k] @ g[k + 1]
        return torch.stack(g, 1)

    E = torch.zeros_like(A[:, :N - 1])
    E[:, 0] += C[:, 0]
    E[:, N - 2] += B[:, N - 2]
    Z = inner(E)
    S = torch.linalg.lu_factor(A[:, N - 1] - B[:, N - 1] @ Z[:, 0] - C[:, N - 1] @ Z[:, N - 2])

    def solve(rhs):
        y = inner(rhs[:, :N - 1])
        last = torch.linalg.lu_solve(*S, rhs[:, N - 1] - B[:, N - 1] @ y[:, 0] - C[:, N - 1] @ y[:, N - 2])
        return torch.cat([y - Z @ last[:, None], last[:, None]], 1)

    x = solve(b)
    res = b - (A @ x + B @ x.roll(-1, 1) + C @ x.roll(1, 1))
    return x + solve(res), None


def exact(case, seed):
    kind = case["kind"]
    if kind == "strip":
        return exact_strip(case, seed)
    if kind == "trunc":
        return None
    p = case["p"]
    n = [len(leaves_of(case, k)[0]) for k in range(case.get("trees", 1))]
    if kind == "layer":
        return exact_layer(case, seed, leaves_of(case)) if n[0] * p * p * case["panels"] * 16 < 4e10 else None
    if kind == "points":
        return exact_points(case, seed, leaves_of(case))
    both, room = [], 6e10
    for k in range(case.get("trees", 1)):
        room -= n[k] ** 2 * p ** 4
        if room < 0:    # too many pairs of nodes: no value for this tree
            both.append((None, None))
            continue
        leaves = leaves_of(case, k)
        both.append(exact_apply(case, leaves, *tree_inputs(case, seed, leaves, k)))
    if all(u is None for u, _ in both):
        return None
    if kind == "batch":
        return [b[0] for b in both] + [b[1] for b in both]
    u, h = both[0]
    if kind == "grad":
        return u, h
    return [v for d, v in (("f", u), ("a", h)) if d in case["dirs"]]
