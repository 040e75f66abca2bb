"""The work a user of this framework has it do, as cases to measure: CLR products over the block
structures and precisions the framework is configured for, building CLR matrices, the Newton-Schulz
S^-1/2 iteration, the adjoints, batched products in one graph, and matrix-vector products.

Matrices (synthetic, the constructions of the workloads this repository runs; N and the jitter from
the case and the seed):
  chain    overlap-like 1D chain, S_ij = exp(-(r_i - r_j)^2 / 2) + 1e-3 delta_ij, clusters of
           96..160 points (48..256 in a batch): block sparse, low-rank neighbours
  lattice  overlap-like jittered 3D lattice, 16 points per site, exp(-r^2 / 1.5) + 1e-2 delta_ij,
           clusters of 64..256 points by bisection
  coulomb  erf(r)/r + 2e-2 delta_ij on the same lattice: no zero block, only low rank ones
  dense    i.i.d. normal entries, every block dense
"""
import math

import numpy as np
import torch

from paper_1509_00309_gb300 import autograd, clr

# stored doubles of S (fraction of N^2, N the case's size) and algorithmic flops of the tile
# products of S S (per N^3), measured on the listed sizes; they fall with N as the band or the
# far field grows, by the powers below
_MODEL = {  # matrix: (stored / N^2, product flops / N^3, stored of the product / N^2, at N, power)
    "chain": (0.0781, 0.0103, 0.0800, 2048, 1.0),
    "lattice": (0.5231, 0.2843, 0.5797, 4096, 0.5),
    "coulomb": (0.5665, 0.3430, 0.5263, 2048, 0.3),
    "dense": (1.0, 2.0, 1.0, 4096, 0.0),
}


def listed():
    return [
        # one matrix-vector product with a compressed matrix: what a Krylov or power iteration
        # around the framework (its own estimate of the Newton-Schulz scale) repeats
        dict(name="matvec_lattice_4096", kind="matvec", matrix="lattice", shape="8x8x4", eps=1e-6),
        # the smallest product in use (the smoke check's): launches and latency
        dict(name="product_chain_512", kind="product", matrix="chain", n=512, eps=1e-8,
             precision="fp64", retest=False),
        # the 1D-chain product the framework is configured with first
        dict(name="product_chain_2048", kind="product", matrix="chain", n=2048, eps=1e-8,
             precision="fp64", retest=False),
        # one product inside Newton-Schulz on the 3D lattice: FP64-accurate tensor-core tiles,
        # dense tiles re-tested for low rank
        dict(name="product_lattice_4096_ozaki", kind="product", matrix="lattice", shape="8x8x4",
             eps=1e-8, precision="ozaki", retest=True),
        # a product without block sparsity, in plain FP64
        dict(name="product_coulomb_2048_fp64", kind="product", matrix="coulomb", shape="8x4x4",
             eps=1e-6, precision="fp64", retest=True),
        # the benchmark's default: all blocks dense, split precision (the largest)
        dict(name="product_dense_16384_bf16x3", kind="product", matrix="dense", n=16384, eps=0.0,
             precision="bf16x3", retest=False),
        # all blocks dense at FP64 accuracy, an odd size
        dict(name="product_dense_4099_ozaki", kind="product", matrix="dense", n=4099, eps=0.0,
             precision="ozaki", retest=False),
        # bringing a dense matrix into CLR form, and back out
        dict(name="build_lattice_4096", kind="build", matrix="lattice", shape="8x8x4", eps=1e-6),
        # a differentiable product of dense tensors: forward and both gradients
        dict(name="grad_chain_1024", kind="grad", matrix="chain", n=1024, eps=1e-8,
             precision="fp64"),
        # the first five Newton-Schulz iterations on the lattice, a fixed number as the rank
        # distribution of the 5th iteration's matrices takes them: the iterates fill in
        dict(name="ns_lattice_2048_ozaki", kind="ns", matrix="lattice", shape="8x4x4", eps=1e-8,
             precision="ozaki", retest=True, iters=5),
        # a whole differentiable S^-1/2 to the stated error: forward with its tape and the gradient
        dict(name="ns_grad_chain_512", kind="ns_grad", matrix="chain", n=512, eps=1e-8,
             precision="fp64"),
        # independent chain products of uneven size replayed as one graph
        dict(name="batch_chain_12", kind="batch", matrix="chain", count=12, lo=1024, hi=3072,
             precision="auto"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "product", "product", "product", "product", "build", "grad", "ns",
                       "ns_grad", "batch"])
    shapes = ["4x4x2", "4x4x3", "5x4x3", "4x4x4", "6x4x3", "5x5x3", "6x4x4", "8x4x4", "7x5x4",
              "6x6x4", "8x5x4", "8x6x4", "7x7x4", "8x8x4"]
    fp = rng.choice(["fp64", "ozaki", "auto"])
    if kind == "product":
        matrix = rng.choice(["chain", "lattice", "coulomb", "dense"])
        if matrix == "dense":
            prec = rng.choice(["bf16x3", "bf16x6", "ozaki"])
            n = _log_int(rng, 500, {"bf16x3": 16384, "bf16x6": 9000, "ozaki": 5000}[prec])
            return dict(kind=kind, matrix=matrix, n=n, eps=0.0, precision=prec, retest=False)
        if matrix == "chain":
            return dict(kind=kind, matrix=matrix, n=_log_int(rng, 400, 6000),
                        eps=rng.choice([1e-6, 1e-8]), precision=fp, retest=False)
        prec = rng.choice(["fp64", "ozaki"])
        top = len(shapes) if prec == "ozaki" else 8
        return dict(kind=kind, matrix=matrix, shape=shapes[rng.randrange(2, top)],
                    eps=rng.choice([1e-6, 1e-8]), precision=prec, retest=rng.random() < 0.7)
    if kind in ("matvec", "build"):
        matrix = rng.choice(["chain", "lattice", "coulomb"])
        eps = rng.choice([1e-6, 1e-8])
        if matrix == "chain":
            return dict(kind=kind, matrix=matrix, n=_log_int(rng, 400, 6000), eps=eps)
        return dict(kind=kind, matrix=matrix, shape=rng.choice(shapes), eps=eps)
    if kind == "grad":
        return dict(kind=kind, matrix="chain", n=_log_int(rng, 400, 2048),
                    eps=rng.choice([1e-6, 1e-8]), precision=rng.choice(["fp64", "ozaki"]))
    if kind == "ns":
        return dict(kind=kind, matrix="lattice", shape=shapes[rng.randrange(0, 8)], eps=1e-8,
                    precision=rng.choice(["fp64", "ozaki"]) if rng.random() < 0.5 else "ozaki",
                    retest=True, iters=rng.randint(2, 5))
    if kind == "ns_grad":
        return dict(kind=kind, matrix="chain", n=_log_int(rng, 300, 800), eps=1e-8,
                    precision=rng.choice(["fp64", "ozaki"]))
    return dict(kind=kind, matrix="chain", count=rng.randint(4, 12), lo=1024,
                hi=rng.randint(1200, 3072), precision=rng.choice(["fp64", "auto"]))


# ---- inputs ----------------------------------------------------------------------------------

def _uneven(rng, n, lo, hi):
    """Uneven clusters of about (lo + hi) / 2 points that sum to n."""
    count = max(1, round(n / (0.5 * (lo + hi))))
    raw = rng.integers(lo, hi + 1, size=count).astype(np.float64)
    sizes = np.maximum(1, np.floor(raw * (n / raw.sum()))).astype(int)
    for i in range(n - int(sizes.sum())):
        sizes[i % count] += 1
    return [int(s) for s in sizes]


def _runs(rng, n, lo, hi):
    """Contiguous clusters of lo..hi points until n are covered; a short rest joins its neighbour
    (split into halves where the two together exceed hi)."""
    sizes, left = [], n
    while left > 0:
        sizes.append(min(int(rng.integers(lo, hi + 1)), left))
        left -= sizes[-1]
    if len(sizes) > 1 and sizes[-1] < lo // 2:
        both = sizes.pop() + sizes.pop()
        sizes += [both] if both <= hi else [both // 2, both - both // 2]
    return sizes


def _bisect(rng, sites, lo, hi):
    """Spatial groups of lo..hi sites, cut across their widest axis at a random fraction."""
    out, todo = [], [np.arange(len(sites))]
    while todo:
        idx = todo.pop()
        if len(idx) <= hi:
            out.append(idx)
            continue
        axis = int(np.argmax(sites[idx].max(0) - sites[idx].min(0)))
        idx = idx[np.argsort(sites[idx, axis], kind="stable")]
        cut = min(max(int(round(rng.uniform(0.35, 0.65) * len(idx))), lo), len(idx) - lo)
        todo += [idx[cut:], idx[:cut]]
    return out


def _sites(case):
    nx, ny, nz = (int(x) for x in case["shape"].split("x"))
    g = np.stack(np.meshgrid(np.arange(nx), np.arange(ny), np.arange(nz), indexing="ij"), -1)
    return 0.5 * g.reshape(-1, 3).astype(np.float64)


def _size(case):
    return case["n"] if "n" in case else 16 * len(_sites(case))


def _gauss(points, width, shift):
    """exp(-|r_i - r_j|^2 / width) + shift delta_ij in float64 on the GPU."""
    p = torch.from_numpy(points).cuda()
    s = torch.zeros((len(points), len(points)), dtype=torch.float64, device="cuda")
    for ax in range(p.shape[1]):
        s += (p[:, None, ax] - p[None, :, ax]) ** 2
    s.mul_(-1.0 / width).exp_()
    s.diagonal().add_(shift)
    return s


def _chain(rng, n, spacing):
    r = spacing * np.arange(n, dtype=np.float64) + rng.uniform(-0.05, 0.05, size=n)
    return _gauss(r.reshape(n, 1), 2.0, 1e-3)


def _matrix(case, seed):
    """(S as a float64 GPU tensor, cluster sizes) of the case."""
    rng = np.random.default_rng(seed)
    if case["matrix"] == "chain":
        return _chain(rng, case["n"], 0.3), _uneven(rng, case["n"], 96, 160)
    sites = _sites(case)
    points = np.repeat(sites, 16, axis=0) + rng.uniform(-0.1, 0.1, size=(16 * len(sites), 3))
    groups = _bisect(rng, points.reshape(-1, 16, 3).mean(axis=1), 4, 16)
    order = np.concatenate([(16 * g[:, None] + np.arange(16)).ravel() for g in groups])
    points, sizes = points[order], [16 * len(g) for g in groups]
    if case["matrix"] == "lattice":
        return _gauss(points, 1.5, 1e-2), sizes
    p = torch.from_numpy(points).cuda()
    d = torch.zeros((len(points), len(points)), dtype=torch.float64, device="cuda")
    for ax in range(3):
        d += (p[:, None, ax] - p[None, :, ax]) ** 2
    d.sqrt_()
    s = torch.erf(d) / d
    s.diagonal().fill_(2.0 / math.sqrt(math.pi) + 2e-2)
    return s, sizes


def _normal(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


def _dense_pair(case, seed):
    n = case["n"]
    sizes = _uneven(np.random.default_rng(seed), n, 128, 224)
    return _normal((n, n), 2 * seed + 1), _normal((n, n), 2 * seed + 2), sizes


def _batch_sizes(case):
    """Uneven sizes over lo..hi in no order."""
    k, lo, hi = case["count"], case["lo"], case["hi"]
    return [lo + ((hi - lo) * ((7 * i) % k) + i * (hi - lo) // (k + 1)) // k for i in range(k)]


def _batch(case, seed):
    """[(S, sizes, eps)] of the batch."""
    rng = np.random.default_rng(seed)
    out = []
    for i, n in enumerate(_batch_sizes(case)):
        sizes = _runs(rng, n, 48, 256)
        out.append((_chain(rng, n, float(rng.uniform(0.2, 0.6))), sizes, (1e-6, 1e-8)[i % 2]))
    return out


# ---- the calls -------------------------------------------------------------------------------

_DROP = {"chain": 1e-12, "lattice": 1e-10, "coulomb": 1e-10, "dense": 0.0}


def prepare(case, seed):
    kind, matrix = case["kind"], case["matrix"]
    opts = dict(eps_lr=case.get("eps", 1e-8), precision=case.get("precision", "fp64"),
                recompress_dense=int(case.get("retest", False)),
                eps_sp=1e-13 if matrix in ("lattice", "coulomb") else 0.0)
    if kind in ("ns", "ns_grad"):  # a fixed number of iterations, or to the stated error
        opts.update(ns_tol=0.0 if "iters" in case else 1e-6, ns_max_iter=case.get("iters", 40))
    ctx = clr.Context(0, **opts)
    st = {"kind": kind, "ctx": ctx}
    if kind == "batch":
        mats = [(ctx.from_dense(s, sizes, eps_lr=eps, drop_norm=1e-12), eps)
                for s, sizes, eps in _batch(case, seed)]
        hs = [m for m, _ in mats]
        st["batch"] = ctx.batch(hs, hs, eps=[e for _, e in mats], tune=False)
        st["c"] = [st["batch"].output(i) for i in range(len(hs))]
        st["out"] = [torch.empty(m.shape, dtype=torch.float64, device="cuda") for m in hs]
        return st
    if matrix == "dense":
        a, b, sizes = _dense_pair(case, seed)
        st["a"], st["b"] = ctx.from_dense(a, sizes), ctx.from_dense(b, sizes)
    else:
        s, sizes = _matrix(case, seed)
        if kind in ("build", "grad", "ns_grad"):
            st["s"], st["sizes"] = s, sizes
        else:
            # iterates of Newton-Schulz on the lattice start from S built at 1e-6
            eps = 1e-6 if kind in ("product", "ns") and matrix == "lattice" else case["eps"]
            st["a"] = st["b"] = ctx.from_dense(s, sizes, eps_lr=eps, drop_norm=_DROP[matrix])
    n = sum(sizes)
    if kind == "matvec":
        st["x"] = _normal((n,), seed)
        st["y"] = torch.empty_like(st["x"])
        return st
    if kind == "product":
        st["c"] = ctx.zeros(sizes)
    if kind == "build":
        st["eps"], st["drop"] = case["eps"], _DROP[matrix]
    if kind in ("grad", "ns_grad"):
        st["eps"] = case["eps"]
        st["w"] = _normal((n, n), seed)
        st["s"].requires_grad_(True)
        if kind == "ns_grad":
            st["w"] = 0.5 * (st["w"] + st["w"].T)
        else:
            st["t"] = st["s"].detach().clone().requires_grad_(True)
    else:
        st["out"] = torch.empty((n, n), dtype=torch.float64, device="cuda")
    return st


def run(state):
    kind, ctx = state["kind"], state["ctx"]
    if kind == "matvec":
        ctx.matvec(state["a"], state["x"], state["y"])
        return state["y"]
    if kind == "product":
        ctx.multiply_into(state["a"], state["b"], state["c"])
        return state["c"].to_dense(state["out"])
    if kind == "build":
        state["m"] = ctx.from_dense(state["s"], state["sizes"], eps_lr=state["eps"],
                                    drop_norm=state["drop"])
        return state["m"].to_dense(state["out"])
    if kind == "grad":
        a, b = state["s"], state["t"]
        c = autograd.multiply(a, b, ctx, state["sizes"], eps_lr=state["eps"])
        ga, gb = torch.autograd.grad(c, (a, b), state["w"])
        return c.detach(), ga, gb
    if kind == "ns":
        state["z"], _, _ = ctx.sqrt_inv(state["a"])
        return state["z"].to_dense(state["out"])
    if kind == "ns_grad":
        z = autograd.sqrt_inv(state["s"], ctx, state["sizes"], eps_lr=state["eps"],
                              drop_norm=1e-12)
        (g,) = torch.autograd.grad(z, state["s"], state["w"])
        return z.detach(), g
    state["batch"].run()
    return [c.to_dense(o) for c, o in zip(state["c"], state["out"])]


# ---- what a pass cannot do without -----------------------------------------------------------

def _model(case, n):
    """(doubles of S, flops of S S, doubles of S S) at size n."""
    s, f, c, at, power = _MODEL[case["matrix"]]
    k = min(1.0 / max(s, c), (at / n) ** power)
    return s * k * n * n, f * k * k * float(n) ** 3, min(1.0, c * k) * n * n


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        parts = [_model(case, n) for n in sizes]
        return {"bytes": 8.0 * sum(s + n * n for (s, _, _), n in zip(parts, sizes)),
                "flops": sum(f for _, f, _ in parts)}
    n = _size(case)
    s, f, c = _model(case, n)
    if kind == "matvec":
        return {"bytes": 8.0 * (s + 2 * n), "flops": 2.0 * s}
    if kind == "build":   # the matrix in and its reconstruction out; one pass of reductions
        return {"bytes": 16.0 * n * n, "flops": 2.0 * n * n}
    if kind == "product":  # the operands in, the dense result out
        return {"bytes": 8.0 * (s * (2 if case["matrix"] == "dense" else 1) + n * n), "flops": f}
    if kind == "grad":     # A, B and the cotangent in; the product and both gradients out
        return {"bytes": 48.0 * n * n, "flops": 3 * f}
    if kind == "ns":       # four products an iteration, one more X and two for the residual
        return {"bytes": 8.0 * (s + n * n), "flops": (4 * case["iters"] + 3) * f}
    # about ten iterations of four products, and of ten adjoint products
    return {"bytes": 32.0 * n * n, "flops": 10 * (4 + 10) * f}


# ---- the same in 64 bits ---------------------------------------------------------------------

def _iterate(s, steps):
    """sqrt(alpha) Z after so many steps of the coupled iteration, alpha = 1 / (1.01 lambda) with
    the Rayleigh quotient after 30 power iterations from the vector of ones."""
    n = s.shape[0]
    v = torch.full((n,), 1.0 / math.sqrt(n), dtype=torch.float64, device=s.device)
    for _ in range(30):
        v = s @ v
        v /= v.norm()
    alpha = 1.0 / (1.01 * float(v @ (s @ v)))
    eye = torch.eye(n, dtype=torch.float64, device=s.device)
    y, z = s, eye
    for _ in range(steps):
        x = alpha * (y @ z)
        t = (15.0 * eye - 10.0 * x + 3.0 * (x @ x)) / 8.0
        y, z = t @ y, z @ t
    return math.sqrt(alpha) * z


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [s @ s for s, _, _ in _batch(case, seed)]
    if case["matrix"] == "dense":
        a, b, _ = _dense_pair(case, seed)
        return a @ b
    s, _ = _matrix(case, seed)
    n = s.shape[0]
    if kind == "matvec":
        return s @ _normal((n,), seed)
    if kind == "build":
        return s
    if kind == "product":
        return s @ s
    if kind == "grad":
        w = _normal((n, n), seed)
        return s @ s, w @ s.T, s.T @ w
    if kind == "ns":
        return _iterate(s, case["iters"])
    lam, v = np.linalg.eigh(s.cpu().numpy())
    z = (v / np.sqrt(lam)) @ v.T
    # gradient of <W, S^-1/2>: V (F o (V^T W V)) V^T with the divided differences of x^-1/2
    w = _normal((n, n), seed).cpu().numpy()
    w = 0.5 * (w + w.T)
    r = np.sqrt(lam)
    f = -1.0 / (r[:, None] * r[None, :] * (r[:, None] + r[None, :]))
    return z, v @ (f * (v.T @ w @ v)) @ v.T
