"""What is measured: calls of the factorization library as its users make them.

A case names a recipe of points (`points`: the distributions of the library's workloads), the sizes
and what is done with them (`do`):

  product    build the factor of a new point set and apply it to a block of columns
  apply      apply a factor that the program keeps (one iteration of an iterative solver)
  gradient   build, apply, and the gradients with respect to the points, the lengthscale and the
             columns: one step of a program that fits points or lengthscales
  solve      build and solve (lambda I + K) X = B: Gaussian-process regression on a new data set
  cross      build K(X, Y) of two point sets, apply it and its transpose
  batch      build and apply many ragged sets at once
  regress    kernel ridge regression: cluster, assemble, solve by conjugate gradients, predict
"""
import math

import numpy as np
import torch

from paper_2202_03655_gb300 import hdf

DEV = "cuda"

# points -> (d, kernel, lengthscale, tolerance, columns of U at that tolerance)
RECIPES = {
    "ball3": (3, "gaussian", 0.5, 1e-6, 429),             # uniform in the unit ball
    "mixture3": (3, "matern32", 1.0, 1e-8, 9876),         # 8 isotropic Gaussian clusters
    "normal5": (5, "cauchy", 2.0, 1e-4, 78263),           # rotated normal, standardised
    "cube4": (4, "gaussian", 0.8, 1e-6, 2085),            # uniform in [-1, 1]^4
    "unit3": (3, "cauchy", 1.0, 1e-3, 29),                # normal, largest norm 1, d = 3 .. 6
    "unit4": (4, "cauchy", 1.0, 1e-3, 69),
    "unit5": (5, "cauchy", 1.0, 1e-3, 125),
    "unit6": (6, "cauchy", 1.0, 1e-3, 405),
    "rank5_cauchy": (5, "cauchy", 1.0, 1e-4, 1071),       # the same points, d = 5, tighter tolerances
    "rank5_gaussian": (5, "gaussian", math.sqrt(0.5), 1e-6, 786),
    "rank5_matern32": (5, "matern32", 1.0, 1e-3, 6195),
    "rank5_matern52": (5, "matern52", 1.0, 1e-5, 21687),
    "two_sets": (3, "gaussian", 1.5, 1e-6, 499),          # the clusters against a wider normal cloud
    "balls": (3, "gaussian", 0.9, 1e-6, 480),             # ragged balls of radius 0.5 .. 2, l = 0.3 .. 1.5
    "features8": (8, "gaussian", 0.5, 1e-3, 300),         # 24 anisotropic clusters scaled to [0, 1]
}


def listed():
    return [
        # the default call on a small data set: double precision, one vector; fixed costs count
        dict(name="small_product_f64", do="product", points="ball3", n=2000, cols=1, precision="fp64"),
        # the headline workload: a million points, 64 columns, single precision bulk
        dict(name="large_product", do="product", points="mixture3", n=1_000_000, cols=64, precision="fp32"),
        # the same data in double precision, a tenth of the points
        dict(name="large_product_f64", do="product", points="mixture3", n=100_000, cols=64, precision="fp64"),
        # one step of fitting points and lengthscale
        dict(name="gradient", do="gradient", points="cube4", n=500_000, cols=1, precision="fp32"),
        # regression on a new data set of ordinary size, direct solve
        dict(name="solve", do="solve", points="cube4", n=200_003, cols=1, precision="fp32"),
        # one iteration of an iterative solver with a kept factor
        dict(name="apply_one", do="apply", points="cube4", n=500_000, cols=1, precision="fp32"),
        # source and target sets
        dict(name="cross", do="cross", points="two_sets", n=1_000_000, n_y=250_000, cols=16, precision="fp32"),
        # 512 data sets of a service, each with its own lengthscale
        dict(name="batch", do="batch", points="balls", sets=512, cols=8, precision="fp32"),
        # a rank whose factor does not fit the card: rows are kept in product form
        dict(name="huge_rank", do="product", points="normal5", n=1_000_000, cols=16, precision="fp32"),
        # kernel ridge regression, fit and predict
        dict(name="regress", do="regress", points="features8", n=20_640, cols=1, precision="fp64"),
        # many points at a loose tolerance (time against n)
        dict(name="many_points", do="product", points="unit5", n=10_000_000, cols=1, precision="fp32"),
        # few points at a tight tolerance (error against rank), double precision
        dict(name="tight_f64", do="product", points="rank5_matern52", n=5000, cols=1, precision="fp64"),
    ]


def _logint(rng, lo, hi):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v | 1 if rng.random() < 0.7 else v))


def draw(rng):
    kind = rng.choice(["small", "large", "large64", "apply", "gradient", "solve", "cross", "batch", "huge", "regress",
                       "many", "tight"])
    if kind == "small":
        return dict(do="product", points="ball3", n=_logint(rng, 500, 50_000), cols=rng.choice([1, 2, 3, 8, 17]),
                    precision=rng.choice(["fp32", "fp64"]))
    if kind == "large":
        return dict(do="product", points="mixture3", n=_logint(rng, 20_000, 1_000_000), cols=_logint(rng, 1, 64),
                    precision="fp32")
    if kind == "large64":
        return dict(do="product", points="mixture3", n=_logint(rng, 5000, 100_000), cols=_logint(rng, 1, 64),
                    precision="fp64")
    if kind == "apply":
        return dict(do="apply", points=rng.choice(["cube4", "ball3"]), n=_logint(rng, 5000, 500_000),
                    cols=rng.choice([1, 1, 2, 5, 16]), precision=rng.choice(["fp32", "fp64"]))
    if kind == "gradient":
        return dict(do="gradient", points="cube4", n=_logint(rng, 2000, 500_000), cols=rng.choice([1, 1, 2, 4]),
                    precision="fp32")
    if kind == "solve":
        return dict(do="solve", points=rng.choice(["cube4", "ball3"]), n=_logint(rng, 3000, 200_000),
                    cols=rng.choice([1, 1, 3, 16]), precision="fp32")
    if kind == "cross":
        return dict(do="cross", points="two_sets", n=_logint(rng, 10_000, 1_000_000), n_y=_logint(rng, 5000, 250_000),
                    cols=rng.choice([1, 4, 7, 16]), precision="fp32")
    if kind == "batch":
        return dict(do="batch", points="balls", sets=_logint(rng, 16, 512), cols=rng.choice([1, 3, 8, 12]),
                    precision="fp32")
    if kind == "huge":
        return dict(do="product", points="normal5", n=_logint(rng, 800_000, 1_000_000), cols=_logint(rng, 4, 16),
                    precision="fp32")
    if kind == "regress":
        return dict(do="regress", points="features8", n=_logint(rng, 3000, 20_640), cols=1, precision="fp64")
    if kind == "many":
        p = rng.choice(["unit3", "unit4", "unit5", "unit6"])
        return dict(do="product", points=p, n=_logint(rng, 10_000, 3_000_000 if p == "unit6" else 10_000_000),
                    cols=rng.choice([1, 1, 2, 8]), precision="fp32")
    return dict(do="product", points="rank5_" + rng.choice(["cauchy", "gaussian", "matern32", "matern52"]),
                n=_logint(rng, 1000, 5000), cols=rng.choice([1, 1, 2, 4]), precision="fp64")


# ------------------------------------------------------------------------------------- inputs

def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _ball(g, n, d):
    x = _randn(g, n, d)
    return x / x.norm(dim=1, keepdim=True) * _rand(g, n, 1) ** (1.0 / d)


def _clusters(g, n):
    means = -2.0 + 4.0 * _rand(g, 8, 3)
    return means[torch.randint(0, 8, (n,), generator=g, device=DEV)] + 0.3 * _randn(g, n, 3)


def _points(g, name, n):
    if name == "ball3":
        return _ball(g, n, 3)
    if name in ("mixture3", "two_sets"):
        return _clusters(g, n)
    if name == "normal5":
        x = _randn(g, n, 5) @ torch.linalg.qr(_randn(g, 5, 5))[0]
        return (x - x.mean(0)) / x.std(0, unbiased=False)
    if name == "cube4":
        return 2.0 * _rand(g, n, 4) - 1.0
    x = _randn(g, n, RECIPES[name][0])
    return x / x.norm(dim=1).max()


def _batch_sets(sets):
    r = np.random.default_rng(sets)
    sizes = np.floor(np.exp(r.uniform(math.log(1000), math.log(65536), size=sets))).astype(np.int64)
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return sizes, offsets, r.uniform(0.5, 2.0, size=sets), r.uniform(0.3, 1.5, size=sets)


def _bulk(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    d, kernel, ell, tol, _ = RECIPES[case["points"]]
    s = dict(case=case, kernel=kernel, ell=ell, tol=tol, precision=case["precision"])
    c, dt = case["cols"], _bulk(case)
    if case["do"] == "batch":
        sizes, s["offsets"], radii, s["ell"] = _batch_sets(case["sets"])
        n = int(s["offsets"][-1])
        r = torch.repeat_interleave(torch.from_numpy(radii).to(DEV), torch.from_numpy(sizes).to(DEV))
        s["x"] = _ball(g, n, d) * r[:, None]
        s["v"] = _randn(g, n, c, dtype=dt)
        return s
    n = case["n"]
    if case["do"] == "regress":
        comp = torch.randint(0, 24, (n,), generator=g, device=DEV)
        means, spreads = 0.2 + 0.6 * _rand(g, 24, d), 0.03 + 0.09 * _rand(g, 24, d)
        x = means[comp] + spreads[comp] * _randn(g, n, d)
        lo, hi = x.amin(0), x.amax(0)
        x = (x - lo) / (hi - lo)
        freq, phase = 1.0 + 2.0 * _rand(g, 4), 2.0 * math.pi * _rand(g, 4)
        y = (torch.sin(x @ _randn(g, d, 4) * freq + phase) * (0.5 + _rand(g, 4))).sum(1) + 0.1 * _randn(g, n)
        m = 2 * n // 3
        s.update(x=x[:m].contiguous(), y=y[:m].contiguous(), xq=x[m:].contiguous(), lam=1.0,
                 init=np.sort(np.random.default_rng(seed).choice(m, size=30, replace=False)))
        return s
    s["x"] = _points(g, case["points"], n)
    if case["do"] == "cross":
        s["y"] = 1.2 * _randn(g, case["n_y"], d)
        s["v"] = _randn(g, case["n_y"], c, dtype=dt)
        s["w"] = _randn(g, n, c, dtype=dt)
        return s
    s["v"] = _randn(g, n, c, dtype=dt) if c > 1 else _randn(g, n, dtype=dt)
    if case["do"] == "gradient":
        s["w"] = _randn(g, *s["v"].shape, dtype=dt)
    if case["do"] == "solve":
        s["lam"] = 1e-4 * n
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    if case["do"] == "apply":
        s["factor"] = _build(s)
    return s


# ----------------------------------------------------------------------------------- one pass

def _build(s):
    return hdf.build(s["x"], s["kernel"], s["ell"], s["tol"], precision=s["precision"])


def run(state):
    s, do = state, state["case"]["do"]
    if do == "product":
        return _build(s).matvec(s["v"])
    if do == "apply":
        return s["factor"].matvec(s["v"])
    if do == "gradient":
        f = _build(s)
        y = f.matvec(s["v"])
        gx, gell, value = f.adjoint(s["x"], s["v"], s["w"])
        return dict(y=y, grad_x=gx, grad_ell=gell, value=value, grad_v=f.matvec(s["w"]))
    if do == "solve":
        return _build(s).solve(s["lam"], s["v"], refine_steps=1)
    if do == "cross":
        f = hdf.build_cross(s["x"], s["y"], s["kernel"], s["ell"], s["tol"], precision=s["precision"])
        return f.matvec(s["v"]), f.matvec_t(s["w"])
    if do == "batch":
        return hdf.build_batched(s["x"], s["offsets"], s["kernel"], s["ell"], s["tol"],
                                 precision=s["precision"]).matvec(s["v"])
    labels, centres, _ = hdf.kmeans(s["x"], s["init"])
    model = hdf.KRR(s["x"], labels, s["kernel"], s["ell"], s["lam"], s["tol"], precision=s["precision"])
    w, _, _ = model.solve(s["y"], rtol=1e-11, max_iter=5000)
    return dict(labels=labels, centres=centres, w=w,
                prediction=hdf.kernel_matvec(s["xq"], s["x"], s["kernel"], s["ell"], w))


# --------------------------------------------------------------------------------------- work

def work(case):
    """Inputs read once and outputs written once; the flops of applying the factor's columns (two per
    entry of U, column and side) and of what the call does with them besides."""
    d, _, _, _, r = RECIPES[case["points"]]
    c, b = case["cols"], 8 if case["precision"] == "fp64" else 4
    do = case["do"]
    if do == "batch":
        n = int(_batch_sets(case["sets"])[1][-1])
        return dict(bytes=n * (8 * d + 2 * c * b), flops=4.0 * n * r * c)
    n = case["n"]
    if do == "regress":
        m, q = 2 * n // 3, n - 2 * n // 3
        # one conjugate-gradient pass over the off-diagonal pairs at the very least, and the predictions
        return dict(bytes=8 * (n * d + 2 * m + q), flops=float(m * m + m * q) * (3 * d + 8))
    if do == "cross":
        m = case["n_y"]
        return dict(bytes=(n + m) * (8 * d + 2 * c * b), flops=8.0 * (n + m) / 2 * r * c)
    if do == "apply":
        return dict(bytes=n * r * b + 2 * n * c * b, flops=4.0 * n * r * c)
    if do == "gradient":
        return dict(bytes=n * (8 * d + (4 * c + d) * b), flops=float(n) * r * (12 * c + 2 * (d + 1)))
    if do == "solve":
        return dict(bytes=n * (8 * d + 2 * c * b), flops=float(n) * r * r + 2.0 / 3.0 * r ** 3 + 12.0 * n * r * c)
    return dict(bytes=n * (8 * d + 2 * c * b), flops=float(n) * r * (4 * c + 1))


# ------------------------------------------------------------------------------ 64-bit results

def _kernel(name, r, ell):
    z = r / ell
    if name == "gaussian":
        return torch.exp(-0.5 * z * z)
    if name == "cauchy":
        return 1.0 / (1.0 + z * z)
    a = math.sqrt(3.0 if name == "matern32" else 5.0) * z
    return (1.0 + a + (0.0 if name == "matern32" else a * a / 3.0)) * torch.exp(-a)


def _dense(xq, x, kernel, ell):
    d2 = torch.zeros(xq.shape[0], x.shape[0], dtype=torch.float64, device=x.device)
    for j in range(x.shape[1]):
        d2 += (xq[:, j, None] - x[None, :, j]) ** 2
    return _kernel(kernel, d2.sqrt(), ell)


def _dense_product(xq, x, kernel, ell, v):
    step = max(1, (1 << 28) // x.shape[0])
    return torch.cat([_dense(xq[i:i + step], x, kernel, ell) @ v for i in range(0, xq.shape[0], step)])


def exact(case, seed):
    """The dense kernel in 64 bits, where that takes seconds."""
    do = case["do"]
    if do == "batch":
        pairs = float((_batch_sets(case["sets"])[0].astype(np.float64) ** 2).sum())
    elif do == "cross":
        pairs = float(case["n"]) * case["n_y"]
    else:
        pairs = float(case["n"]) ** 2
    if pairs > (4e8 if do in ("solve", "regress", "gradient") else 1.2e10):
        return None
    s = _inputs(case, seed)
    x, kernel, ell = s["x"], s["kernel"], s["ell"]
    if do == "regress":
        A = _dense(x, x, kernel, ell)
        A.diagonal().add_(s["lam"])
        w = torch.linalg.solve(A, s["y"])
        return dict(labels=None, centres=None, w=w, prediction=_dense_product(s["xq"], x, kernel, ell, w))
    v = s["v"].double()
    if do in ("product", "apply"):
        return _dense_product(x, x, kernel, ell, v)
    if do == "cross":
        return (_dense_product(x, s["y"], kernel, ell, v), _dense_product(s["y"], x, kernel, ell, s["w"].double()))
    if do == "batch":
        o = s["offsets"]
        return torch.cat([_dense_product(x[a:b], x[a:b], kernel, float(e), v[a:b])
                          for a, b, e in zip(o[:-1], o[1:], ell)])
    if do == "solve":
        A = _dense(x, x, kernel, ell)
        A.diagonal().add_(s["lam"])
        return torch.linalg.solve(A, v)
    # gradient of sum(w * K v) for the Gaussian kernel: dK_ij/dx_i = -K_ij (x_i - x_j) / l^2
    w = s["w"].double()
    v2, w2 = v.reshape(len(x), -1), w.reshape(len(x), -1)
    y, gv, gx, gell = [], [], [], 0.0
    step = max(1, (1 << 27) // len(x))
    for i in range(0, len(x), step):
        K = _dense(x[i:i + step], x, kernel, ell)
        y.append(K @ v)
        gv.append(K @ w)
        P = (w2[i:i + step] @ v2.T + v2[i:i + step] @ w2.T) * K
        gx.append((P @ x - P.sum(1, keepdim=True) * x[i:i + step]) / ell ** 2)
        d2 = torch.cdist(x[i:i + step], x) ** 2
        gell += float((0.5 * P * d2).sum()) / ell ** 3
    y = torch.cat(y)
    return dict(y=y, grad_x=torch.cat(gx), grad_ell=gell, value=float((w * y).sum()), grad_v=torch.cat(gv))
