"""Cases that stand for what a program does with this library.

A program builds an H2 matrix from points and a kernel, multiplies with it (one vector, a
few columns, a panel of columns), smooths and runs multigrid cycles with it, solves (one
matrix with several right-hand sides, many matrices together), and differentiates a loss
through the solves. The kernels, dimensions, leaf sizes, node counts, nuggets and
tolerances are those of the repository's workloads and tests: the exponential kernel on the
unit square, the Gaussian and Matern-3/2 kernels in the unit cube (Chebyshev nodes, or
skeleton bases at the density of the 2^20-point problem), and the single-layer kernel on
perturbed spheres.

A case is a dict of plain values:
  do      matvec | smooth | vcycle | solve | batch | build | grad
  points  square | cube | dense_cube (the cube scaled to the density of 2^20 points) | sphere
  n       points (spheres: rounded to 20 m^2 panels)
  ...     the options of the call
"""
import math

import numpy as np
import torch

import paper_2501_17656_gb300 as h2
import workloads

DEV = "cuda"


# --------------------------------------------------------------------------- listed cases
def listed():
    return [
        # the smallest product: one vector, 4096 points on the square (the first workload)
        dict(name="matvec_square_4096_f64", do="matvec", points="square", n=4096, kernel="exponential", length=0.1,
             nugget=1e-2, leaf=64, q=4, storage="f64", precision="", nrhs=1),
        # the largest product: one vector, float64, an odd number of points in the cube
        dict(name="matvec_cube_100003_f64", do="matvec", points="cube", n=100003, kernel="gaussian", length=0.05,
             nugget=1e-3, leaf=64, q=4, storage="f64", precision="", nrhs=1),
        # the double-float storage, three columns (a group of two and a single one)
        dict(name="matvec_square_50021_df64_3", do="matvec", points="square", n=50021, kernel="exponential",
             length=0.1, nugget=1e-2, leaf=64, q=4, storage="df64", precision="", nrhs=3),
        # the FP32 copy on a surface, seven columns (groups of four, two and one)
        dict(name="matvec_sphere_18000_f32_7", do="matvec", points="sphere", n=18000, kernel="laplace_sl", length=1.0,
             nugget=0.0, leaf=64, q=4, storage="f64", precision="mixed_f32", nrhs=7),
        # many right-hand sides through the tensor-core product: a panel of 100 columns
        dict(name="matvec_cube_16411_panel_100", do="matvec", points="dense_cube", n=16411, kernel="gaussian",
             length=0.05, nugget=1e-3, leaf=64, basis="skeleton", storage="f64", precision="tf32x3", nrhs=100),
        # the smoother of a mixed cycle: 40 CG steps on the second level, FP32 products
        dict(name="smooth_cube_30011_level2_f32", do="smooth", points="cube", n=30011, kernel="gaussian", length=0.05,
             nugget=1e-3, leaf=64, q=4, storage="f64", precision="mixed_f32", level=2, steps=40),
        # one float64 V-cycle of the first workload: many steps on few unknowns (ten per level:
        # with forty the last ones only turn rounding into other steps)
        dict(name="vcycle_square_4096_f64", do="vcycle", points="square", n=4096, kernel="exponential", length=0.1,
             nugget=1e-2, leaf=64, q=4, storage="f64", precision="f64", cycle="V", n_c=10),
        # one mixed V-cycle on skeleton bases at the density of the large Gaussian problem
        dict(name="vcycle_cube_16384_mixed", do="vcycle", points="dense_cube", n=16384, kernel="gaussian", length=0.05,
             nugget=1e-3, leaf=64, basis="skeleton", storage="f64", precision="mixed_f32", cycle="V", n_c=40),
        # a solve to 1e-10 on a surface: four right-hand sides, mixed precision, replayed cycles
        dict(name="solve_sphere_18000_mixed_4", do="solve", points="sphere", n=18000, kernel="laplace_sl", length=1.0,
             nugget=0.0, leaf=64, q=4, storage="f64", precision="mixed_f32", nrhs=4),
        # independent surface problems of uneven size solved together
        dict(name="batch_spheres_6_mixed", do="batch", points="sphere", sizes="4500,5780,8000,12500,18000,32000",
             kernel="laplace_sl", length=1.0, nugget=0.0, leaf=64, q=4, storage="f64", precision="mixed_f32"),
        # a new matrix (skeleton bases to 1e-9, FP32 copy, hierarchy) and its first product
        dict(name="build_cube_8192_skeleton", do="build", points="dense_cube", n=8192, kernel="gaussian", length=0.05,
             nugget=1e-3, leaf=64, basis="skeleton", storage="f64"),
        # one step of a hyperparameter fit: loss and gradients, the matrices built anew
        dict(name="grad_cube_4096_matern", do="grad", points="cube", n=4096, kernel="matern32", length=0.1,
             nugget=1e-2, leaf=64, q=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["matvec", "matvec", "matvec", "smooth", "vcycle", "solve", "batch", "build", "grad"])
    # leaf sizes and node counts of the repository's tests: blocks of 16, 32 and 64
    leaf = rng.choice([64, 64, 64, 48, 32, 16])
    square = dict(points="square", kernel="exponential", length=0.1, nugget=1e-2, leaf=leaf, q=rng.choice([4, 4, 3, 6]))
    cube = dict(points="cube", kernel="gaussian", length=0.05, nugget=1e-3, leaf=leaf, q=rng.choice([4, 4, 3]))
    matern = dict(points="cube", kernel="matern32", length=0.1, nugget=1e-2, leaf=leaf, q=rng.choice([4, 4, 3]))
    sphere = dict(points="sphere", kernel="laplace_sl", length=1.0, nugget=0.0, leaf=64, q=4)
    dense = dict(points="dense_cube", kernel="gaussian", length=0.05, nugget=1e-3, leaf=64, basis="skeleton")
    if do == "matvec":
        kind = rng.choice(["f64", "f64", "df64", "f32", "panel"])
        if kind == "panel":
            return dict(do=do, **rng.choice([dense, sphere]), n=_log(rng, 1000, 16411), storage="f64",
                        precision="tf32x3", nrhs=rng.choice([16, 33, 64, 100, 128]))
        c = rng.choice([square, cube, matern, sphere])
        top = 100003 if c["points"] == "square" else 50000
        return dict(do=do, **c, n=_log(rng, 1000, top), storage="df64" if kind == "df64" else "f64",
                    precision="mixed_f32" if kind == "f32" else "", nrhs=rng.choice([1, 1, 1, 2, 3, 4, 5, 16]))
    if do == "smooth":
        c = rng.choice([square, cube, sphere])
        return dict(do=do, **c, n=_log(rng, 4000, 30011), storage="f64", precision=rng.choice(["f64", "mixed_f32"]),
                    level=rng.choice([1, 2, 2, 3]), steps=rng.choice([1, 10, 40]))
    if do == "vcycle":
        c = rng.choice([square, dense, sphere])
        return dict(do=do, **c, n=_log(rng, 2000, 16384), storage="f64", precision=rng.choice(["f64", "mixed_f32"]),
                    cycle=rng.choice(["V", "V", "W", "F"]), n_c=rng.choice([5, 10]))
    if do == "solve":
        return dict(do=do, **sphere, n=_log(rng, 2000, 18000), storage="f64",
                    precision=rng.choice(["f64", "mixed_f32", "mixed_f32"]), nrhs=rng.choice([1, 2, 4, 5]))
    if do == "batch":
        sizes = sorted(_log(rng, 2000, 18000) for _ in range(rng.choice([2, 3, 5])))
        return dict(do=do, **sphere, sizes=",".join(str(s) for s in sizes), storage="f64", precision="mixed_f32")
    if do == "build":
        c = rng.choice([dense, square, cube, sphere])
        return dict(do=do, **c, n=_log(rng, 1000, 8192), storage=rng.choice(["f64", "f64", "df64"]))
    return dict(do=do, points="cube", kernel="matern32", length=0.1, nugget=1e-2, leaf=64, q=rng.choice([4, 3]),
                n=_log(rng, 3000, 4096))


# --------------------------------------------------------------------------- inputs
def _seed(case, seed, k=0):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, int(case.get("n", 0)), k])


def _geometry(case, seed, n=None, k=0):
    """(points, weights or None) as float64 tensors on the GPU."""
    n = int(n if n is not None else case["n"])
    if case["points"] == "sphere":
        m = max(1, int(round(math.sqrt(n / 20.0))))
        c, a, _ = workloads.perturbed_icosphere(m, (int(seed) * 16 + k) % 1000003)
        return torch.from_numpy(c).to(DEV), torch.from_numpy(a).to(DEV)
    x = _seed(case, seed, k).random((n, 2 if case["points"] == "square" else 3))
    if case["points"] == "dense_cube":
        x *= (n / 2.0 ** 20) ** (1.0 / 3.0)
    return torch.from_numpy(x).to(DEV), None


def _normal(case, seed, n, nrhs=1, k=100):
    v = _seed(case, seed, k).standard_normal((nrhs, n))
    t = torch.from_numpy(v).to(DEV)
    return t[0] if nrhs == 1 else t.t()      # columns in the library's column-major layout


def _matrix(case, x, w, with_f32):
    o = dict(basis="skeleton", basis_tol=1e-9) if case.get("basis") == "skeleton" else dict(q=case["q"])
    return h2.H2Matrix(x, case["kernel"], length=case["length"], nugget=case["nugget"], weights=w, leaf=case["leaf"],
                       storage=case["storage"], with_f32=with_f32, **o)


def prepare(case, seed):
    do = case["do"]
    s = dict(case=case)
    if do == "batch":
        s["mats"], s["bs"] = [], []
        for k, n in enumerate(case["sizes"].split(",")):
            x, w = _geometry(case, seed, int(n), k)
            s["mats"].append(_matrix(case, x, w, True))
            s["bs"].append(_normal(case, seed, x.shape[0], 1, 100 + k))
        return s
    x, w = _geometry(case, seed)
    n = x.shape[0]
    if do == "build":
        s.update(x=x, w=w, v=_normal(case, seed, n))
        return s
    if do == "grad":
        s["x"] = x
        s["y"] = _normal(case, seed, n, 1, 100).requires_grad_()
        s["b"] = _normal(case, seed, n, 1, 101).requires_grad_()
        s["l"] = torch.tensor(case["length"], dtype=torch.float64, device=DEV, requires_grad=True)
        s["s"] = torch.tensor(case["nugget"], dtype=torch.float64, device=DEV, requires_grad=True)
        return s
    A = s["A"] = _matrix(case, x, w, case["precision"] in ("mixed_f32", "tf32x3"))
    if do == "matvec":
        s["v"] = _normal(case, seed, n, case["nrhs"])
        s["y"] = torch.empty_like(s["v"])
    elif do == "smooth":
        s["level"] = max(1, min(case["level"], A.levels - 1))
        s["f"] = _normal(case, seed, A.level_size(s["level"]))
    else:
        s["b"] = _normal(case, seed, n, case.get("nrhs", 1))
        s["zero"] = torch.zeros(n, dtype=torch.float64, device=DEV)
    return s


# --------------------------------------------------------------------------- one pass
def run(s):
    case = s["case"]
    do = case["do"]
    if do == "matvec":
        if case["precision"]:
            return s["A"].apply(s["v"], y=s["y"], precision=case["precision"])
        return s["A"].apply(s["v"], y=s["y"])
    if do == "smooth":
        return s["A"].smooth(s["level"], s["f"], n=case["steps"], precision=case["precision"])
    if do == "vcycle":
        return s["A"].vcycle(s["zero"], s["b"], precision=case["precision"], cycle=case["cycle"],
                             n_c=case["n_c"])
    if do == "solve":
        return s["A"].solve(s["b"], tol=1e-10, max_cycles=60, outer="fcg", precision=case["precision"],
                            use_graph=True)[0]
    if do == "batch":
        return h2.solve_batched(s["mats"], s["bs"], tol=1e-10, max_cycles=60, outer="fcg",
                                precision=case["precision"], use_graph=True)[0]
    if do == "build":
        A = _matrix(case, s["x"], s["w"], True)
        y = A.apply(s["v"])
        ranks = [A.export("RANKS", k) for k in range(A.query("TSTAR"), A.query("L") + 1)] if A.query("TSTAR") >= 0 else []
        A.close()
        return {"y": y, "ranks": ranks}
    for t in (s["y"], s["b"], s["l"], s["s"]):
        t.grad = None
    loss = h2.MaternLoss.apply(s["x"], s["y"], s["b"], s["l"], s["s"], case["leaf"], case["q"], 1.0, 1e-12, 200, "fcg")
    loss.backward()
    return {"loss": loss.detach(), "dy": s["y"].grad, "db": s["b"].grad, "dl": s["l"].grad, "ds": s["s"].grad}


# --------------------------------------------------------------------------- work
def _counts(A):
    """Stored blocks of the level-1 product, clusters with a transfer, and block edges."""
    L, ts = A.query("L"), A.query("TSTAR")
    far = sum(A.query("FAR_PAIRS", k) for k in range(ts, L + 1)) if ts >= 0 else 0
    clusters = sum(1 << k for k in range(ts + 1, L + 1)) if ts >= 0 else 0
    return A.query("NEAR_PAIRS"), far, clusters, A.query("KD"), A.query("KC"), L, ts


def _product(A, level, eb, nrhs):
    """Bytes and operations of one product with A_level: each stored block, transfer and leaf
    basis read once, the vectors read and written once."""
    near, far, clusters, kd, kc, L, ts = _counts(A)
    if level == 1:
        n, blocks, small = A.n, near * kd * kd + far * kc * kc, clusters * kc * kc + ((1 << L) * kd * kc if ts >= 0 else 0)
    else:
        n = A.level_size(level)
        m = L - level + 2
        far = sum(A.query("FAR_PAIRS", k) for k in range(ts, m + 1))
        # the non-far pairs of tree level m: all pairs under the far ones of the levels above
        full = (1 << m) * ((1 << m) + 1) // 2
        full -= sum(A.query("FAR_PAIRS", k) << (2 * (m - k)) for k in range(ts, m + 1))
        blocks, small = (far + full) * kc * kc, sum(1 << k for k in range(ts + 1, m + 1)) * kc * kc
    return (blocks + small) * eb + 16 * n * nrhs, (4 * blocks + 4 * small) * nrhs


def _cycle(A, eb, nrhs, n_c=40):
    by, fl = 0, 0
    for i in range(1, A.levels):
        steps = 2 if i == 1 else 2 * n_c
        b, f = _product(A, i, eb, nrhs)
        by, fl = by + steps * b, fl + steps * f
    return by + 8 * A.level_size(A.levels) ** 2, fl


def _build(A, with_f32):
    """Every stored block and basis written once; the products that form the couplings and
    the coarse near fields, and the factor and inverse of the coarsest operator."""
    near, far, clusters, kd, kc, L, ts = _counts(A)
    by = A.query("BYTES_PRIMARY") + (A.query("BYTES_F32") if with_f32 else 0) + 8 * clusters * kc * kc
    fl = far * 2 * kc ** 3 + near * (4 * kd * kd * kc)
    nl = A.level_size(A.levels) if A.levels > 1 else A.n
    return by + 8 * nl * nl, fl + nl ** 3


def work(case):
    do, eb = case["do"], 4 if case.get("precision") in ("mixed_f32", "tf32x3") else 8
    if do == "batch":
        by = fl = 0
        for k, n in enumerate(case["sizes"].split(",")):
            x, w = _geometry(case, 0, int(n), k)
            A = _matrix(case, x, w, False)
            b, f = _cycle(A, 4, 1)
            b2, f2 = _product(A, 1, 8, 1)
            by, fl = by + 2 * b + 4 * b2, fl + 2 * f + 4 * f2
            A.close()
        return {"bytes": float(by), "flops": float(fl)}
    x, w = _geometry(case, 0)
    A = _matrix(dict(case, storage=case.get("storage", "f64")), x, w, do == "build")
    if do == "matvec":
        by, fl = _product(A, 1, eb, case["nrhs"])
    elif do == "smooth":
        by, fl = _product(A, max(1, min(case["level"], A.levels - 1)), eb, 1)
        by, fl = by * case["steps"], fl * case["steps"]
    elif do == "vcycle":
        by, fl = _cycle(A, eb, 1, case["n_c"])
    elif do == "solve":
        by, fl = _cycle(A, eb, case["nrhs"])
        b2, f2 = _product(A, 1, 8, case["nrhs"])
        by, fl = 2 * by + 4 * b2, 2 * fl + 4 * f2
    elif do == "build":
        by, fl = _build(A, True)
        b, f = _product(A, 1, 8, 1)
        by, fl = by + b, fl + f
    else:
        by, fl = _build(A, False)
        near, far, _, kd, kc, _, _ = _counts(A)
        by += (near * kd * kd + far * kc * kc) * 8          # the derivative matrix
        b, f = _cycle(A, 8, 3)
        by, fl = by + 4 * b, fl + 4 * f                     # a few cycles of the three-column solve
    A.close()
    return {"bytes": float(by), "flops": float(fl)}


# --------------------------------------------------------------------------- exact values
def _kernel_rows(case, x, w, rows, length=None, derivative=False):
    """Rows of the dense kernel matrix (float64), with the nugget on its diagonal."""
    ell = case["length"] if length is None else length
    r = torch.cdist(x[rows], x, compute_mode="donot_use_mm_for_euclid_dist")
    if case["kernel"] == "exponential":
        k = torch.exp(-r / ell)
    elif case["kernel"] == "gaussian":
        k = torch.exp(-(r / ell) ** 2)
    elif case["kernel"] == "matern32":
        u = math.sqrt(3.0) * r / ell
        k = (3.0 * r * r / ell ** 3) * torch.exp(-u) if derivative else (1.0 + u) * torch.exp(-u)
    else:
        sw = torch.sqrt(w)
        k = sw[rows, None] * sw[None, :] / (4.0 * math.pi * r)
    i = torch.arange(rows.stop - rows.start, device=x.device)
    if case["kernel"] == "laplace_sl":
        k[i, i + rows.start] = 0.5 * torch.sqrt(w[rows] / math.pi)
    if not derivative:
        k[i, i + rows.start] += case["nugget"]
    return k


def _dense_product(case, x, w, v):
    out = torch.empty_like(v)
    step = max(1, int(1.5e8) // x.shape[0])
    for a in range(0, x.shape[0], step):
        rows = slice(a, min(a + step, x.shape[0]))
        out[rows] = _kernel_rows(case, x, w, rows) @ v
    return out


def exact(case, seed):
    do = case["do"]
    if do in ("smooth", "vcycle", "batch"):
        return None                  # steps of the hierarchy's own operators; large solves
    x, w = _geometry(case, seed)
    n = x.shape[0]
    if do == "matvec":
        return _dense_product(case, x, w, _normal(case, seed, n, case["nrhs"]))
    if do == "build":
        return {"y": _dense_product(case, x, w, _normal(case, seed, n)), "ranks": None}
    if do == "solve":
        k = _kernel_rows(case, x, w, slice(0, n))
        b = _normal(case, seed, n, case["nrhs"])
        return torch.cholesky_solve(b.reshape(n, -1), torch.linalg.cholesky(k)).reshape(b.shape)
    y, b = _normal(case, seed, n, 1, 100), _normal(case, seed, n, 1, 101)
    f = torch.linalg.cholesky(_kernel_rows(case, x, w, slice(0, n)))
    a, s, u = torch.cholesky_solve(torch.stack([y, b, torch.ones_like(b)], 1), f).unbind(1)
    d = _kernel_rows(case, x, w, slice(0, n), derivative=True)
    return {"loss": 0.5 * (y @ a) + s.sum(), "dy": a, "db": u, "dl": -0.5 * (a @ (d @ a)) - u @ (d @ s),
            "ds": -0.5 * (a @ a) - u @ s}
