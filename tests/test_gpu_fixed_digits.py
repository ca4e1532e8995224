"""Digits of the float64 block product in fixed point (csrc/fixed.cuh): where they end."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2501_17656_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)
EPS = 2.0 ** -53


def cuda(x):
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


# single columns A e_j: every entry is one block's value times a power of two, so its error is
# the rounding of the block's values and of the sums, both relative to the block's scale s <= 2
@pytest.mark.parametrize("leaf", [64, 32])
@pytest.mark.parametrize("cols", [1, 2])
def test_single_columns(leaf, cols):
    n = 2000
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 2)), "gaussian", length=0.05, nugget=1e-3, leaf=leaf, q=2, eta=0.0)
    for j in range(0, n, 125):
        X = torch.zeros((cols, n), dtype=torch.float64, device="cuda")
        for c in range(cols):
            X[c, j + c] = 1.0
        Y = A.apply(X.t() if cols > 1 else X[0]).reshape(n, -1)
        for c in range(cols):
            ref = A.apply_level(1, X[c].contiguous(), precision="f64_dd")
            small = ref.abs() < 2.0 ** -8                  # their float64 results round below 2^-61
            # values at 2^-59 s; sums at 2^-58 s (rows) or 2^-57 s (columns), with x = 1 at half its scale
            err = float((Y[:, c] - ref)[small].abs().max())
            assert err <= 2 * (2.0 ** -59 + 2 * 2.0 ** -58) + 2.0 ** -61
    A.close()


# a vector that spans many decades inside every leaf: each row is as accurate as a float64 sum
# of its own terms (close blocks only, where every entry of A is stored)
@pytest.mark.parametrize("kernel,length", [("gaussian", 0.05), ("exponential", 0.3)])
@pytest.mark.parametrize("cols", [1, 3])
def test_spread_vectors_keep_their_digits(kernel, length, cols):
    n = 2000
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 2)), kernel, length=length, nugget=1e-3, leaf=64, q=2, eta=0.0)
    rng = np.random.default_rng(n)
    X = rng.standard_normal((cols, n))
    X[0] = np.exp(6 * X[0])
    Y = A.apply(cuda(X).t() if cols > 1 else cuda(X[0])).reshape(n, -1)
    ref = A.apply_level(1, cuda(X[0]), precision="f64_dd")
    assert float(((Y[:, 0] - ref) / ref).abs().max()) <= 200 * EPS      # positive terms
    A.close()


# leaves below the limit of 2^20 are what the fixed point serves: the error is that of its
# values, relative to the largest entry and the largest piece
def test_vectors_of_moderate_spread():
    n = 2000
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 2)), "gaussian", length=0.05, nugget=1e-3, leaf=64, q=2, eta=0.0)
    rng = np.random.default_rng(3)
    x = cuda(2.0 ** rng.uniform(-14, 0, n))
    err = (A.apply(x) - A.apply_level(1, x, precision="f64_dd")).abs()
    # per row: n terms below 2 (|A| <= 2, |x| <= 1 at scales of 2) off by 2^-57.4 each at random
    # signs, and the float64 additions of the blocks' parts
    assert float(err.max()) <= n ** 0.5 * 4 * 2.0 ** -57.4 + 64 * EPS * 2
    A.close()


# block and vector both so small that the product of their scales is no normal number
@pytest.mark.parametrize("cols", [1, 2])
def test_tiny_blocks_times_tiny_vectors(cols):
    n = 2000
    X = np.abs(np.random.default_rng(4).standard_normal((cols, n)))
    w = cuda(np.full(n, 1e-150))
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 2)), "exponential", length=0.3, leaf=64, q=2, eta=0.0, weights=w)
    cast = (lambda V: cuda(V).t()) if cols > 1 else (lambda V: cuda(V[0]))
    y, ys = A.apply(cast(X)), A.apply(cast(X * 1e-158))
    # products near 1e-308 round at 2^-1075 in float64: 2000 of them below 1e-13 of a sum of 1e-306
    assert float((ys / 1e-158 / y - 1.0).abs().max()) <= 1e-12
    A.close()
