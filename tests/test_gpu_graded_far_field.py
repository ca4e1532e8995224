"""Weights over many decades with a far field: rows keep digits relative to their own size in
the product, and the dense coarse operator with a far field in it can be solved with."""
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


def graded(n, dim, decades=24, **kw):
    rng = np.random.default_rng(5)
    w = 10.0 ** rng.uniform(-decades, 0, n)
    o = dict(length=0.3, nugget=0.0, leaf=64)
    o.update(kw)
    X = W.uniform_points(n, dim, 6)
    return pkg.H2Matrix(cuda(X), "exponential", weights=cuda(w), **o), X, w, rng


# full and part-filled bases of 64 and 32 columns; skeletons
@pytest.mark.parametrize("dim,kw", [(3, dict(q=4)), (2, dict(q=6)), (3, dict(q=3)),
                                    (3, dict(basis="skeleton", basis_tol=1e-8))])
def test_rows_keep_their_digits(dim, kw):
    A, _, w, rng = graded(3000, dim, **kw)
    x = cuda(np.abs(rng.standard_normal(3000)) * np.sqrt(w))
    y, ref = A.apply(x), A.apply_level(1, x, precision="f64_dd")
    err = ((y - ref) / ref).abs()                      # positive terms: no cancellation
    # Householder's Chebyshev bases carry roundings of their own in the rows of least weight, so
    # that their products cancel there in any precision; a skeleton's rows do not
    worst = err.max() if "basis" in kw else err.median()
    assert float(worst) <= 200 * EPS
    A.close()


# a diagonal given by the caller hides the weights
def test_rows_keep_their_digits_under_a_given_diagonal():
    n = 1000
    rng = np.random.default_rng(5)
    w = 10.0 ** rng.uniform(-24, 0, n)
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 6)), "exponential", length=0.3, leaf=64, q=4, eta=0.0,
                     weights=cuda(w), diag=cuda(np.full(n, 1e-24)))
    x = cuda(np.abs(rng.standard_normal(n)) * np.sqrt(w))
    y, ref = A.apply(x), A.apply_level(1, x, precision="f64_dd")
    assert float(((y - ref) / ref).abs().max()) <= 200 * EPS
    A.close()


def test_single_level_solve_with_a_far_field():
    n = 2500
    A, X, w, rng = graded(n, 3, q=4, coarse_level=1)
    sw = cuda(np.sqrt(w))
    x = cuda(rng.standard_normal(n)) / sw
    b = A.apply_level(1, x, precision="f64_dd")
    e = A.coarse_solve(b)
    # rows of the represented matrix carry the error that the product's have; K = A / (sw sw^T)
    lam = np.linalg.eigvalsh(np.exp(-np.linalg.norm(X[:, None] - X[None], axis=2) / 0.3))
    rows = A.apply_level(1, x.abs(), precision="f64_dd")
    row_err = float(((A.apply(x) - b) / rows).abs().max())
    assert row_err <= 1e-9
    assert float(((e - x) * sw).norm()) <= lam[-1] / lam[0] * max(row_err, EPS) * float((x * sw).norm())
    A.close()
