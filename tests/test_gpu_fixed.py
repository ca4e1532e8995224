"""The float64 block product on the integer pipe (csrc/fixed.cuh) against the double-double
product, and the inputs that leave it for the float64 path."""
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


def matrix(n, dim=3, k=1, **kw):
    o = dict(kernel="exponential", length=0.3, nugget=1e-2, leaf=64, q=4)
    o.update(kw)
    return pkg.H2Matrix(cuda(W.uniform_points(n, dim, k)), **o)


# sizes: one leaf, a few leaves with no far field, ragged leaves, several levels; blocks of
# 64 and 32, bases of 16, 27 and 64 columns
@pytest.mark.parametrize("n,dim,leaf,q", [(33, 3, 64, 4), (64, 2, 64, 4), (65, 2, 64, 4), (300, 3, 32, 3),
                                          (1500, 2, 64, 4), (1501, 2, 32, 5), (4999, 3, 64, 4), (5000, 3, 32, 3),
                                          (9973, 2, 64, 8)])
@pytest.mark.parametrize("cols", [1, 2, 3])
def test_product_against_double_double(n, dim, leaf, q, cols):
    A = matrix(n, dim, leaf=leaf, q=q)
    rng = np.random.default_rng(n + cols)
    X = rng.standard_normal((n, cols))
    X[:, -1] *= np.exp(6 * rng.standard_normal(n))          # a column whose entries spread widely
    if n > 200:
        X[: n // 3, 0] = 0.0                                # whole leaves of zeros among them
    Y = A.apply(cuda(X))
    for c in range(cols):
        x = cuda(X[:, c])
        ref = A.apply_level(1, x, precision="f64_dd")
        # rounding of a float64 sum relative to the sum of magnitudes: the passes add a few
        # hundred terms in chains of about 64, the transfers a few levels of 64 more
        size = A.apply_level(1, x.abs(), precision="f64_dd")
        assert float((Y[:, c] - ref).norm()) <= 64 * EPS * float(size.norm())
    A.close()


@pytest.mark.parametrize("scale", [1e-300, 1e-280, 1e120, 1e200, 1e290])
def test_scales_outside_fixed_point_take_the_float64_path(scale):
    A = matrix(3000)
    x = np.random.default_rng(3).standard_normal(3000)
    y = A.apply(cuda(x))
    ys = A.apply(cuda(x * scale))
    assert float((ys / scale - y).norm()) <= 64 * EPS * float(A.apply(cuda(np.abs(x))).norm())
    two = np.stack([x, x * scale], 1)                        # both kinds in one group
    Y = A.apply(cuda(two))
    assert float((Y[:, 0] - y).norm()) <= 64 * EPS * float(A.apply(cuda(np.abs(x))).norm())
    A.close()


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_inputs_reach_the_outputs(bad):
    A = matrix(3000)
    x = np.random.default_rng(4).standard_normal(3000)
    x[1234] = bad
    y = A.apply(cuda(x)).cpu().numpy()
    assert not np.isfinite(y[1234])
    A.close()


def test_widely_varying_weights_keep_their_digits():
    """Panel weights over 24 decades give rows with scales of their own: every row of the
    close field keeps float64 accuracy relative to its own size."""
    n = 1000
    rng = np.random.default_rng(5)
    w = 10.0 ** rng.uniform(-24, 0, n)
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 6)), "exponential", length=0.3, nugget=0.0, leaf=64, q=4, eta=0.0,
                     weights=cuda(w))
    x = cuda(np.abs(rng.standard_normal(n)) * np.sqrt(w))
    y, ref = A.apply(x), A.apply_level(1, x, precision="f64_dd")
    assert float(((y - ref) / ref).abs().max()) <= 200 * EPS       # positive terms: no cancellation
    A.close()
