"""The factor of the coarsest operator does not depend on the scale of its rows: a dense solve
with weights over many decades is as accurate, relative to each row's scale, as one without."""
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


# one, a few and several 64-row blocks; weights that vary inside each of them, by blocks, and
# all of them far below and above one
@pytest.mark.parametrize("n", [50, 130, 500])
@pytest.mark.parametrize("lo,hi", [(0, 0), (-12, 0), (-24, 0), (-32, 0), (-200, -180), (100, 124)])
def test_dense_solve_with_graded_weights(n, lo, hi):
    X = W.uniform_points(n, 3, 6)
    rng = np.random.default_rng(n + abs(lo))
    w = 10.0 ** rng.uniform(lo, hi, n)
    A = pkg.H2Matrix(torch.from_numpy(X).cuda(), "exponential", length=0.3, nugget=0.0, leaf=64, q=2, eta=0.0,
                     weights=torch.from_numpy(w).cuda())
    K = np.exp(-np.linalg.norm(X[:, None] - X[None], axis=2) / 0.3)
    b, sw = rng.standard_normal(n), np.sqrt(w)
    # A = sw K sw, so A e = sw b has sw e = K^-1 b
    e = A.coarse_solve(torch.from_numpy(sw * b).cuda()).cpu().numpy() * sw
    want = np.linalg.solve(K, b)
    assert np.linalg.norm(e - want) <= 8 * n ** 0.5 * np.linalg.cond(K) * EPS * np.linalg.norm(want)
    A.close()
