"""The factor and inverse of the coarsest operator against NumPy."""
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


# orders of the dense operator around the 64-row blocks of the factorisation
@pytest.mark.parametrize("n,leaf", [(5, 16), (17, 16), (40, 16), (63, 64), (65, 16), (130, 32), (500, 64), (700, 64)])
def test_dense_inverse(n, leaf):
    """No far field (eta = 0): the coarse solve is the dense solve of the whole matrix."""
    X = W.uniform_points(n, 3, 7)
    A = pkg.H2Matrix(cuda(X), "matern32", length=0.2, nugget=1e-2, leaf=leaf, q=2, eta=0.0)
    d = np.linalg.norm(X[:, None] - X[None], axis=2) * np.sqrt(3.0) / 0.2
    K = (1 + d) * np.exp(-d) + 1e-2 * np.eye(n)
    b = np.random.default_rng(n).standard_normal(n)
    e = A.coarse_solve(cuda(b)).cpu().numpy()
    cond = np.linalg.cond(K)
    assert np.linalg.norm(e - np.linalg.solve(K, b)) <= 8 * n ** 0.5 * cond * EPS * np.linalg.norm(e) + 1e-300
    A.close()


def test_dense_factor_reports_an_indefinite_matrix():
    A = pkg.H2Matrix(cuda(W.uniform_points(200, 3, 8)), "exponential", length=0.3, nugget=-2.0, leaf=64, q=2, eta=0.0)
    with pytest.raises(pkg.H2MGError) as e:
        A.coarse_solve(torch.zeros(200, dtype=torch.float64, device="cuda"))
    assert e.value.name == "NOT_SPD"
    A.close()
