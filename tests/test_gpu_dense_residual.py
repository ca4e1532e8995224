"""The coarse solve is backward stable: its residual stays at the rounding of |A| |e| however
ill-conditioned the coarsest operator is."""
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


# one, a few and several 64-row blocks; condition numbers from 1e3 to 1e10
@pytest.mark.parametrize("n", [40, 130, 430, 700])
@pytest.mark.parametrize("kernel,nugget", [("exponential", 0.0), ("matern32", 1e-5), ("gaussian", 1e-2),
                                           ("gaussian", 1e-5), ("gaussian", 1e-8)])
def test_residual_of_a_dense_solve(n, kernel, nugget):
    X = W.uniform_points(n, 3, 7)
    A = pkg.H2Matrix(torch.from_numpy(X).cuda(), kernel, length=0.3, nugget=nugget, leaf=64, q=2, eta=0.0)
    r = np.linalg.norm(X[:, None] - X[None], axis=2) / 0.3
    u = np.sqrt(3.0) * r
    K = {"exponential": np.exp(-r), "gaussian": np.exp(-r * r), "matern32": (1 + u) * np.exp(-u)}[kernel]
    K = K + nugget * np.eye(n)
    b = K @ np.random.default_rng(n).standard_normal(n)      # a solution much smaller than A^-1 |b|
    e = A.coarse_solve(torch.from_numpy(b).cuda()).cpu().numpy()
    # float64 sums of n terms, in the residual inside and in the one here, whose kernel
    # values differ by a rounding or two: about sqrt(n) roundings of the sum of magnitudes
    size = np.linalg.norm(K @ np.abs(e))
    assert np.linalg.norm(K @ e - b) <= 4 * n ** 0.5 * EPS * size
    A.close()


# several columns through the cycle's coarse solve, below a far field: one V-cycle of four
# columns is the V-cycles of one (to the 1e-9 of single cycles against the oracle)
def test_columns_of_a_cycle_agree():
    n = 3000
    A = pkg.H2Matrix(torch.from_numpy(W.uniform_points(n, 3, 8)).cuda(), "exponential", length=0.3, nugget=1e-2, leaf=64, q=4)
    B = torch.from_numpy(np.random.default_rng(8).standard_normal((n, 4))).cuda()
    kw = dict(tol=1e-30, max_cycles=1, n_c=3, raise_on_fail=False)
    X = A.solve(B, **kw)[0]
    for c in range(4):
        x = A.solve(B[:, c].contiguous(), **kw)[0]
        assert float((X[:, c] - x).norm()) <= 1e-9 * float(x.norm())
    A.close()
