"""Skeletonization around the edges of its row chunks (32), groups of chunks (2 and 3) and
column limits (64 and 128 candidates): decisions equal to the oracle's, products to 1e-12."""
import numpy as np
import pytest

import workloads as W
from oracle import H2Matrix, KernelSpec

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2501_17656_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)


# 1-D: few far rows per cluster (fewer chunks than groups); odd leaf sizes: part-filled chunks
# and columns; 3-D with rank 64 children: 128 candidates
@pytest.mark.parametrize("n,dim,leaf,tol,cap", [(67, 1, 16, 1e-8, 16), (131, 1, 17, 1e-10, 32), (333, 1, 64, 1e-9, 64),
                                                (509, 2, 33, 1e-6, 64), (1201, 2, 64, 1e-10, 64),
                                                (1999, 3, 48, 1e-8, 64), (3001, 3, 64, 1e-10, 64)])
def test_skeletons_and_product(n, dim, leaf, tol, cap):
    X = W.uniform_points(n, dim, 5)
    A = pkg.H2Matrix(torch.from_numpy(X).cuda(), "exponential", length=0.2, nugget=1e-2, leaf=leaf, eta=1.0,
                     basis="skeleton", basis_tol=tol, rank_max=cap)
    h = H2Matrix(X, KernelSpec("exponential", 0.2, 1e-2), leaf, 4, 1.0, basis="skeleton", tol=tol, rank_max=cap)
    for ell in range(h.tstar, h.L + 1):
        np.testing.assert_array_equal(A.export("RANKS", ell), [h.rank[(ell, j)] for j in range(1 << ell)])
    x = np.random.default_rng(n).standard_normal(n)
    y, yo = A.apply(torch.from_numpy(x).cuda()).cpu().numpy(), h.apply(x)
    assert np.linalg.norm(y - yo) <= 1e-12 * np.linalg.norm(yo)
    A.close()
