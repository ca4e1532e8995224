"""The dense coarse operator built from 64 x 64 blocks, and its inverse."""
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


# one and several steps of the chain (tree levels above the coarsest operator's), part-filled
# bases (2-D, q = 6), skeletons, and an operator of single-level hierarchies (leaf bases)
@pytest.mark.parametrize("n,dim,kw", [(2500, 3, dict(q=4)), (6001, 2, dict(q=6)), (6001, 2, dict(q=6, coarse_level=2)),
                                      (3000, 3, dict(basis="skeleton", basis_tol=1e-7)),
                                      (2500, 3, dict(q=4, coarse_level=1))])
def test_coarse_operator_and_inverse(n, dim, kw):
    o = dict(kernel="exponential", length=0.3, nugget=1e-2, leaf=64)
    o.update(kw)
    A = pkg.H2Matrix(torch.from_numpy(W.uniform_points(n, dim, 3)).cuda(), **o)
    l = A.levels
    r = torch.from_numpy(np.random.default_rng(n).standard_normal(A.level_size(l))).cuda()
    if l > 1:
        r = A.restrict(l - 1, A.prolong(l - 1, r))           # zero in padded slots
    e = A.coarse_solve(r)
    # kappa: the largest eigenvalue over the nugget; the inverse is off by a few n eps of kappa
    v = r.abs()
    for _ in range(20):
        v = v / v.norm()
        v = A.apply_level(l, v)
    kappa = 2 * float(v.norm()) / 1e-2
    assert float((A.apply_level(l, e) - r).norm()) <= 64 * n ** 0.5 * EPS * kappa * float(r.norm())
    A.close()
