"""The coarse near fields P_i of 64 x 64 blocks: A_(i+1) = U_i^T A_i U_i at every level."""
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


# 64-column bases full (3-D, q = 4) and part-filled (2-D, q = 6), skeletons, both storages
@pytest.mark.parametrize("n,dim,kw", [(4999, 3, dict(q=4)), (6001, 2, dict(q=6)), (4999, 3, dict(q=4, storage="df64")),
                                      (4000, 3, dict(basis="skeleton", basis_tol=1e-7))])
def test_galerkin_blocks(n, dim, kw):
    A = matrix(n, dim, **kw)
    rng = np.random.default_rng(n)
    for i in range(1, A.levels):
        v = cuda(rng.standard_normal(A.level_size(i + 1)))
        v = A.restrict(i, A.prolong(i, v))                   # zero in padded slots
        want = A.restrict(i, A.apply_level(i, A.prolong(i, v)))
        got = A.apply_level(i + 1, v)
        # double-float storage rounds every block at 2^-48
        tol = 64 * (EPS if kw.get("storage") != "df64" else 2.0 ** -46)
        size = A.apply_level(i, A.prolong(i, v).abs())
        assert float((got - want).norm()) <= tol * max(float(size.norm()), float(want.norm()))
    A.close()
