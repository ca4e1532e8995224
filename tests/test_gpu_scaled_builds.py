"""A matrix scaled by a power of two (its weights) near the ends of the float64 range has the
scaled operators and the scaled inverse."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2501_17656_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)
N = 2500


def matrix(e, dim=3, **kw):
    w = torch.full((N,), 2.0 ** e, dtype=torch.float64, device="cuda")
    return pkg.H2Matrix(torch.from_numpy(W.uniform_points(N, dim, 6)).cuda(), "exponential", length=0.3, nugget=0.0, leaf=64,
                        weights=w, **kw)


# 2^980 and 2^-940: beyond the exponents of fixed point; the others inside
@pytest.mark.parametrize("e", [-940, -500, 20, 700, 980])
@pytest.mark.parametrize("kw", [dict(q=4), dict(dim=2, q=6)])        # two levels, and several
def test_level_operators(e, kw):
    A, B = matrix(0, **kw), matrix(e, **kw)
    rng = np.random.default_rng(1)
    for i in range(1, A.levels + 1):
        v = torch.from_numpy(rng.standard_normal(A.level_size(i))).cuda()
        a = A.apply_level(i, v)
        b = B.apply_level(i, v) * 2.0 ** -e
        # the same sums in another order, and in another arithmetic for some of them
        assert float((a - b).norm()) <= 64 * 2.0 ** -53 * float(A.apply_level(i, v.abs()).norm() + a.norm())
    A.close()
    B.close()


@pytest.mark.parametrize("e", [-940, 20, 980])
def test_dense_solve(e):
    A, B = matrix(0, q=4, coarse_level=1), matrix(e, q=4, coarse_level=1)
    x = torch.from_numpy(np.random.default_rng(2).standard_normal(N)).cuda()
    b = A.apply(x)
    a, c = A.coarse_solve(b), B.coarse_solve(b) * 2.0 ** e
    # condition number below 1e5; the expansions round differently
    assert float((a - c).norm()) <= 64 * N ** 0.5 * 2.0 ** -53 * 1e5 * float(a.norm())
    A.close()
    B.close()
