"""The autotuner times the arithmetic that ordinary vectors take, whatever the last product
left in the workspaces."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2501_17656_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)


def test_tuning_after_a_product_with_nan():
    n = 50000
    A = pkg.H2Matrix(torch.from_numpy(W.uniform_points(n, 3, 2)).cuda(), "gaussian", length=0.05, nugget=1e-3,
                     leaf=64, q=4)
    x = torch.from_numpy(np.random.default_rng(2).standard_normal(n)).cuda()

    def times():
        return {(op, nr): fixed for op, nr, fixed, _ in A.autotune() if op <= 1}

    A.apply(x)
    before = times()
    A.apply(torch.full_like(x, float("nan")))
    after = times()
    for k, t in before.items():
        assert after[k] <= 1.3 * t, (k, t, after[k])
    assert torch.isfinite(A.apply(x)).all()
    A.close()
