"""Digits of the float64 block product in fixed point (csrc/fixed.cuh): where they end."""
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


# single columns A e_j: every entry is one block's value times a power of two, so its error is
# the rounding of the block's values and of the sums, both relative to the block's scale s <= 2
@pytest.mark.parametrize("leaf", [64, 32])
@pytest.mark.parametrize("cols", [1, 2])
def test_single_columns(leaf, cols):
    n = 2000
    A = pkg.H2Matrix(cuda(W.uniform_points(n, 3, 2)), "gaussian", length=0.05, nugget=1e-3, leaf=leaf, q=2, eta=0.0)
    for j in range(0, n, 125):
        X = torch.zeros((cols, n), dtype=torch.float64, device="cuda")
        for c in range(cols):
            X[c, j + c] = 1.0
        Y = A.apply(X.t() if cols > 1 else X[0]).reshape(n, -1)
        for c in range(cols):
            ref = A.apply_level(1, X[c].contiguous(), precision="f64_dd")
            small = ref.abs() < 2.0 ** -8                  # their float64 results round below 2^-61
            # values at 2^-59 s; sums at 2^-58 s (rows) or 2^-57 s (columns), with x = 1 at half its scale
            err = float((Y[:, c] - ref)[small].abs().max())
            assert err <= 2 * (2.0 ** -59 + 2 * 2.0 ** -58) + 2.0 ** -61
    A.close()
