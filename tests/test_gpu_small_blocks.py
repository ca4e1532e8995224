"""Products whose blocks are 16 or 32 wide (k_bsgemv_small) in every format and column
group, against the double-double product of the float64 matrix."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2501_17656_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)


# (points, leaf, nodes per axis): blocks D / coupling 16 / 16, 32 / 16, 32 / 32, 16 / 32; one
# row, a few rows without a far field, ragged leaves
@pytest.mark.parametrize("n,leaf,q", [(9, 16, 4), (40, 16, 4), (999, 16, 4), (2500, 32, 4), (2501, 32, 5), (1777, 13, 5)])
@pytest.mark.parametrize("fmt", ["f64", "df64", "f32"])
@pytest.mark.parametrize("cols", [1, 2, 3, 4, 5])
def test_product(n, leaf, q, fmt, cols):
    X = torch.from_numpy(W.uniform_points(n, 2, n)).cuda()
    o = dict(kernel="exponential", length=0.2, nugget=1e-2, leaf=leaf, q=q)
    A = pkg.H2Matrix(X, **o)
    B = pkg.H2Matrix(X, **o, storage="df64" if fmt == "df64" else "f64", with_f32=fmt == "f32")
    V = torch.from_numpy(np.random.default_rng(cols).standard_normal((n, cols))).cuda()
    Y = B.apply(V, precision="mixed_f32") if fmt == "f32" else B.apply(V)
    # units in the last place of the format's sums, over chains of some 64 terms per level
    eps = {"f64": 2.0 ** -53, "df64": 2.0 ** -44, "f32": 2.0 ** -24}[fmt]
    for c in range(cols):
        x = V[:, c].contiguous()
        ref = A.apply_level(1, x, precision="f64_dd")
        size = A.apply_level(1, x.abs(), precision="f64_dd")
        assert float((Y[:, c] - ref).norm()) <= 64 * eps * float(size.norm())
    A.close()
    B.close()
