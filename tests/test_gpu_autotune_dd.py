"""The double-double product after the autotuner: its launches keep their shape (the tuned
numbers are those of other kernels), and its results their values."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2501_17656_gb300 as pkg  # noqa: E402

pkg.load_library(build_if_missing=True)


def best_ms(f):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t = []
    for _ in range(10):
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return min(t[2:])


# many block rows with few blocks each (points on a line), where a CTA more per row is most of
# its work; blocks of 64 and of 32
@pytest.mark.parametrize("leaf,q", [(64, 64), (32, 32)])
def test_double_double_product_after_autotune(leaf, q):
    n = 200000
    A = pkg.H2Matrix(torch.from_numpy(W.uniform_points(n, 1, 3)).cuda(), "exponential", length=0.1, nugget=1e-2,
                     leaf=leaf, q=q)
    x = torch.from_numpy(np.random.default_rng(1).standard_normal(n)).cuda()
    y0, y1 = torch.empty_like(x), torch.empty_like(x)
    t0 = best_ms(lambda: A.apply_level(1, x, precision="f64_dd", y=y0))
    A.autotune()
    t1 = best_ms(lambda: A.apply_level(1, x, precision="f64_dd", y=y1))
    assert float((y0 - y1).norm()) <= 2.0 ** -52 * float(y0.norm())     # sums of 100 bits, rounded once
    assert t1 <= 1.3 * t0, (t0, t1)
    A.close()
