"""Kernels that overlap with the one before them: products and smoothing steps queued one after
the other on changing inputs equal the same calls with a synchronisation after each, on a
stream and in a captured graph."""
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


# blocks of 16, 32 and 64; every format; one CTA per kernel and many; no far field
@pytest.mark.parametrize("n,dim,leaf,q,storage,precision", [
    (50, 2, 64, 4, "f64", ""), (777, 2, 16, 4, "f64", ""), (3001, 2, 64, 4, "df64", ""), (3001, 3, 32, 3, "f64", ""),
    (5000, 3, 64, 4, "f64", ""), (5000, 3, 64, 4, "f64", "mixed_f32"), (20011, 3, 64, 4, "f64", "mixed_f32")])
def test_queued_products(n, dim, leaf, q, storage, precision):
    X = torch.from_numpy(W.uniform_points(n, dim, 3)).cuda()
    A = pkg.H2Matrix(X, "exponential", length=0.2, nugget=1e-2, leaf=leaf, q=q, storage=storage, with_f32=bool(precision))
    kw = dict(precision=precision) if precision else {}
    # atomic sums: n terms may be added in another order
    tol = (n ** 0.5) * (2.0 ** -24 if precision else (2.0 ** -46 if storage == "df64" else EPS)) * 8
    rng = np.random.default_rng(n)
    xs = [torch.from_numpy(rng.standard_normal(n)).cuda() for _ in range(6)]
    want = []
    for x in xs:
        want.append(A.apply(x, **kw).clone())
        torch.cuda.synchronize()
    v, y = torch.empty_like(xs[0]), torch.empty_like(xs[0])
    got = []
    for x in xs:                                     # v and y are reused at once
        v.copy_(x)
        A.apply(v, y=y, **kw)
        got.append(y.clone())
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s):
        A.apply(v, y=y, **kw)
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        A.apply(v, y=y, **kw)
    for x in xs:
        v.copy_(x)
        g.replay()
        got.append(y.clone())
    for a, b in zip(got, want + want):
        assert float((a - b).norm()) <= tol * float(b.norm())
    A.close()
