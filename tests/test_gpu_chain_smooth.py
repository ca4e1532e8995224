"""Smoothing steps queued back to back, whose kernels overlap with the ones before
them (the direction formed by the next product's first kernel, partial sums, the state of the
column, the tickets of the upward pass), equal the same calls with a synchronisation after
each."""
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


def matrix(n, dim, leaf, q):
    return pkg.H2Matrix(torch.from_numpy(W.uniform_points(n, dim, 3)).cuda(), "exponential", length=0.2, nugget=1e-2,
                        leaf=leaf, q=q, with_f32=True)


def close(a, b, tol):
    return float((a - b).norm()) <= tol * float(b.norm())


# blocks of 16, 32 and 64; small levels and larger ones. Few steps: rounding in the order of
# the atomic sums is multiplied by the condition of each step
@pytest.mark.parametrize("n,dim,leaf,q", [(1000, 2, 16, 4), (3001, 3, 32, 3), (5000, 3, 64, 4), (20011, 3, 64, 4)])
@pytest.mark.parametrize("precision", ["f64", "mixed_f32"])
@pytest.mark.parametrize("steps", [1, 3])
def test_queued_smoothing(n, dim, leaf, q, precision, steps):
    A = matrix(n, dim, leaf, q)
    rng = np.random.default_rng(n)
    # (kappa < 1e6) a step's coefficients are off by sqrt(n) roundings of the products, the
    # iterates by a few times as much per step
    tol = 64 * steps * n ** 0.5 * (2.0 ** -24 if precision == "mixed_f32" else EPS)
    levels = [i for i in (1, 2, 3) if i < A.levels]
    jobs = [(i, torch.from_numpy(rng.standard_normal(A.level_size(i))).cuda(), k) for k in range(3) for i in levels]
    want = []
    for i, f, k in jobs:
        x0 = f * 0.5 if k == 1 else None                    # from zero and from a start
        want.append([t.clone() for t in A.smooth(i, f, x0=x0, n=steps, precision=precision)])
        torch.cuda.synchronize()
    bufs = {i: torch.empty(A.level_size(i), dtype=torch.float64, device="cuda") for i in levels}
    got = []
    for i, f, k in jobs:                                    # the inputs' buffers are reused at once
        bufs[i].copy_(f)
        got.append(A.smooth(i, bufs[i], x0=f * 0.5 if k == 1 else None, n=steps, precision=precision))
    for (xa, ra), (xb, rb), (i, f, k) in zip(got, want, jobs):
        assert close(xa, xb, tol)
        assert float((ra - rb).norm()) <= tol * (float(f.norm()) + float(rb.norm()))
    A.close()
