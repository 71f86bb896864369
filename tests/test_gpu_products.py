"""J v, J^T w and H v formed from the expression graph (FP64) and from the derivative entries (mixed), on
patterns where the two ways differ most: shared factors, repeated and colliding symbols, powers,
quotients, library functions, sums that cancel, and instance counts around the CTA size."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import Model, sin, cos, exp, log, sqrt, tanh, atan2, hypot

pytestmark = pytest.mark.gpu


def graph_model(n, seed=0):
    rng = np.random.default_rng(seed)
    m = Model()
    x = m.add_var(n + 3)
    th = m.add_par([0.7])
    i = rng.integers(0, n + 3, n).astype(np.int32)
    j = np.where(rng.random(n) < 0.3, i, rng.integers(0, n + 3, n)).astype(np.int32)  # i == j now and then
    d = dict(i=i, j=j, a=rng.uniform(0.5, 1.5, n), b=rng.uniform(0.5, 1.5, n))
    m.add_obj(lambda d: d.a * x[d.i] ** 3 * x[d.j] + sin(x[d.i] - x[d.j]), data=d)
    blk = m.add_con(lambda d: x[d.i] * x[d.j] * (d.a * cos(x[d.i] - x[d.j]) + d.b * sin(x[d.i] - x[d.j])), data=d)
    m.add_con(lambda d: x[d.i] * x[d.j] * (d.b * cos(x[d.j] - x[d.i]) - d.a * sin(x[d.j] - x[d.i])), data=d)
    m.add_con(lambda d: (x[d.i] ** 2 - x[d.j] ** 2) / (2 + x[d.i] * x[d.j]) - th[0] * x[d.k], data=d)
    m.add_con(lambda d: x[d.i] ** -2 * exp(-x[d.j]) + log(1 + x[d.i] ** 2) * sqrt(2 + x[d.j]), data=d)
    m.add_con(lambda d: tanh(x[d.i]) * atan2(x[d.j], 1 + x[d.i]) + hypot(x[d.i], x[d.j]) * (1 + x[d.i]) ** x[d.j], data=d)
    m.add_con(lambda d: 3 * x[d.k] - x[d.k + 1], n=n)
    m.add_con_aug(blk, lambda d: (d.r, x[d.i] * x[d.j] * x[d.i] - d.a * x[d.r]),
                  data=dict(r=rng.integers(0, n, n).astype(np.int32), **d))
    return m.flat()


# tolerance: every term is a product of at most ~20 rounded factors and functions (each within 2 ulp), and
# a result sums at most ~40 of them; 1e-13 is a hundred times their accumulated 2^-53.  Mixed: the
# entries are FP32 (2^-24 per operation), 1e-5 by the same count.
@pytest.mark.parametrize("precision,tol", [(binding.EXA_FP64, 1e-13), (binding.EXA_MIXED_FP32, 1e-5)])
@pytest.mark.parametrize("n", [1, 63, 64, 65, 1000])
@pytest.mark.parametrize("scale", [0.3, 3.0])  # warps within and beyond pi/4
def test_products(precision, tol, n, scale):
    flat = graph_model(n)
    m = binding.exa_create(flat, precision, flags=binding.EXA_FLAG_NO_TUNE)
    o = oracle.Oracle(flat)
    rng = np.random.default_rng(n)
    x = 0.5 + scale * rng.random(flat.nvar)
    y, v, w = rng.standard_normal(flat.ncon), rng.standard_normal(flat.nvar), rng.standard_normal(flat.ncon)
    t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    got = dict(jv=m.jprod(t(x), t(v)), jtw=m.jtprod(t(x), t(w)), hv=m.hprod(t(x), t(y), 1.3, t(v)))
    ref = dict(jv=o.jprod(x, v), jtw=o.jtprod(x, w), hv=o.hprod(x, y, 1.3, v))
    for k, r in ref.items():
        assert np.linalg.norm(got[k].cpu().numpy() - r) <= tol * np.linalg.norm(r), k


@pytest.mark.parametrize("precision,tol", [(binding.EXA_FP64, 1e-13), (binding.EXA_MIXED_FP32, 1e-5)])
@pytest.mark.parametrize("n", [1, 40, 700])
def test_wide_stencil(precision, tol, n):
    """Patterns over many shared variables: H v from the summed Hessian entries."""
    m = Model()
    x = m.add_var(n + 24)
    m.add_con(lambda d: sum((0.5 + 0.1 * t) * x[d.k + 2 * t] * x[d.k + 2 * t + 1] ** 2 for t in range(12)), n=n)
    m.add_obj(lambda d: x[d.k] ** 2 * x[d.k + 1], n=n)
    flat = m.flat()
    mm, o = binding.exa_create(flat, precision, flags=binding.EXA_FLAG_NO_TUNE), oracle.Oracle(flat)
    rng = np.random.default_rng(n)
    xv, y, v = rng.uniform(0.5, 1.5, flat.nvar), rng.standard_normal(flat.ncon), rng.standard_normal(flat.nvar)
    t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    got, ref = mm.hprod(t(xv), t(y), 0.7, t(v)).cpu().numpy(), o.hprod(xv, y, 0.7, v)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
