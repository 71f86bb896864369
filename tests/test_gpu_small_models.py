"""Models of every size around the sharing of small device arrays (32 KB), whose arrays fill shared allocations
to different points: products, gradient and CSC values against the oracle, with earlier models still alive."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding as B
from paper_2608_16265_gb300.ir import Model, sin

pytestmark = pytest.mark.gpu


def model(n):
    m = Model()
    x, s = m.add_var(n + 1), m.add_var(1)
    m.add_obj(lambda d: x[d.k] ** 2 * x[d.k + 1], n=n)
    blk = m.add_con(lambda d: s[0] * x[d.k] ** 2 + sin(x[d.k + 1]), n=n)
    m.add_con_aug(blk, lambda d: (d.r, x[d.r] * x[d.k]), data=dict(r=np.arange(n, dtype=np.int32)[::-1].copy()))
    return m.flat()


@pytest.mark.parametrize("precision,tol", [(B.EXA_FP64, 1e-13), (B.EXA_MIXED_FP32, 1e-5)])  # as in test_gpu_products.py
def test_sizes(precision, tol):
    alive = []
    for n in [1, 2, 7, 40, 300, 511, 1000, 1023, 1024, 1025, 1365, 1366, 2000, 2047, 2048, 2049, 2730, 3000, 4095, 4096, 4097,
              5000, 8191, 8192, 8193, 9000]:
        flat = model(n)
        m, o = B.exa_create(flat, precision, flags=B.EXA_FLAG_NO_TUNE), oracle.Oracle(flat)
        r = np.random.default_rng(n)
        x, y = r.uniform(0.5, 1.5, flat.nvar), r.standard_normal(flat.ncon)
        alive.append((m, o, x, y, r.standard_normal(flat.nvar), r.standard_normal(flat.ncon)))
    for m, o, x, y, v, w in alive:
        X, Y, V, W = (torch.as_tensor(a, device="cuda") for a in (x, y, v, w))
        got = dict(g=m.grad(X), c=m.cons(X), jac=m.jac_csc(X), hess=m.hess_csc(X, Y, 0.5), jv=m.jprod(X, V),
                   jtw=m.jtprod(X, W), hv=m.hprod(X, Y, 0.5, V))
        ref = dict(g=o.grad(x), c=o.cons(x), jac=o.jac_csc(x), hess=o.hess_csc(x, y, 0.5), jv=o.jprod(x, v),
                   jtw=o.jtprod(x, w), hv=o.hprod(x, y, 0.5, v))
        for k, r in ref.items():
            assert np.linalg.norm(got[k].cpu().numpy() - r) <= tol * np.linalg.norm(r), (k, m.nvar)
