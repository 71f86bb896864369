"""Which way H v is formed: per-instance terms, or the CSC values where terms outnumber them, unless some
variable's row or column of the Hessian is long (one lane would walk it)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_16265_gb300 import binding as B
from paper_2608_16265_gb300.ir import Model

pytestmark = pytest.mark.gpu


def wide(n, shared):
    m = Model()
    x, s = m.add_var(n + 16), m.add_var(1)
    m.add_con(lambda d: (s[0] if shared else 1.5) * sum((0.5 + 0.1 * t) * x[d.k + t] ** 2 for t in range(16)), n=n)
    return m.flat()


# the shared variable has an entry with every x: n + 15 of them, 32 at n = 17.  One instance's 16 or 17
# terms are no more than four times its entries.
@pytest.mark.parametrize("precision,tol", [(B.EXA_FP64, 1e-13), (B.EXA_MIXED_FP32, 1e-5)])  # as in test_gpu_products.py
@pytest.mark.parametrize("n,shared,fp64,mixed", [(1, False, 0, 1), (200, False, 1, 1), (3000, False, 1, 1), (1, True, 0, 1),
                                                 (17, True, 1, 1), (18, True, 0, 2), (3000, True, 0, 2)])
def test_route(n, shared, fp64, mixed, precision, tol):
    flat = wide(n, shared)
    m, o = B.exa_create(flat, precision, flags=B.EXA_FLAG_NO_TUNE), oracle.Oracle(flat)
    assert int(m.stat("hprod_route")) == (fp64 if precision == B.EXA_FP64 else mixed)
    rng = np.random.default_rng(n)
    x, y, v = rng.uniform(0.5, 1.5, flat.nvar), rng.uniform(0.5, 1.5, flat.ncon), rng.standard_normal(flat.nvar)
    X, Y, V = (torch.as_tensor(a, device="cuda") for a in (x, y, v))
    got, ref = m.hprod(X, Y, 0.7, V).cpu().numpy(), o.hprod(x, y, 0.7, v)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)
